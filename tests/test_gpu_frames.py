"""Streaming frames around the sizes where the launch form changes (one cluster, two overlapped
kernels, a captured sequence), back to back without a synchronisation between them (GPU only).

Bar: values bit-exact against the oracle after every sequence, touched counts equal to the sparsity
pattern's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 39, 40, 41, 64, 1, 1023, 1024, 1025, 40, 3, 1500, 2100, 41, 0, 12]


@pytest.fixture(scope="module")
def sta():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_11673_gb300 as P
    P.load_library()
    return P


def _frames(rng, mask, sizes):
    """Frames of exactly `size` edited tetrahedra, swaps among them."""
    mask = mask.copy()
    out = []
    for n in sizes:
        act, ina = np.flatnonzero(mask), np.flatnonzero(mask == 0)
        ns = min(n // 3, ina.size)
        rest = n - 2 * ns
        a = rng.permutation(act)[: ns + rest]
        swaps = list(zip(a[:ns], rng.permutation(ina)[:ns]))
        on = np.setdiff1d(ina, [s[1] for s in swaps])[: rest // 2]
        off = a[ns: ns + rest - on.size]
        out.append(W.make_edits(off=off, on=on, swaps=swaps))
        for s in swaps:
            mask[s[0]], mask[s[1]] = 0, 1
        mask[off], mask[on] = 0, 1
    return out, mask


def _touched(tets, edits):
    """CSR entries of the diagonal and pair blocks of the edited tetrahedra."""
    t = np.concatenate([edits[:, 1], edits[edits[:, 0] == 2, 2]])
    v = np.sort(tets[t], axis=1).astype(np.int64)
    pairs = {(a, b) for a in range(4) for b in range(a + 1, 4)}
    pr = np.unique(np.concatenate([v[:, a] * (1 << 32) + v[:, b] for a, b in pairs]))
    return 9 * np.unique(v).size + 18 * pr.size


@pytest.mark.parametrize("graph", [0, 4096, 1100])
@pytest.mark.parametrize("policy, eps", [(0, 0.0), (0, 0.5), (1, 0.5)])
def test_frames_at_the_launch_form_edges(sta, orc, graph, policy, eps):
    rng = np.random.default_rng(7 + graph + policy)
    X, tets, _ = W.kuhn_cube(9, 0.1, rng)
    T = tets.shape[0]
    E, nu = W.lognormal_E(rng, T), np.full(T, 0.3)
    mask0 = (rng.uniform(size=T) < 0.7).astype(np.uint8)
    P = orc.Pattern(X.shape[0], tets)
    Ke, _ = orc.element_all(X, tets, E, nu)
    asm = sta.Assembler(X, tets, E, nu, eps=eps)
    if policy:
        asm.set_policy(sta.STA_POLICY_FIXED)
    asm.full_rebuild(mask0)
    if graph:
        asm.graph_enable(graph)
    frames, end = _frames(rng, mask0, SIZES)
    for i, f in enumerate(frames):
        asm.apply_edits(f)
        if i % 4 == 3:
            assert asm.last_touched() == (_touched(tets, f) if len(f) else 0), (i, len(f))
    ref = P.fx_rebuild(Ke, P.fx_exponents(Ke), end, eps)[1] if policy else P.rebuild(Ke, end, eps)
    got = asm.values().cpu().numpy().view(np.uint64)
    assert np.array_equal(got, ref.view(np.uint64)), int((got != ref.view(np.uint64)).sum())
    assert np.array_equal(asm.mask().cpu().numpy(), end)
    asm.close()
