"""A frame captured into a CUDA graph of the caller's and replayed, alone and after rebuilds (GPU only):
one launch (8 edits), two overlapped ones (100), and the allocation-free entry point.

Bar: after every replay the values are bit-exact against the oracle for the frame's end state, and the
touched count is the frame's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sta():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_11673_gb300 as P
    P.load_library()
    return P


def _frame(rng, mask, n):
    act, ina = np.flatnonzero(mask), np.flatnonzero(mask == 0)
    a, b = rng.permutation(act)[: n // 2], rng.permutation(ina)[: n - n // 2]
    k = n // 4
    end = mask.copy()
    end[a], end[b] = 0, 1
    return W.make_edits(off=a[k:], on=b[k:], swaps=list(zip(a[:k], b[:k]))), end


@pytest.mark.parametrize("entry, n", [("frame", 8), ("frame", 100), ("noalloc", 50)])
@pytest.mark.parametrize("mesh", ["block", "fan"])
@pytest.mark.parametrize("fixed", [False, True])
def test_replayed_frames(sta, orc, entry, n, mesh, fixed):
    import torch
    rng = np.random.default_rng(n)
    if mesh == "fan":  # units of 300 contributors
        wl = W.edge_fan(K=300)
        X, tets, E, nu = wl.X, wl.tets, wl.E, wl.nu
    else:
        X, tets, _ = W.kuhn_cube(6, 0.1, rng)
        E, nu = W.lognormal_E(rng, len(tets)), np.full(len(tets), 0.3)
    mask = (rng.uniform(size=len(tets)) < 0.5).astype(np.uint8)
    frame, end = _frame(rng, mask, n)
    P = orc.Pattern(X.shape[0], tets)
    Ke, _ = orc.element_all(X, tets, E, nu)
    ref = P.fx_rebuild(Ke, P.fx_exponents(Ke), end, 0.0)[1] if fixed else P.rebuild(Ke, end)
    asm = sta.Assembler(X, tets, E, nu)
    asm.full_rebuild(mask)
    if fixed:
        asm.set_policy(sta.STA_POLICY_FIXED)
    apply = asm.apply_edits if entry == "frame" else lambda e, stream=None: sta.sta_apply_edits_noalloc(asm.h, e, stream)
    # once outside a capture: the first call sets up its buffers
    apply(frame)
    want = asm.last_touched()
    torch.cuda.synchronize()
    asm.full_rebuild(mask)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        apply(frame, stream=torch.cuda.current_stream())
    for k in range(6):
        if fixed or k % 2:  # (the fixed-point frame adds to its sums: it starts from the mask each time)
            asm.full_rebuild(mask)
        g.replay()
        torch.cuda.synchronize()
        got = asm.values().cpu().numpy().view(np.uint64)
        assert np.array_equal(got, ref.view(np.uint64)), k
        assert np.array_equal(asm.mask().cpu().numpy(), end), k
        assert asm.last_touched() == want, k
    asm.close()
