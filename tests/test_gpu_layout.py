"""The unit-major element cache and the fold that streams it (GPU only): contributor counts on
either side of the activity words (32, 64 contributors), units of one chunk, many chunks and more
chunks than resident CTAs, activity with gaps, empty chunks, both rebuild forms and policies.

Bar: values bit-exact against the oracle (rebuild, then a streamed frame, then a refold)."""
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


def _same(asm, ref, what):
    got = asm.values().cpu().numpy().view(np.uint64)
    assert np.array_equal(got, ref.view(np.uint64)), f"{what}: {int((got != ref.view(np.uint64)).sum())} differ"


def _check(sta, orc, X, tets, E, nu, masks, eps, forms):
    P = orc.Pattern(X.shape[0], tets)
    Ke, bad = orc.element_all(X, tets, E, nu)
    assert bad == 0
    for form in forms:
        asm = sta.Assembler(X, tets, E, nu, eps=eps)
        K = asm.element_matrices(np.arange(tets.shape[0])).cpu().numpy()
        assert np.array_equal(K.reshape(-1).view(np.uint64), Ke.reshape(-1).view(np.uint64)), "element cache"
        asm.set_rebuild_form(form)
        for k, m in enumerate(masks):
            asm.full_rebuild(m)
            _same(asm, P.rebuild(Ke, m, eps), f"form {form} mask {k}")
            nxt = masks[(k + 1) % len(masks)]
            asm.apply_edits(W.make_edits(off=np.flatnonzero((m != 0) & (nxt == 0)),
                                         on=np.flatnonzero((m == 0) & (nxt != 0))))
            _same(asm, P.rebuild(Ke, nxt, eps), f"form {form} mask {k}: streamed")
            asm.refold()
            _same(asm, P.rebuild(Ke, nxt, eps), f"form {form} mask {k}: refolded")
        asm.set_policy(sta.STA_POLICY_FIXED)
        e = P.fx_exponents(Ke)
        for m in masks[:2]:
            asm.full_rebuild(m)
            _same(asm, P.fx_rebuild(Ke, e, m, eps)[1], f"form {form}: fixed point")
        asm.close()


@pytest.mark.parametrize("K", [31, 32, 33, 63, 64, 65, 96, 97, 130])
def test_fans_at_the_activity_word_edges(sta, orc, K):
    """K tetrahedra around one edge: its pair unit and both axis nodes have K contributors."""
    wl = W.edge_fan(K=K)
    rng = np.random.default_rng(K)
    last = np.zeros(K, np.uint8)
    last[-1] = 1
    masks = [wl.mask0, (rng.uniform(size=K) < 0.5).astype(np.uint8), np.ones(K, np.uint8), last,
             np.zeros(K, np.uint8)]
    _check(sta, orc, wl.X, wl.tets, wl.E, wl.nu, masks, 0.25 if K % 2 else 0.0,
           (sta.STA_REBUILD_FUSED, sta.STA_REBUILD_ZERO_FILL))


@pytest.mark.parametrize("kind, size, eps", [("block", 1, 0.5), ("block", 13, 0.0), ("block", 24, 0.5),
                                             ("refine", 9, 0.0), ("refine", 15, 0.5), ("fracture", 22, 0.0)])
def test_sizes_and_activity_patterns(sta, orc, kind, size, eps):
    """From one hex to several chunks per resident CTA; masks with scattered, contiguous and very
    few active tetrahedra (copies split at long inactive stretches, chunks without any)."""
    rng = np.random.default_rng(size)
    if kind == "block":
        X, tets, _ = W.kuhn_cube(size, 0.1, rng)
        base = np.ones(tets.shape[0], np.uint8)
    else:
        wl = (W.refinement_hierarchy(N=size, radius=0.3, frames=1) if kind == "refine"
              else W.prefractured_block(N=size, sites=9, frames=1))
        X, tets, base = wl.X, wl.tets, wl.mask0
    T = tets.shape[0]
    half = np.zeros(T, np.uint8)
    half[: T // 2] = 1
    masks = [base, (rng.uniform(size=T) < 0.5).astype(np.uint8), half,
             (rng.uniform(size=T) < 0.01).astype(np.uint8)]
    _check(sta, orc, X, tets, W.lognormal_E(rng, T), np.full(T, 0.3), masks, eps,
           (sta.STA_REBUILD_FUSED, sta.STA_REBUILD_ZERO_FILL))


@pytest.mark.parametrize("K", [2047, 2048, 2049, 4100])
def test_units_longer_than_a_pass_over_the_mask(sta, orc, K):
    """Activity words of one unit formed from several windows of its contributors."""
    wl = W.edge_fan(K=K)
    rng = np.random.default_rng(K)
    masks = [(rng.uniform(size=K) < 0.5).astype(np.uint8), np.ones(K, np.uint8)]
    _check(sta, orc, wl.X, wl.tets, wl.E, wl.nu, masks, 0.0, (sta.STA_REBUILD_FUSED,))
