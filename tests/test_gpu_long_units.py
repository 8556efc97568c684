"""Back-to-back streaming frames on units whose activity words are kept apart from the unit's record
(more than 64 contributors): the frame's claims change those words and its folds read them back (GPU
only).

Bar: values bit-exact against the oracle after every run of frames that nothing waits between."""
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


@pytest.mark.parametrize("K", [65, 96, 97, 130])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("most", [40, 64])
def test_frames_back_to_back(sta, orc, K, graph, most):
    """Up to `most` edits a frame: one launch (up to 40), or two overlapped ones among them."""
    wl = W.edge_fan(K=K)
    rng = np.random.default_rng(K + most)
    P = orc.Pattern(wl.X.shape[0], wl.tets)
    Ke, _ = orc.element_all(wl.X, wl.tets, wl.E, wl.nu)
    asm = sta.Assembler(wl.X, wl.tets, wl.E, wl.nu)
    mask = np.ones(K, np.uint8)
    asm.full_rebuild(mask)
    if graph:
        asm.graph_enable(256)
    for run in range(8):
        for _ in range(12):
            t = rng.permutation(K)[: rng.integers(1, most + 1)]
            asm.apply_edits(W.make_edits(off=t[mask[t] == 1], on=t[mask[t] == 0]))
            mask[t] ^= 1
        got = asm.values().cpu().numpy().view(np.uint64)
        assert np.array_equal(got, P.rebuild(Ke, mask).view(np.uint64)), run
    asm.close()
