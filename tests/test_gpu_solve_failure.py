"""A solve whose grid-wide wait runs out (GPU only): the limit of the waits is set to a few polls, so
that some or all thread blocks give up.  The call returns STA_ECUDA and leaves the caller's x, or the
state of the implicit-Euler loop, as it was; with the usual limit the same context solves again."""
import numpy as np
import pytest

import workloads as W
from tests import ctx_access

pytestmark = pytest.mark.gpu

LIMITS = [0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 32]
USUAL = 1 << 22


@pytest.fixture(scope="module")
def sta():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_11673_gb300 as P
    P.load_library()
    return P


@pytest.fixture(scope="module")
def access(tmp_path_factory):
    return ctx_access.load(tmp_path_factory.mktemp("ctx_access"))


@pytest.mark.parametrize("N", [6, 20])
@pytest.mark.parametrize("kind", ["elasticity", "proxy"])
def test_solve_leaves_x(sta, access, N, kind):
    import torch
    rng = np.random.default_rng(N)
    X, tets, _ = W.kuhn_cube(N, 0.1, rng)
    T = tets.shape[0]
    if kind == "proxy":
        asm = sta.ProxyAssembler(X.shape[0], tets, eps=0.1)
    else:
        asm = sta.Assembler(X, tets, W.lognormal_E(rng, T), np.full(T, 0.3), eps=50.0)
    asm.full_rebuild(np.ones(T, np.uint8))
    b = torch.as_tensor(rng.standard_normal(asm.n_rows), device="cuda")
    free = torch.ones(asm.n_rows, dtype=torch.uint8, device="cuda")
    start = torch.as_tensor(rng.standard_normal(asm.n_rows), device="cuda")
    want, it, _ = sta.sta_solve(asm.h, b, free, x0=start, max_iter=2)
    L = sta.load_library()
    failed = 0
    for max_iter in (0, 2):  # the last exchange is the one after which x is written
        for limit in LIMITS:
            access.ctx_set_spins(asm.h, limit)
            x = start.clone()
            rc = L.sta_solve(asm.h, None, b.data_ptr(), free.data_ptr(), 1e-12, max_iter, x.data_ptr(), None, None,
                             torch.cuda.current_stream().cuda_stream)
            assert rc in (sta.STA_OK, sta.STA_ECUDA)
            if rc != sta.STA_OK:
                failed += 1
                assert torch.equal(x, start), limit
            elif max_iter:
                assert torch.equal(x, want), limit
    assert failed > 0  # (a limit of 0 always fails)
    access.ctx_set_spins(asm.h, USUAL)
    again, it2, _ = sta.sta_solve(asm.h, b, free, x0=start, max_iter=2)
    assert torch.equal(again, want) and it2 == it
    asm.close()


def test_step_leaves_the_state(sta, access):
    wl = W.plain_small(seed=2)
    asm = sta.Assembler(wl.X, wl.tets, wl.E, wl.nu)
    asm.full_rebuild(wl.mask0)
    rng = np.random.default_rng(0)
    asm.dyn_setup(1000.0, 1e-3, rng.standard_normal(asm.n_rows))
    asm.dyn_step()
    u, v, _ = asm.dyn_state()
    for limit in LIMITS:
        access.ctx_set_spins(asm.h, limit)
        u0, v0 = u.clone(), v.clone()
        try:
            asm.dyn_step(max_iter=1)
        except sta.StaError as e:
            assert e.status == sta.STA_ECUDA
            assert bool((u == u0).all()) and bool((v == v0).all()), limit
        else:
            assert not bool((u == u0).all())
    access.ctx_set_spins(asm.h, USUAL)
    it, rel = asm.dyn_step()
    assert it > 0 and rel <= 1e-10
    asm.close()
