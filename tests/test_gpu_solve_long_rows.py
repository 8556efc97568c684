"""The solve's plan on a mesh with a few rows far longer than the rest (GPU only): a block large enough
for a lane per node, joined by an edge fan whose two axis nodes have K + 2 neighbours.

Bar: a quad per node where the long rows decide, the lane per node where they don't; the returned x
satisfies the system to 10 tol (||A x - b||, formed by scipy from the context's CSR values)."""
import numpy as np
import pytest

import workloads as W
from tests import ctx_access

pytestmark = pytest.mark.gpu

TOL = 1e-10


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


@pytest.mark.parametrize("scalar, K, lanes", [(False, 0, 1), (False, 20, 1), (False, 300, 4), (True, 0, 1),
                                              (True, 60, 1), (True, 600, 4)])
def test_block_with_a_fan(sta, access, scalar, K, lanes):
    import scipy.sparse as sp
    import torch
    rng = np.random.default_rng(K)
    X, tets, _ = W.kuhn_cube(40, 0.1, rng)
    if K:
        fan = W.edge_fan(K=K)
        X, tets = np.concatenate([X, fan.X]), np.concatenate([tets, fan.tets + len(X)])
    T = len(tets)
    if scalar:
        asm = sta.ProxyAssembler(len(X), tets, eps=0.5)
    else:
        asm = sta.Assembler(X, tets, W.lognormal_E(rng, T), np.full(T, 0.3), eps=500.0)
    asm.full_rebuild(np.ones(T, np.uint8))
    n = asm.n_rows
    b_np = rng.standard_normal(n)
    free = torch.ones(n, dtype=torch.uint8, device="cuda")
    x, it, rel = sta.sta_solve(asm.h, torch.as_tensor(b_np, device="cuda"), free, tol=TOL)
    assert access.ctx_plan_lanes(asm.h) == lanes
    assert 0 < it < 20000 and rel <= TOL
    rp, col, v = (a.cpu().numpy() for a in asm.csr())
    A = sp.csr_matrix((v, col, rp), shape=(n, n))
    assert np.linalg.norm(A @ x.cpu().numpy() - b_np) <= 10 * TOL * np.linalg.norm(b_np)
    asm.close()
