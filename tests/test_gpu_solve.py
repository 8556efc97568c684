"""The conjugate-gradient solve over the sizes at which its plan changes (GPU only): systems of
less than a warp, of one node more or less than a slice, quads or single lanes per node, matrix
kept in shared memory or streamed, vectors in shared or in global memory, scalar and 3 x 3 blocks.

Bar: the returned x satisfies the system to 10 tol (||A x - b|| over the free rows, formed by
scipy from the context's CSR values, which other tests pin to the oracle bit for bit); rows that
are not solved for are 0; a second solve gives the same bits; max_iter is honoured."""
import numpy as np
import pytest

import workloads as W

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


def _solve_and_check(sta, asm, seed, free_np, val=None):
    import scipy.sparse as sp
    import torch
    n = asm.n_rows
    rp, col, v = (a.cpu().numpy() for a in asm.csr())
    if val is not None:
        v = val.cpu().numpy()
    A = sp.csr_matrix((v, col, rp), shape=(n, n))
    b_np = np.random.default_rng(seed).standard_normal(n)
    b = torch.as_tensor(b_np, device="cuda")
    free = torch.as_tensor(free_np, device="cuda")
    x, it, rel = sta.sta_solve(asm.h, b, free, val, tol=TOL, max_iter=20000)
    y, it2, rel2 = sta.sta_solve(asm.h, b, free, val, tol=TOL, max_iter=20000)
    assert torch.equal(x, y) and it == it2 and rel == rel2, "a solve is deterministic"
    xn = x.cpu().numpy()
    live = free_np & (A.diagonal() != 0)
    assert np.all(xn[~live] == 0.0)
    assert 0 < it < 20000 and rel <= TOL
    r = (A @ xn - b_np)[live]
    assert np.linalg.norm(r) <= 10 * TOL * np.linalg.norm(b_np[live])
    _, it3, _ = sta.sta_solve(asm.h, b, free, val, tol=TOL, max_iter=3)
    assert it3 == min(3, it)


@pytest.mark.parametrize("nx, ny, nz", [(1, 1, 1), (1, 2, 1), (1, 1, 5), (7, 2, 3), (9, 9, 9), (20, 20, 20),
                                        (38, 38, 39)])
def test_elasticity_sizes(sta, nx, ny, nz):
    rng = np.random.default_rng(nx + ny + nz)
    X, tets, _ = W.kuhn_cube(nz, 0.1, rng, nx=nx, ny=ny)
    T = tets.shape[0]
    asm = sta.Assembler(X, tets, W.lognormal_E(rng, T), np.full(T, 0.3), eps=50.0)
    asm.full_rebuild((rng.uniform(size=T) < 0.8).astype(np.uint8))
    _solve_and_check(sta, asm, 5, rng.uniform(size=3 * X.shape[0]) < 0.9)
    asm.close()


@pytest.mark.parametrize("N", [1, 4, 20, 40, 54])
def test_scalar_sizes(sta, N):
    rng = np.random.default_rng(N)
    X, tets, _ = W.kuhn_cube(N)
    T = tets.shape[0]
    # one node of no tetrahedron: an empty row
    px = sta.ProxyAssembler(X.shape[0] + 1, tets, eps=0.1)
    px.full_rebuild((rng.uniform(size=T) < 0.7).astype(np.uint8))
    _solve_and_check(sta, px, 6, rng.uniform(size=X.shape[0] + 1) < 0.95)
    px.close()


def test_vectors_in_global_memory_and_unaligned_values(sta):
    """About 2,000 nodes an SM: the vectors no longer fit shared memory.  The values are passed
    as a view that starts 8 bytes past a 16-byte boundary."""
    import torch
    rng = np.random.default_rng(1)
    X, tets, _ = W.kuhn_cube(67, 0.1, rng)
    T = tets.shape[0]
    asm = sta.Assembler(X, tets, W.lognormal_E(rng, T), np.full(T, 0.3), eps=500.0)
    asm.full_rebuild((rng.uniform(size=T) < 0.9).astype(np.uint8))
    buf = torch.empty(asm.nnz + 1, dtype=torch.float64, device="cuda")
    buf[1:] = asm.values()
    _solve_and_check(sta, asm, 7, rng.uniform(size=asm.n_rows) < 0.9, buf[1:])
    asm.close()


def test_long_rows(sta):
    """An edge fan: two rows of 302 blocks among rows of 5."""
    wl = W.edge_fan(K=300)
    asm = sta.Assembler(wl.X, wl.tets, wl.E, wl.nu, eps=1e3)
    asm.full_rebuild(wl.mask0)
    _solve_and_check(sta, asm, 8, np.ones(asm.n_rows, bool))
    asm.close()
