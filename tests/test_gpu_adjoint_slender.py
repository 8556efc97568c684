"""The adjoint on slender tetrahedra (GPU only): spires and flakes of aspect 1 to 100, every node in
turn the far tip, an upstream gradient on one node's diagonal block, on one entry, or with one node's
block far above the rest.

Bar: every output within 1e-13 of the size of the terms it sums, against the defining sums in extended
precision.  (Each gradient carries a few roundings times the aspect where the volume cancels, 100 x
1.1e-16 x 4; each form at most 27 products per block, as no gradient is larger than sqrt(3) times
the eliminated one.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
E0, NU0 = 1.3e5, 0.3
TOL = 1e-13


@pytest.fixture(scope="module")
def sta():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_11673_gb300 as P
    P.load_library()
    return P


def _tet(rng, kind, aspect, tip):
    """A positively oriented tetrahedron whose node `tip` is the one off the base triangle."""
    z = aspect if kind == "spire" else 1.0 / aspect
    X = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0.3, 0.3, z]]) + 0.05 * rng.standard_normal((4, 3)) * [1, 1, min(1, z)]
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    X = X @ q.T
    order = [0, 1, 2]
    order.insert(tip, 3)
    X = X[order]
    if np.linalg.det(X[1:] - X[0]) < 0:
        a, b = [k for k in range(4) if k != tip][:2]
        X[[a, b]] = X[[b, a]]
    return X


def _gradients(rng):
    for node in range(4):
        s = slice(3 * node, 3 * node + 3)
        G = np.zeros((12, 12))
        G[s, s] = rng.standard_normal((3, 3))
        yield G
        G = rng.standard_normal((12, 12))
        G[s, s] *= 1e6
        yield G
    G = np.zeros((12, 12))
    G[rng.integers(12), rng.integers(12)] = 1.0
    yield G
    yield rng.standard_normal((12, 12))


def _cross(u, v):
    return np.array([u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]])


def reference(X, G):
    """(dE, dnu, dX) of one tetrahedron in extended precision, each with the size of its terms."""
    X, G, E, nu = X.astype(LD), G.astype(LD), LD(E0), LD(NU0)
    c = [_cross(X[3] - X[1], X[2] - X[1]), _cross(X[2] - X[0], X[3] - X[0]), _cross(X[3] - X[0], X[1] - X[0]),
         _cross(X[1] - X[0], X[2] - X[0])]
    det = (X[1] - X[0]) @ c[1]
    g, V = np.array([v / det for v in c]), det / 6
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    lam_nu, mu_nu = E * (1 + 2 * nu * nu) / ((1 + nu) * (1 - 2 * nu)) ** 2, -E / (2 * (1 + nu) ** 2)
    n = np.sqrt((g * g).sum(1))
    SA = SB = size = LD(0)
    h = np.zeros((4, 3), LD)
    for a in range(4):
        for b in range(4):
            B = G[3 * a:3 * a + 3, 3 * b:3 * b + 3]
            SA += g[a] @ B @ g[b]
            SB += g[b] @ B @ g[a] + np.trace(B) * (g[a] @ g[b])
            size += n[a] * n[b] * np.abs(B).sum()
            h[a] += lam * (B @ g[b]) + mu * (B.T @ g[b] + np.trace(B) * g[b])
            h[b] += lam * (B.T @ g[a]) + mu * (B @ g[a] + np.trace(B) * g[a])
    dX = np.array([V * ((lam * SA + mu * SB) * g[k] - sum((h[a] @ g[k]) * g[a] for a in range(4))) for k in range(4)])
    return ((V * (lam * SA + mu * SB) / E, V * (lam_nu * SA + mu_nu * SB), dX),
            (V * (lam + 2 * mu) / E * size, V * (lam_nu - 2 * mu_nu) * size, V * (lam + 2 * mu) * size * n))


def cases():
    rng = np.random.default_rng(3)
    return [(_tet(rng, kind, aspect, tip), G) for kind in ("spire", "flake") for aspect in (1, 10, 100)
            for tip in range(4) for G in _gradients(rng)]


def worst(got, X, G):
    """The largest error over the size of its terms, of dE, dnu and dX."""
    ref, size = reference(X, G)
    return max(abs(got[0] - ref[0]) / size[0], abs(got[1] - ref[1]) / size[1],
               (np.abs(got[2] - ref[2]).max(1) / size[2]).max())


def test_slender_tetrahedra(sta):
    """All cases in one mesh of separate tetrahedra, node ids in a random order in each."""
    import torch
    rng = np.random.default_rng(4)
    todo = cases()
    T = len(todo)
    X, tets = np.zeros((4 * T, 3)), np.zeros((T, 4), np.int32)
    for t, (x, _) in enumerate(todo):
        tets[t] = 4 * t + rng.permutation(4)
        X[tets[t]] = x
    asm = sta.Assembler(X, tets, np.full(T, E0), np.full(T, NU0))
    asm.full_rebuild(np.ones(T, np.uint8))
    rp, col, val = (a.cpu().numpy() for a in asm.csr())
    gv = np.zeros(val.size)
    for t, (_, G) in enumerate(todo):
        for p in range(12):
            r = 3 * tets[t, p // 3] + p % 3
            dof = {int(c): k for k, c in enumerate(col[rp[r]:rp[r + 1]])}
            for q in range(12):
                gv[rp[r] + dof[int(3 * tets[t, q // 3] + q % 3)]] = G[p, q]
    dE, dnu, dX = (a.cpu().numpy() for a in sta.sta_adjoint(asm.h, torch.as_tensor(gv, device="cuda")))
    for t, (x, G) in enumerate(todo):
        assert worst((dE[t], dnu[t], dX[tets[t]]), x, G) <= TOL, t
    asm.close()
