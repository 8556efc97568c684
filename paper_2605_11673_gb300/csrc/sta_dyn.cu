// Implicit-Euler dynamic loop on the maintained operator (STA-FEM Sec. 6.2, Eq. 9):
//     (M_t + h^2 K_t) u_{t+1} = M_t (u_t + h v_t) + h^2 f,   v_{t+1} = (u_{t+1} - u_t) / h,
// K_t the context's maintained values (eps included), M_t a maintained lumped mass.
//
// Lumped mass (the paper gives no formula): row-sum lumping of the consistent P1 mass, each
// active tetrahedron gives (rho V) / 4 to each of its nodes (every DOF of the node), folded per
// node from +0.0 in ascending tetrahedron id -- the canonical order of the stiffness, so the
// maintained mass equals a rebuild bit for bit.  V = det / 6 with det in the element matrix's
// fixed order.  The per-tet quarter masses are computed once (sta_dyn_setup, sta_set_params);
// a streaming frame re-folds the nodes of its edited tetrahedra after the mask update; a
// rebuild re-folds every node.
//
// Solve: conjugate gradients with the Jacobi preconditioner (sta_cg.cu) on the free DOFs -- not
// clamped, of a node with mass; a clamped DOF stays 0, a DOF of a node without mass keeps its
// displacement with velocity 0.  Start: x = u_t.  Stop: ||r|| <= tol ||b|| or max_iter.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sta_internal.cuh"

namespace sta {
namespace {

constexpr int DYN_TPB = 256;

// -------------------------------------------------------------------------------- mass

__global__ void k_dyn_qmass(const double4_32a *__restrict__ X, const int4 *__restrict__ tets,
                            int64_t T, double rho, double *__restrict__ qmass) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int4 q = tets[t];
        const double4_32a x0 = X[q.x], x1 = X[q.y], x2 = X[q.z], x3 = X[q.w];
        const double d1x = x1.x - x0.x, d1y = x1.y - x0.y, d1z = x1.z - x0.z;
        const double d2x = x2.x - x0.x, d2y = x2.y - x0.y, d2z = x2.z - x0.z;
        const double d3x = x3.x - x0.x, d3y = x3.y - x0.y, d3z = x3.z - x0.z;
        // c_1 = d_2 x d_3, det = d_1 . c_1 (the element matrix's order)
        const double cx = __fma_rn(d2y, d3z, -(d2z * d3y));
        const double cy = __fma_rn(d2z, d3x, -(d2x * d3z));
        const double cz = __fma_rn(d2x, d3y, -(d2y * d3x));
        const double det = __fma_rn(d1z, cz, __fma_rn(d1y, cy, d1x * cx));
        qmass[t] = (rho * (det / 6.0)) * 0.25;
    }
}

__device__ __forceinline__ double node_mass(int32_t a, const int32_t *__restrict__ nt_ptr,
                                            const int32_t *__restrict__ nt_list,
                                            const uint8_t *__restrict__ mask,
                                            const double *__restrict__ qmass) {
    double m = 0.0;
    for (int32_t q = nt_ptr[a]; q < nt_ptr[a + 1]; ++q) {
        const int32_t t = nt_list[q];
        if (mask[t]) m += qmass[t];
    }
    return m;
}

// Lumped mass of every node: the fold of its active tetrahedra's quarter masses, ascending
// tetrahedron id, from +0.0.
__global__ void k_dyn_mass_all(int64_t n, const int32_t *__restrict__ nt_ptr,
                               const int32_t *__restrict__ nt_list, const uint8_t *__restrict__ mask,
                               const double *__restrict__ qmass, double *__restrict__ mass) {
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n;
         a += (int64_t)gridDim.x * blockDim.x)
        mass[a] = node_mass((int32_t)a, nt_ptr, nt_list, mask, qmass);
}

// The nodes of the frame's edited tetrahedra, after the mask update.  A node shared by several
// edited tetrahedra is re-folded by each of them; all read the same mask and write the same
// value.
__global__ void k_dyn_mass_edited(const int32_t *__restrict__ edited, int64_t m,
                                  const int64_t *__restrict__ m_dev, const int4 *__restrict__ tets,
                                  const int32_t *__restrict__ nt_ptr,
                                  const int32_t *__restrict__ nt_list,
                                  const uint8_t *__restrict__ mask,
                                  const double *__restrict__ qmass, double *__restrict__ mass) {
    const int64_t items = 4 * (m_dev ? *m_dev : m);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = (uint32_t)edited[i >> 2] & 0x7fffffffu;
        const int4 q = tets[t];
        const int j = (int)(i & 3);
        const int32_t a = j == 0 ? q.x : (j == 1 ? q.y : (j == 2 ? q.z : q.w));
        mass[a] = node_mass(a, nt_ptr, nt_list, mask, qmass);
    }
}

// -------------------------------------------------------------------------------- CG

// b, x0 = u, Jacobi inverse diagonal and the free flags, per DOF.
__global__ void k_cg_init(int64_t n3, const int32_t *__restrict__ adj_ptr,
                          const int32_t *__restrict__ adj, const int32_t *__restrict__ row_ptr,
                          const double *__restrict__ val, const double *__restrict__ mass,
                          const uint8_t *__restrict__ clamped, const double *__restrict__ u,
                          const double *__restrict__ v, const double *__restrict__ f, double h,
                          double *__restrict__ x, double *__restrict__ b,
                          double *__restrict__ dinv, uint8_t *__restrict__ fr) {
    const double h2 = h * h;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = (int32_t)(i / 3), k = (int32_t)(i - 3 * (int64_t)a);
        const double m = mass[a];
        const bool free = !clamped[a] && m > 0.0;
        fr[i] = free ? 1 : 0;
        if (!free) {
            x[i] = 0.0;
            b[i] = 0.0;
            dinv[i] = 0.0;
            continue;
        }
        int32_t lo = adj_ptr[a], hi = adj_ptr[a + 1];  // the diagonal block of node a
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (adj[mid] < a) lo = mid + 1; else hi = mid;
        }
        const double kii = val[row_ptr[i] + 3 * (lo - adj_ptr[a]) + k];
        x[i] = u[i];
        b[i] = m * (u[i] + h * v[i]) + h2 * f[i];
        dinv[i] = 1.0 / (m + h2 * kii);
    }
}

// q = A x on the free DOFs (0 elsewhere), four lanes per node over its three rows (they share
// their columns): lane j of the quad takes the entries j, j + 4, ... of each row, ascending,
// and the quad adds its four partial sums as (s0 + s1) + (s2 + s3).  GB300 issues an FP64
// instruction for a whole warp whatever its active lanes, and the FP64 pipe is the scarce unit
// here, so every lane works on its own entries and the only cross-lane adds are the two quad
// levels.  The nodes are taken in the order `perm` (ascending row length), so that the eight
// nodes of a warp have rows of nearly one length.
__global__ void __launch_bounds__(DYN_TPB)
k_dyn_spmv(int64_t n, const int32_t *__restrict__ perm, const int32_t *__restrict__ row_ptr,
           const int32_t *__restrict__ col, const double *__restrict__ val,
           const double *__restrict__ mass, double h2, const uint8_t *__restrict__ fr,
           const double *__restrict__ xin, double *__restrict__ qout) {
    const int lane = threadIdx.x & 31, qd = lane & 3;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = 8 * warp; base < n; base += 8 * nwarps) {  // warp-uniform
        const int64_t j = base + (lane >> 2);
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        int64_t a = -1;
        if (j < n) {
            a = perm[j];
            const int32_t r0 = row_ptr[3 * a], len = (row_ptr[3 * a + 3] - r0) / 3;
            const int32_t r1 = r0 + len, r2 = r1 + len;
            int32_t k = qd;
            for (; k + 12 < len; k += 16) {
                int32_t cj[4];
                double v0[4], v1[4], v2[4], xj[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    cj[u] = col[r0 + k + 4 * u];
                    v0[u] = val[r0 + k + 4 * u];
                    v1[u] = val[r1 + k + 4 * u];
                    v2[u] = val[r2 + k + 4 * u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) xj[u] = xin[cj[u]];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    s0 = __fma_rn(v0[u], xj[u], s0);
                    s1 = __fma_rn(v1[u], xj[u], s1);
                    s2 = __fma_rn(v2[u], xj[u], s2);
                }
            }
            for (; k < len; k += 4) {
                const double xj = xin[col[r0 + k]];
                s0 = __fma_rn(val[r0 + k], xj, s0);
                s1 = __fma_rn(val[r1 + k], xj, s1);
                s2 = __fma_rn(val[r2 + k], xj, s2);
            }
        }
        for (int o = 1; o <= 2; o <<= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (a >= 0 && qd < 3) {
            const int64_t d = 3 * a + qd;
            const double sd = qd == 0 ? s0 : (qd == 1 ? s1 : s2);
            qout[d] = fr[d] ? __fma_rn(mass[a], xin[d], h2 * sd) : 0.0;
        }
    }
}

// Static solve (sta_solve): b, x0 and the Jacobi inverse diagonal on the caller's free DOFs.
__global__ void k_cg_init_static(int64_t n3, const int32_t *__restrict__ adj_ptr,
                                 const int32_t *__restrict__ adj,
                                 const int32_t *__restrict__ row_ptr,
                                 const double *__restrict__ val, const uint8_t *__restrict__ free_in,
                                 const double *__restrict__ b_in, const double *__restrict__ x_in,
                                 double *__restrict__ x, double *__restrict__ b,
                                 double *__restrict__ dinv, uint8_t *__restrict__ fr) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = (int32_t)(i / 3), k = (int32_t)(i - 3 * (int64_t)a);
        double kii = 0.0;
        if (free_in[i] && adj_ptr[a + 1] > adj_ptr[a]) {
            int32_t lo = adj_ptr[a], hi = adj_ptr[a + 1];  // the diagonal block of node a
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if (adj[mid] < a) lo = mid + 1; else hi = mid;
            }
            kii = val[row_ptr[i] + 3 * (lo - adj_ptr[a]) + k];
        }
        const bool free = free_in[i] && kii != 0.0;  // a free DOF needs a diagonal
        fr[i] = free ? 1 : 0;
        x[i] = free ? x_in[i] : 0.0;
        b[i] = free ? b_in[i] : 0.0;
        dinv[i] = free ? 1.0 / kii : 0.0;
    }
}

// Static solve of the scalar proxy operator (one row per node): b, x0 and the inverse diagonal.
__global__ void k_cg_init_scalar(int64_t n, const int32_t *__restrict__ pdiag,
                                 const double *__restrict__ val, const uint8_t *__restrict__ free_in,
                                 const double *__restrict__ b_in, const double *__restrict__ x_in,
                                 double *__restrict__ x, double *__restrict__ b,
                                 double *__restrict__ dinv, uint8_t *__restrict__ fr) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t g = pdiag[i];
        const double kii = free_in[i] && g >= 0 ? val[g] : 0.0;
        const bool free = kii != 0.0;
        fr[i] = free ? 1 : 0;
        x[i] = free ? x_in[i] : 0.0;
        b[i] = free ? b_in[i] : 0.0;
        dinv[i] = free ? 1.0 / kii : 0.0;
    }
}

// The adjoint rule of a solve (A_ff u_f = f_f): dL/dA_ij = -lam_i u_j on entries between free
// DOFs, 0 elsewhere.  One thread per row.
__global__ void k_outer_grad(int64_t nrows, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const double *__restrict__ lam,
                             const double *__restrict__ u, const uint8_t *__restrict__ free,
                             double *__restrict__ g) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nrows;
         i += (int64_t)gridDim.x * blockDim.x) {
        const bool fi = free[i] != 0;
        const double li = -lam[i];
        for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) {
            const int32_t j = col[k];
            g[k] = fi && free[j] ? li * u[j] : 0.0;
        }
    }
}

// x restricted to the free DOFs (0 elsewhere), with the free flags from mass and clamping.
__global__ void k_dyn_restrict(int64_t n3, const double *__restrict__ mass,
                               const uint8_t *__restrict__ clamped, const double *__restrict__ x,
                               double *__restrict__ xf, uint8_t *__restrict__ fr) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = i / 3;
        const bool free = !clamped[a] && mass[a] > 0.0;
        fr[i] = free ? 1 : 0;
        xf[i] = free ? x[i] : 0.0;
    }
}

unsigned dyn_grid(const Ctx *c, int64_t items, int per_sm = 4) {
    int64_t g = (items + DYN_TPB - 1) / DYN_TPB;
    const int64_t cap = (int64_t)c->num_sms * per_sm;
    if (g > cap) g = cap;
    return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

// ------------------------------------------------------------------------------ launchers

int launch_dyn_mass_all(Ctx *c, cudaStream_t s) {
    if (!c->dyn || c->n == 0) return STA_OK;
    k_dyn_mass_all<<<dyn_grid(c, c->n), DYN_TPB, 0, s>>>(c->n, c->nt_ptr, c->nt_list, c->mask,
                                                         c->qmass, c->mass);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

int launch_dyn_mass_edited(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev,
                           int64_t cap, cudaStream_t s) {
    if (!c->dyn) return STA_OK;
    k_dyn_mass_edited<<<dyn_grid(c, 4 * (cap > 0 ? cap : 1), 8), DYN_TPB, 0, s>>>(
        edited, m, m_dev, c->tets, c->nt_ptr, c->nt_list, c->mask, c->qmass, c->mass);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

int launch_dyn_qmass(Ctx *c, cudaStream_t s) {
    if (!c->dyn || c->T == 0) return STA_OK;
    k_dyn_qmass<<<dyn_grid(c, c->T, 8), DYN_TPB, 0, s>>>(c->X, c->tets, c->T, c->dyn_rho, c->qmass);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

// sta_dyn_apply's node order: ascending row length (ties by node id).
static int dyn_order(Ctx *c) {
    if (c->dyn_perm) return STA_OK;
    const int64_t n = c->n;
    STA_TRY(dev_alloc(c, &c->dyn_perm, n));
    std::vector<int32_t> rp(3 * n + 1), perm(n);
    STA_CUDA_TRY(cudaMemcpy(rp.data(), c->row_ptr, sizeof(int32_t) * (3 * n + 1), cudaMemcpyDeviceToHost));
    for (int64_t a = 0; a < n; ++a) perm[a] = (int32_t)a;
    std::stable_sort(perm.begin(), perm.end(), [&](int32_t p, int32_t q) {
        return rp[3 * p + 3] - rp[3 * p] < rp[3 * q + 3] - rp[3 * q];
    });
    STA_CUDA_TRY(cudaMemcpy(c->dyn_perm, perm.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice));
    return STA_OK;
}

}  // namespace sta

using namespace sta;

extern "C" int sta_dyn_setup(sta_ctx *x, double rho, double h, const double *f,
                             const uint8_t *clamped, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (c->op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    if (c->graph_on) return fail(STA_ESTATE, "disable graph mode before setting up the dynamics");
    if (!(rho > 0.0) || !(h > 0.0) || !std::isfinite(rho) || !std::isfinite(h))
        return fail(STA_EINVAL, "rho and h must be positive and finite");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = c->n, n3 = 3 * n;
    if (!c->qmass) {
        STA_TRY(dev_alloc(c, &c->qmass, c->T));
        STA_TRY(dev_alloc(c, &c->mass, n));
        STA_TRY(dev_alloc(c, &c->du, n3));
        STA_TRY(dev_alloc(c, &c->dv, n3));
        STA_TRY(dev_alloc(c, &c->df, n3));
        STA_TRY(dev_alloc(c, &c->clamped, n));
    }
    STA_TRY(cg_alloc(c));
    STA_TRY(dyn_order(c));
    std::vector<double> hf(n3 > 0 ? n3 : 1, 0.0);
    std::vector<uint8_t> hc(n > 0 ? n : 1, 0);
    if (f) std::copy(f, f + n3, hf.begin());
    if (clamped)
        for (int64_t a = 0; a < n; ++a) hc[a] = clamped[a] ? 1 : 0;
    STA_CUDA_TRY(cudaMemcpyAsync(c->df, hf.data(), sizeof(double) * n3, cudaMemcpyHostToDevice, s));
    STA_CUDA_TRY(cudaMemcpyAsync(c->clamped, hc.data(), (size_t)n, cudaMemcpyHostToDevice, s));
    STA_CUDA_TRY(cudaMemsetAsync(c->du, 0, sizeof(double) * (size_t)(n3 > 0 ? n3 : 1), s));
    STA_CUDA_TRY(cudaMemsetAsync(c->dv, 0, sizeof(double) * (size_t)(n3 > 0 ? n3 : 1), s));
    c->dyn = true;
    c->dyn_rho = rho;
    c->dyn_h = h;
    STA_TRY(launch_dyn_qmass(c, s));
    STA_TRY(launch_dyn_mass_all(c, s));
    STA_CUDA_TRY(cudaStreamSynchronize(s));  // the host vectors go out of scope
    return STA_OK;
}

extern "C" int sta_dyn_step(sta_ctx *x, double tol, int32_t max_iter, int32_t *iters,
                            double *rel_res, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (!c->dyn) return fail(STA_ESTATE, "call sta_dyn_setup first");
    if (!(tol >= 0.0) || max_iter < 0) return fail(STA_EINVAL, "tol and max_iter must be >= 0");
    STA_TRY(check_values(c));
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n3 = 3 * c->n;
    CgResult res{};
    if (n3 > 0) {
        k_cg_init<<<dyn_grid(c, n3), DYN_TPB, 0, s>>>(n3, c->adj_ptr, c->adj, c->row_ptr, c->val, c->mass,
                                                      c->clamped, c->du, c->dv, c->df, c->dyn_h, c->cg,
                                                      c->cg + n3, c->cg + 2 * n3, c->cg_free);
        STA_CUDA_TRY(cudaGetLastError());
        STA_TRY(launch_cg_solve(c, c->val, c->mass, c->dyn_h * c->dyn_h, tol, max_iter, false, nullptr,
                                s, &res));
    }
    STA_TRY(check_values(c));  // (a rebuild that was still running before)
    if (iters) *iters = res.iters;
    if (rel_res) *rel_res = res.bb > 0.0 ? std::sqrt(res.rr / res.bb) : 0.0;
    return STA_OK;
}

extern "C" int sta_dyn_apply(sta_ctx *x, const double *xv, double *y, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (!c->dyn) return fail(STA_ESTATE, "call sta_dyn_setup first");
    const int64_t n3 = 3 * c->n;
    if (n3 == 0) return STA_OK;
    if (!xv || !y) return fail(STA_EINVAL, "NULL argument");
    STA_TRY(check_values(c));
    cudaStream_t s = (cudaStream_t)stream;
    double *xf = c->cg + 3 * n3;  // the solve's z buffer (free between steps)
    const unsigned gv = dyn_grid(c, n3);
    k_dyn_restrict<<<gv, DYN_TPB, 0, s>>>(n3, c->mass, c->clamped, xv, xf, c->cg_free);
    k_dyn_spmv<<<gv, DYN_TPB, 0, s>>>(c->n, c->dyn_perm, c->row_ptr, c->col, c->val, c->mass,
                                     c->dyn_h * c->dyn_h, c->cg_free, xf, y);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

extern "C" int sta_solve(sta_ctx *x, const double *val, const double *b, const uint8_t *free,
                         double tol, int32_t max_iter, double *xv, int32_t *iters,
                         double *rel_res, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (!(tol >= 0.0) || max_iter < 0) return fail(STA_EINVAL, "tol and max_iter must be >= 0");
    const int64_t n3 = c->nrows;  // DOFs: 3 per node, or 1 for the proxy operator
    if (n3 > 0 && (!b || !free || !xv)) return fail(STA_EINVAL, "NULL argument");
    STA_TRY(check_values(c));
    cudaStream_t s = (cudaStream_t)stream;
    STA_TRY(cg_alloc(c));
    const double *A = val ? val : c->val;
    CgResult res{};
    if (n3 > 0) {
        const unsigned gv = dyn_grid(c, n3);
        double *xw = c->cg, *bw = xw + n3, *dinv = bw + n3;
        if (c->op == STA_OP_PROXY)
            k_cg_init_scalar<<<gv, DYN_TPB, 0, s>>>(n3, c->pdiag, A, free, b, xv, xw, bw, dinv,
                                                    c->cg_free);
        else
            k_cg_init_static<<<gv, DYN_TPB, 0, s>>>(n3, c->adj_ptr, c->adj, c->row_ptr, A, free, b,
                                                    xv, xw, bw, dinv, c->cg_free);
        STA_CUDA_TRY(cudaGetLastError());
        STA_TRY(launch_cg_solve(c, A, nullptr, 1.0, tol, max_iter, true, xv, s, &res));
    }
    STA_TRY(check_values(c));  // (a rebuild that was still running before)
    if (iters) *iters = res.iters;
    if (rel_res) *rel_res = res.bb > 0.0 ? std::sqrt(res.rr / res.bb) : 0.0;
    return STA_OK;
}

extern "C" int sta_outer_grad(sta_ctx *x, const double *lam, const double *u,
                              const uint8_t *free, double *grad_val, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (c->nrows > 0 && (!lam || !u || !free || !grad_val)) return fail(STA_EINVAL, "NULL argument");
    if (c->nrows == 0) return STA_OK;
    const unsigned g = dyn_grid(c, c->nrows, 8);
    k_outer_grad<<<g, DYN_TPB, 0, (cudaStream_t)stream>>>(c->nrows, c->row_ptr, c->col, lam, u,
                                                          free, grad_val);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

extern "C" int sta_dyn_state(const sta_ctx *x, const double **u, const double **v,
                             const double **mass) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (!x->c.dyn) return fail(STA_ESTATE, "call sta_dyn_setup first");
    if (u) *u = x->c.du;
    if (v) *v = x->c.dv;
    if (mass) *mass = x->c.mass;
    return STA_OK;
}

extern "C" int sta_dyn_set_state(sta_ctx *x, const double *u, const double *v, int on_device,
                                 void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (!c->dyn) return fail(STA_ESTATE, "call sta_dyn_setup first");
    const size_t bytes = sizeof(double) * 3 * (size_t)c->n;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    cudaStream_t s = (cudaStream_t)stream;
    if (u) STA_CUDA_TRY(cudaMemcpyAsync(c->du, u, bytes, kind, s));
    if (v) STA_CUDA_TRY(cudaMemcpyAsync(c->dv, v, bytes, kind, s));
    if (!on_device) STA_CUDA_TRY(cudaStreamSynchronize(s));
    return STA_OK;
}
