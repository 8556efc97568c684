// Element stiffness kernel: the 12x12 linear-tetrahedron elasticity matrix K^(tau)
// (STA-FEM Sec. 3.4 and Sec. 5.2; the standard P1 isotropic small-strain element,
// K = V B^T D B), 78 unique entries per tetrahedron written to the element cache.
//
// The evaluation order is fixed (see include/sta.h, sta_recompute_elements) and this file
// is compiled with --fmad=false: every fma below is an explicit __fma_rn, every other
// operation is a separately rounded IEEE double operation.  On GB300 the FP64 pipe is the
// scarce unit (about 0.5 Top/s against 35 Top/s of int32), so the order is also chosen to
// need few FP64 operations: about 300 per tetrahedron.
#include "sta_internal.cuh"

namespace sta {
namespace {

constexpr int EL_TPB = 128;

struct V3 {
    double x, y, z;
};

__device__ __forceinline__ V3 sub(const double4_32a &a, const double4_32a &b) {
    return {a.x - b.x, a.y - b.y, a.z - b.z};
}

// (u x v) with each component fma(u1, v2, -(u2 * v1))
__device__ __forceinline__ V3 cross_fma(const V3 &u, const V3 &v) {
    return {__fma_rn(u.y, v.z, -(u.z * v.y)), __fma_rn(u.z, v.x, -(u.x * v.z)),
            __fma_rn(u.x, v.y, -(u.y * v.x))};
}

__device__ __forceinline__ double gc(const V3 &g, int i) { return i == 0 ? g.x : (i == 1 ? g.y : g.z); }

// Computes the 78-entry record of one tetrahedron (node ids q) into rec[] (registers or shared
// memory).  Returns false when det <= 0 (record filled with zeros).
__device__ __forceinline__ bool element_record(double4_32a x0, double4_32a x1, double4_32a x2, double4_32a x3,
                                               double E, double nu, int4 q, double *rec) {
    const int gid[4] = {q.x, q.y, q.z, q.w};
    V3 d1 = sub(x1, x0), d2 = sub(x2, x0), d3 = sub(x3, x0);
    V3 c1 = cross_fma(d2, d3), c2 = cross_fma(d3, d1), c3 = cross_fma(d1, d2);
    double det = __fma_rn(d1.z, c1.z, __fma_rn(d1.y, c1.y, d1.x * c1.x));
    if (!(det > 0.0)) {
#pragma unroll
        for (int k = 0; k < KE_STRIDE; ++k) rec[k] = 0.0;
        return false;
    }
    double r = 1.0 / det;
    V3 g[4];
    g[1] = {c1.x * r, c1.y * r, c1.z * r};
    g[2] = {c2.x * r, c2.y * r, c2.z * r};
    g[3] = {c3.x * r, c3.y * r, c3.z * r};
    g[0] = {-((g[1].x + g[2].x) + g[3].x), -((g[1].y + g[2].y) + g[3].y),
            -((g[1].z + g[2].z) + g[3].z)};
    double V = det / 6.0;
    double onu = 1.0 + nu;
    double lam = (E * nu) / (onu * (1.0 - (nu + nu)));
    double mu = E / (onu + onu);
    double Vl = V * lam, Vm = V * mu;
    double P[4][3], Q[4][3];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            P[a][i] = Vl * gc(g[a], i);
            Q[a][i] = Vm * gc(g[a], i);
        }
    // diagonal blocks (a, a), entries i <= j
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        double D = Vm * __fma_rn(g[a].z, g[a].z, __fma_rn(g[a].y, g[a].y, g[a].x * g[a].x));
        double *o = rec + ke_diag_off(a);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                double v = (i != j)
                               ? __fma_rn(P[a][i], gc(g[a], j), Q[a][j] * gc(g[a], i))
                               : __fma_rn(P[a][i], gc(g[a], i), __fma_rn(Q[a][i], gc(g[a], i), D));
                o[ke_tri(i, j)] = v;
            }
    }
    // off-diagonal blocks (a, b), a < b, all (i, j)
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a + 1; b < 4; ++b) {
            double D = Vm * __fma_rn(g[a].z, g[b].z, __fma_rn(g[a].y, g[b].y, g[a].x * g[b].x));
            double *o = rec + ke_off_off(a, b);
            const bool tr = gid[a] > gid[b];  // run stored with the lower node id's rows
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    double v = (i != j)
                                   ? __fma_rn(P[a][i], gc(g[b], j), Q[a][j] * gc(g[b], i))
                                   : __fma_rn(P[a][i], gc(g[b], i), __fma_rn(Q[a][i], gc(g[b], i), D));
                    o[tr ? 3 * j + i : 3 * i + j] = v;
                }
            o[9] = 0.0;  // pad to a 16-byte aligned run
        }
    return true;
}

// New positions and materials (device arrays, null: kept) into the context's padded layout, and
// the element kernel's counters reset.  One thread per node and per tetrahedron; a pitched copy
// per array (24- and 8-byte rows) took 128 us for 384,000 tetrahedra, this 8 us.
__global__ void k_pack_params(const double *__restrict__ nodes, const double *__restrict__ young,
                              const double *__restrict__ poisson, int64_t n, int64_t T,
                              double4_32a *__restrict__ X, double2 *__restrict__ mat,
                              unsigned long long *counters) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (tid == 0) {
        counters[0] = counters[1] = 0ull;
        counters[2] = ~0ull;
    }
    if (nodes)
        for (int64_t v = tid; v < n; v += stride) {
            double4_32a p;
            p.x = nodes[3 * v];
            p.y = nodes[3 * v + 1];
            p.z = nodes[3 * v + 2];
            p.w = 0.0;
            X[v] = p;
        }
    if (young || poisson)
        for (int64_t t = tid; t < T; t += stride) {
            double2 m = young && poisson ? make_double2(0.0, 0.0) : mat[t];
            if (young) m.x = young[t];
            if (poisson) m.y = poisson[t];
            mat[t] = m;
        }
}

// Active tetrahedra, unordered: the FP64 kernels below run over this list so that every FP64
// instruction carries full lanes when part of the superset is inactive.  Four tetrahedra a thread
// (one mask word), one append per CTA of 1024 (appending warp by warp, 12,000 atomics on one word
// took 10 us for 384,000 tetrahedra).  With dE non-null, the adjoint outputs of inactive tets are
// zeroed on the way.
constexpr int AL_TPB = 256;

__global__ void __launch_bounds__(AL_TPB)
k_active_list(const uint8_t *__restrict__ mask, int64_t T, int32_t *__restrict__ list,
              unsigned long long *count, double *__restrict__ dE, double *__restrict__ dnu,
              double *__restrict__ dXe) {
    __shared__ int s_cnt[AL_TPB / 32];
    __shared__ unsigned long long s_base;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * (4 * AL_TPB);
    for (int64_t i0 = (int64_t)blockIdx.x * (4 * AL_TPB); i0 < T; i0 += stride) {  // CTA-uniform
        const int64_t t = i0 + 4 * threadIdx.x;
        unsigned act = 0, in = 0;  // bit k: tet t + k is active, exists
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t + k < T) {
                in |= 1u << k;
                if (__ldg(mask + t + k)) act |= 1u << k;
            }
        if (dE && in & ~act) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((in & ~act) >> k & 1) {
                    dE[t + k] = 0.0;
                    dnu[t + k] = 0.0;
#pragma unroll
                    for (int e = 0; e < 6; ++e)
                        reinterpret_cast<double2 *>(dXe + 12 * (t + k))[e] = make_double2(0.0, 0.0);
                }
        }
        const int own = __popc(act);
        int pre = own;  // inclusive prefix over the warp
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, pre, o);
            if (lane >= o) pre += y;
        }
        if (lane == 31) s_cnt[wid] = pre;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int w = 0; w < AL_TPB / 32; ++w) {
                const int c = s_cnt[w];
                s_cnt[w] = tot;
                tot += c;
            }
            s_base = tot ? atomicAdd(count, (unsigned long long)tot) : 0ull;
        }
        __syncthreads();
        int32_t *out = list + s_base + s_cnt[wid] + (pre - own);
        __syncthreads();  // s_cnt and s_base are rewritten in the next round
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (act >> k & 1) *out++ = (int32_t)(t + k);
    }
}

// Element records of tets list[0 .. *count) (or of all tets 0 .. T-1 when list is null), one
// per thread, staged per warp in shared memory and written out as contiguous records.
__global__ void __launch_bounds__(EL_TPB)
k_elements(const double4_32a *__restrict__ X, const int4 *__restrict__ tets,
           const double2 *__restrict__ mat, const int32_t *__restrict__ list,
           const unsigned long long *__restrict__ count, int64_t T, double *__restrict__ Ke,
           unsigned long long *bad) {
    extern __shared__ double smem[];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double *wrec = smem + (size_t)wid * 32 * KE_STRIDE;
    const int64_t n = list ? (int64_t)*count : T;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {  // block-uniform
        const int64_t i = base + threadIdx.x;
        const bool doit = i < n;
        const int32_t t = doit ? (list ? list[i] : (int32_t)i) : 0;
        if (doit) {
            const int4 q = tets[t];
            const double2 m = mat[t];
            const bool ok = element_record(X[q.x], X[q.y], X[q.z], X[q.w], m.x, m.y, q,
                                           wrec + (size_t)lane * KE_STRIDE);
            if (!ok) {
                atomicAdd(&bad[0], 1ull);
                atomicMin(&bad[2], (unsigned long long)t);
            }
        }
        unsigned todo = __ballot_sync(FULL, doit);
        __syncwarp();
        while (todo) {  // coalesced copy-out, one record at a time, to its diagonal and pair rows
            const int r = __ffs(todo) - 1;
            todo &= todo - 1;
            const int32_t tr = __shfl_sync(FULL, t, r);
            const double2 *src = reinterpret_cast<const double2 *>(wrec + (size_t)r * KE_STRIDE);
            double2 *dd = reinterpret_cast<double2 *>(Ke + ke_diag_at(T, tr, 0));
            double2 *dp = reinterpret_cast<double2 *>(Ke + ke_pair_at(T, tr, 0));
            for (int k = lane; k < KE_STRIDE / 2; k += 32) {
                if (k < KE_DIAG / 2)
                    dd[k] = src[k];
                else
                    dp[k - KE_DIAG / 2] = src[k];
            }
        }
        __syncwarp();
    }
}


// y = A x over the context's CSR (one thread per row, ascending columns).
__global__ void k_spmv(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                       const double *__restrict__ val, const double *__restrict__ x, int64_t nrows,
                       double *__restrict__ y) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
         r += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int32_t k = row_ptr[r]; k < row_ptr[r + 1]; ++k) s += val[k] * x[col[k]];
        y[r] = s;
    }
}

// Expand cached records of selected tetrahedra to full 12x12 row-major matrices.
__global__ void k_expand(const double *__restrict__ Ke, const int4 *__restrict__ tets, int64_t T,
                         const int32_t *ids, int64_t n, double *out) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < 144 * n;
         k += (int64_t)gridDim.x * blockDim.x) {
        int64_t e = k / 144;
        int pq = (int)(k % 144), p = pq / 12, q = pq % 12;
        int32_t t = ids[e];
        if (t < 0 || t >= T) {
            out[k] = 0.0;
            continue;
        }
        int a = p / 3, i = p % 3, b = q / 3, j = q % 3;
        if (a > b || (a == b && i > j)) {  // mirror into the stored upper triangle
            int ta = a, ti = i;
            a = b; i = j; b = ta; j = ti;
        }
        const int4 tq = tets[t];
        const int gid[4] = {tq.x, tq.y, tq.z, tq.w};
        const double *dg = Ke + ke_diag_at(T, t, a), *pr = Ke + ke_pair_at(T, t, ke_pair(a, b));
        out[k] = (a == b)             ? dg[ke_tri(i, j)]
                 : gid[a] < gid[b] ? pr[3 * i + j]
                                   : pr[3 * j + i];
    }
}

}  // namespace

int launch_pack_params(Ctx *c, const double *nodes, const double *young, const double *poisson,
                       cudaStream_t s) {
    const int64_t items = c->T > c->n ? c->T : c->n;
    int64_t grid = (items + 255) / 256;
    const int64_t cap = (int64_t)c->num_sms * 8;
    grid = grid < 1 ? 1 : (grid > cap ? cap : grid);
    k_pack_params<<<(unsigned)grid, 256, 0, s>>>(nodes, young, poisson, c->n, c->T, c->X, c->mat,
                                                 c->counters);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

// The unordered list of active tets (c->act_list, count in c->act_count), allocated on first use.
int launch_active_list(Ctx *c, double *dE, double *dnu, double *dXe, cudaStream_t s) {
    if (!c->act_list) {
        STA_TRY(dev_alloc(c, &c->act_list, c->T));
        STA_TRY(dev_alloc(c, &c->act_count, 1));
    }
    STA_CUDA_TRY(cudaMemsetAsync(c->act_count, 0, sizeof(unsigned long long), s));
    int64_t grid = (c->T + 4 * AL_TPB - 1) / (4 * AL_TPB);
    const int64_t cap = (int64_t)c->num_sms * 8;
    if (grid > cap) grid = cap;
    k_active_list<<<(unsigned)grid, AL_TPB, 0, s>>>(c->mask, c->T, c->act_list, c->act_count, dE,
                                                 dnu, dXe);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

int launch_elements(Ctx *c, bool active_only, cudaStream_t s) {
    if (c->T == 0) return STA_OK;
    size_t smem = (size_t)EL_TPB * KE_STRIDE * sizeof(double);  // 84 KB
    STA_CUDA_TRY(cudaFuncSetAttribute(k_elements, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
    if (active_only) STA_TRY(launch_active_list(c, nullptr, nullptr, nullptr, s));
    int64_t blocks = (c->T + EL_TPB - 1) / EL_TPB;
    int per_sm = 0;
    STA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_elements, EL_TPB, smem));
    if (per_sm < 1) per_sm = 1;
    int64_t cap = (int64_t)per_sm * c->num_sms;
    if (blocks > cap) blocks = cap;
    k_elements<<<(unsigned)blocks, EL_TPB, smem, s>>>(c->X, c->tets, c->mat,
                                                      active_only ? c->act_list : nullptr,
                                                      active_only ? c->act_count : nullptr, c->T,
                                                      c->Ke, c->counters);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

int launch_spmv(Ctx *c, const double *val, const double *x, double *y, cudaStream_t s) {
    if (c->nrows == 0) return STA_OK;
    int64_t grid = (c->nrows + 255) / 256;
    const int64_t cap = (int64_t)c->num_sms * 16;
    if (grid > cap) grid = cap;
    k_spmv<<<(unsigned)grid, 256, 0, s>>>(c->row_ptr, c->col, val, x, c->nrows, y);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

int launch_expand_elements(Ctx *c, const int32_t *ids, int64_t n, double *out, cudaStream_t s) {
    if (n == 0) return STA_OK;
    int64_t items = 144 * n;
    int64_t blocks = (items + 255) / 256;
    if (blocks > 65535LL * 16) blocks = 65535LL * 16;
    k_expand<<<(unsigned)blocks, 256, 0, s>>>(c->Ke, c->tets, c->T, ids, n, out);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

}  // namespace sta
