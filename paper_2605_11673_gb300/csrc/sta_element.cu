// Element stiffness kernel: the 12x12 linear-tetrahedron elasticity matrix K^(tau)
// (STA-FEM Sec. 3.4 and Sec. 5.2; the standard P1 isotropic small-strain element,
// K = V B^T D B), 78 unique entries per tetrahedron written to the element cache as 10 runs.
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

// What the entries of one element matrix are formed from: barycentric gradients g, P = V lam g,
// Q = V mu g, V mu.
struct Element {
    V3 g[4], P[4], Q[4];
    double Vm;
};

// Returns false when det <= 0 (everything zero: a zero matrix).
__device__ __forceinline__ bool element(double4_32a x0, double4_32a x1, double4_32a x2,
                                        double4_32a x3, double E, double nu, Element &e) {
    V3 d1 = sub(x1, x0), d2 = sub(x2, x0), d3 = sub(x3, x0);
    V3 c1 = cross_fma(d2, d3), c2 = cross_fma(d3, d1), c3 = cross_fma(d1, d2);
    double det = __fma_rn(d1.z, c1.z, __fma_rn(d1.y, c1.y, d1.x * c1.x));
    if (!(det > 0.0)) {
#pragma unroll
        for (int a = 0; a < 4; ++a) e.g[a] = e.P[a] = e.Q[a] = {0.0, 0.0, 0.0};
        e.Vm = 0.0;
        return false;
    }
    double r = 1.0 / det;
    e.g[1] = {c1.x * r, c1.y * r, c1.z * r};
    e.g[2] = {c2.x * r, c2.y * r, c2.z * r};
    e.g[3] = {c3.x * r, c3.y * r, c3.z * r};
    e.g[0] = {-((e.g[1].x + e.g[2].x) + e.g[3].x), -((e.g[1].y + e.g[2].y) + e.g[3].y),
              -((e.g[1].z + e.g[2].z) + e.g[3].z)};
    double V = det / 6.0;
    double onu = 1.0 + nu;
    double lam = (E * nu) / (onu * (1.0 - (nu + nu)));
    double mu = E / (onu + onu);
    double Vl = V * lam;
    e.Vm = V * mu;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        e.P[a] = {Vl * e.g[a].x, Vl * e.g[a].y, Vl * e.g[a].z};
        e.Q[a] = {e.Vm * e.g[a].x, e.Vm * e.g[a].y, e.Vm * e.g[a].z};
    }
    return true;
}

// The local node with the largest gradient component, compared by high words (no FP64 operation):
// its gradient is the largest to within a factor of sqrt(3).  For the adjoint.
__device__ __forceinline__ int steepest(const Element &e) {
    int node = 0, most = -1;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int m = max(max(__double2hiint(e.g[a].x) & 0x7fffffff, __double2hiint(e.g[a].y) & 0x7fffffff),
                          __double2hiint(e.g[a].z) & 0x7fffffff);
        if (m > most) {
            most = m;
            node = a;
        }
    }
    return node;
}

// Entries of the block (a, b): a == b the 6 entries i <= j, else all 9, row-major, transposed when
// `tr` (a run is stored with the lower node id's rows).
template <int a, int b>
__device__ __forceinline__ void element_run(const Element &e, bool tr, double *o) {
    const V3 &ga = e.g[a], &gb = e.g[b];
    const double D = e.Vm * __fma_rn(ga.z, gb.z, __fma_rn(ga.y, gb.y, ga.x * gb.x));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = a == b ? i : 0; j < 3; ++j) {
            const double v =
                i != j ? __fma_rn(gc(e.P[a], i), gc(gb, j), gc(e.Q[a], j) * gc(gb, i))
                       : __fma_rn(gc(e.P[a], i), gc(gb, i), __fma_rn(gc(e.Q[a], i), gc(gb, i), D));
            if (a == b)
                o[ke_tri(i, j)] = v;
            else
                o[tr ? 3 * j + i : 3 * i + j] = v;
        }
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

// The warp's 32 runs of one slot from its buffer to the element cache: consecutive lanes write
// consecutive doubles of a run.
template <int N>
__device__ __forceinline__ void write_runs(const double *buf, int32_t off, double *__restrict__ Ke,
                                           int lane) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int e = 32 * k + lane, r = e / N;
        const int32_t o = __shfl_sync(0xffffffffu, off, r);
        if (o >= 0) Ke[o + (e - N * r)] = buf[e];
    }
    __syncwarp();
}

// Element matrices of tets list[0 .. *count) (or of all tets 0 .. T-1 when list is null), one per
// thread, written to the cache run by run.  Bound by the FP64 pipe: 307 instructions a tetrahedron.
// One run at a time is staged (2.3 KB a warp), so registers alone limit the CTAs of an SM and the
// quadrant's other warps compute while one writes; staging whole records (84 KB a CTA of 4 warps,
// 2 warps a quadrant) left the pipe idle a quarter of the time: 384,000 tetrahedra 257 -> 225 us
// (FP64 floor 190 us; with 3 CTAs an SM instead of 4, without the 64 spilled bytes: 236 us).
__global__ void __launch_bounds__(EL_TPB, 4)
k_elements(const double4_32a *__restrict__ X, const int4 *__restrict__ tets,
           const double2 *__restrict__ mat, const int32_t *__restrict__ list,
           const unsigned long long *__restrict__ count, int64_t T,
           const int32_t *__restrict__ krun, double *__restrict__ Ke, uint8_t *__restrict__ steep,
           unsigned long long *bad) {
    __shared__ double bufs[EL_TPB / 32][32 * RUN_PAIR];
    const int lane = threadIdx.x & 31;
    double *buf = bufs[threadIdx.x >> 5];
    const int64_t n = list ? (int64_t)*count : T;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
         base += (int64_t)gridDim.x * blockDim.x) {  // block-uniform
        const int64_t i = base + threadIdx.x;
        const bool doit = i < n;
        int32_t off[10];  // of the tet's runs; -1: none
        Element e;
        bool t01 = false, t02 = false, t03 = false, t12 = false, t13 = false, t23 = false;
        if (doit) {
            const int32_t t = list ? list[i] : (int32_t)i;
            const int4 q = tets[t];
            const double2 m = mat[t];
            const int2 *kr = reinterpret_cast<const int2 *>(krun + 10 * (int64_t)t);
#pragma unroll
            for (int h = 0; h < 5; ++h) {
                const int2 v = __ldg(kr + h);
                off[2 * h] = v.x;
                off[2 * h + 1] = v.y;
            }
            if (!element(X[q.x], X[q.y], X[q.z], X[q.w], m.x, m.y, e)) {
                atomicAdd(&bad[0], 1ull);
                atomicMin(&bad[2], (unsigned long long)t);
            }
            steep[t] = (uint8_t)steepest(e);
            t01 = q.x > q.y; t02 = q.x > q.z; t03 = q.x > q.w;
            t12 = q.y > q.z; t13 = q.y > q.w; t23 = q.z > q.w;
        } else {
#pragma unroll
            for (int h = 0; h < 10; ++h) off[h] = -1;
#pragma unroll
            for (int a = 0; a < 4; ++a) e.g[a] = e.P[a] = e.Q[a] = {0.0, 0.0, 0.0};
            e.Vm = 0.0;
        }
        double *d = buf + RUN_DIAG * lane, *p = buf + RUN_PAIR * lane;
        element_run<0, 0>(e, false, d); write_runs<RUN_DIAG>(buf, off[0], Ke, lane);
        element_run<1, 1>(e, false, d); write_runs<RUN_DIAG>(buf, off[1], Ke, lane);
        element_run<2, 2>(e, false, d); write_runs<RUN_DIAG>(buf, off[2], Ke, lane);
        element_run<3, 3>(e, false, d); write_runs<RUN_DIAG>(buf, off[3], Ke, lane);
        element_run<0, 1>(e, t01, p); write_runs<RUN_PAIR>(buf, off[4], Ke, lane);
        element_run<0, 2>(e, t02, p); write_runs<RUN_PAIR>(buf, off[5], Ke, lane);
        element_run<0, 3>(e, t03, p); write_runs<RUN_PAIR>(buf, off[6], Ke, lane);
        element_run<1, 2>(e, t12, p); write_runs<RUN_PAIR>(buf, off[7], Ke, lane);
        element_run<1, 3>(e, t13, p); write_runs<RUN_PAIR>(buf, off[8], Ke, lane);
        element_run<2, 3>(e, t23, p); write_runs<RUN_PAIR>(buf, off[9], Ke, lane);
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
__global__ void k_expand(const double *__restrict__ Ke, const int32_t *__restrict__ krun,
                         const int4 *__restrict__ tets, int64_t T, const int32_t *ids, int64_t n,
                         double *out) {
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
        const double *run = Ke + krun[10 * (int64_t)t + slot_of(a, b)];
        out[k] = run[a == b ? ke_tri(i, j) : (gid[a] < gid[b] ? 3 * i + j : 3 * j + i)];
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
    if (active_only) STA_TRY(launch_active_list(c, nullptr, nullptr, nullptr, s));
    int64_t blocks = (c->T + EL_TPB - 1) / EL_TPB;
    int per_sm = 0;
    STA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_elements, EL_TPB, 0));
    if (per_sm < 1) per_sm = 1;
    int64_t cap = (int64_t)per_sm * c->num_sms;
    if (blocks > cap) blocks = cap;
    k_elements<<<(unsigned)blocks, EL_TPB, 0, s>>>(c->X, c->tets, c->mat,
                                                   active_only ? c->act_list : nullptr,
                                                   active_only ? c->act_count : nullptr, c->T,
                                                   c->krun, c->Ke, c->steep, c->counters);
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
    k_expand<<<(unsigned)blocks, 256, 0, s>>>(c->Ke, c->krun, c->tets, c->T, ids, n, out);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

}  // namespace sta
