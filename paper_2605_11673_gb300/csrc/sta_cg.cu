// Jacobi-preconditioned conjugate gradients of the implicit-Euler step and of sta_solve: one
// persistent cooperative kernel runs a whole solve (the paper's solver, Sec. 4: CG with diagonal
// preconditioning).
//
// What bounds a solve.  An iteration is one product A z and a handful of vector updates between
// two grid-wide sums.  Run as two launches an iteration (one lane group per row over the CSR, an
// update kernel whose last CTA finished the sums), an iteration of a 27,783-DOF block took 29 us
// of which under 3 us is work: the rest was launches, last-CTA tails and, every eighth iteration, a
// host round trip.  On large systems the product was bound by the FP64 pipe (a warp FP64
// instruction holds its SM quadrant's for 64 cycles whatever its lanes do): the four-lane row sums and their
// half-empty ends cost 1.4 times the FMAs.
//
// Layout.  The matrix is copied once per solve into slices (k_cg_fill): a slice is 32 lanes, a
// lane holds one node (S = 1) or every fourth block of one node (S = 4, systems too small to give
// each warp 32 nodes), step t of the slice holds the lanes' t-th B x B blocks value by value
// (B = 3, or 1 for the scalar proxy operator) and their column nodes.  Every load is 32
// consecutive words, every FMA instruction works on 32 rows, and no lane sums across lanes but the
// quads of S = 4.  The nodes of a CTA's contiguous range are taken in descending row length, so a
// slice's lanes end together.  Blocks missing at the end of a lane are zero with the lane's own
// node as column.
//
// CTA c owns slices cta[c] .. cta[c + 1) for the whole solve: x, r, p, q and D^-1 of its rows stay
// in shared memory (global memory when they do not fit), and so does its part of the matrix when
// it fits (a 27,783-DOF block, the proxy operator of 113,000 nodes); only z, which the products
// gather, goes through global memory.
//
// Grid-wide sums.  A CTA adds its threads' partial sums in a fixed order and stores the sum with the
// iteration's number as one 16-byte word; one warp of every CTA then reads all CTAs' words until
// each carries that number and adds them in CTA order.  So every CTA has the same bits without a
// second exchange, and the sum is the barrier as well.  An iteration has three exchanges: p.q,
// the new z (a word without a sum: the stores are visible), and r.z with r.r, which only the end
// of the next product needs: warps of their own add and exchange them while the others already
// multiply.  Each has its own words; a CTA can store the next word of an exchange only after an
// exchange that every CTA enters when it has read the last one.  The waits are bounded;
// a CTA whose wait runs out marks the solve as failed and leaves, and so do, one after another,
// all others.  The solution goes to the context's x, and from there to the caller's vector or the
// state by a kernel of its own that first looks whether any CTA has failed (k_cg_finish): a CTA that
// was the only one late at the last exchange would otherwise leave its rows alone behind.
//
// Measured (GB300, time of an iteration with two launches -> now): 27,783-DOF block 29 -> 10.2 us,
// 341,000-DOF pre-fractured block 62 -> 40 us (FP64 floor of its product 24 us), scalar operator of
// 113,800 rows 34 -> 11.6 us.  With both sums on the path of the iteration (11.4, 48 and 13 us), the
// small block's product took 3 us, the sums 3 and 3.8 us, the updates 0.6 us.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sta_internal.cuh"

namespace sta {
namespace {

// Working warps of a CTA at most (one CTA per SM).  Measured at 750 nodes an SM, 24 slices (two for each
// of 12 warps, three for each of 8, one or two for 15), and not at other sizes: steps of the 341,000-DOF
// block with 8, 12 and 15 take 1.25, 1.15 and 1.19 ms, the scalar operator's frame 4.2, 4.1 and 4.3 ms.
constexpr int CG_WARPS = 12;
constexpr int CG_SUMS = 2;               // warps for the sums: r.z and r.r side by side
constexpr int CG_MAX_GRID = 160;         // CTAs at most: 5 words a lane in an exchange
constexpr int CG_CHECK = 8;              // iterations between two looks at stagnation
constexpr size_t CG_SMEM = 216 * 1024;   // dynamic shared memory at most (CgShared: 9 KB)

// One CTA's word of a grid-wide sum, alone in its 128-byte line: packed 16 bytes apart, the words
// took 5,500 cycles a sum instead of 3,600 (152 CTAs polling the same few lines).
struct __align__(128) CgSlot {
    unsigned long long v, epoch;
};

__device__ __forceinline__ void st_slot(CgSlot *p, double v, unsigned long long epoch) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(__double_as_longlong(v)), "l"(epoch)
                 : "memory");
}
__device__ __forceinline__ void ld_slot(const CgSlot *p, double &v, unsigned long long &epoch) {
    long long b;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\t"
                 "mov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(b), "=l"(epoch)
                 : "l"(p)
                 : "memory");
    v = __longlong_as_double(b);
}

struct CgArgs {
    const int32_t *snode;  // per slice and lane: its node, -1 for none
    const int32_t *sbase;  // slices + 1: first step of each slice
    const int32_t *cta;    // grid + 1: first slice of each CTA
    const int32_t *col;    // per step and lane: column node
    const double *val;     // per step: B * B values of 32 lanes each
    const double *b, *dinv;
    double *x, *z;         // z: a node's B values at z_stride<B>
    double *vec;           // 5 vectors in slice order when shared memory does not hold them
    int64_t vec_len;       // of one of them
    bool plan_shared;
    CgSlot *slots;         // CG_WORDS exchanges x CG_MAX_GRID, and the failure's
    unsigned long long epoch;
    unsigned spins;        // polls of a wait at most
    CgResult *out;         // host-mapped
    double tol2;
    int32_t max_iter;
    bool stagnate;
};

// The exchanges: r.z, r.r and (once) b.b, p.q, z.
enum { W_RZ, W_RR, W_BB, W_PQ, W_Z, CG_WORDS };
constexpr int CG_FAILED = CG_WORDS * CG_MAX_GRID;  // its epoch: the first one of the last solve that failed

// Nodes of three values are gathered as one aligned word of four: the three loads of a 24-byte
// record cost the L1 cache nearly three times as much.
template <int B> constexpr int z_stride = B == 3 ? 4 : 1;

// Shared scratch of the sums.
struct CgShared {
    double part[3][CG_WARPS * 32];
    double sum[3], beta;  // of the sum warps
    double pq, alpha;
    int late[3], failed, quit;
};

// Barriers between a CTA's warps: the working warps among themselves, partial sums to the sum
// warps, sums to the working warps.  (bar.sync and bar.arrive are aligned instructions, which a warp
// has to execute as a whole: it is brought together first, as it may come from a branch of one lane.)
enum { BAR_WORK = 1, BAR_PARTS, BAR_SUMS };
__device__ __forceinline__ void named_sync(int id, int threads) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ double warp_sum(double t) {
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// The sum of n (a multiple of 32) partial sums, in every lane.  Through shared memory: a shuffle
// tree in every warp would cost 5 FP64 instructions per warp and value.
__device__ __forceinline__ double sum_parts(const double *p, int n, int lane) {
    double t0 = p[lane], t1 = 0.0, t2 = 0.0, t3 = 0.0;
    int i = 32 + lane;
    for (; i + 96 < n; i += 128) {
        t0 += p[i];
        t1 += p[i + 32];
        t2 += p[i + 64];
        t3 += p[i + 96];
    }
    for (; i < n; i += 32) t0 += p[i];
    return warp_sum((t0 + t1) + (t2 + t3));
}

// Waits until every CTA's word of one exchange carries `epoch`.  Returns the lane's part of their
// sum; `late` (same in all lanes): the wait ran out.
__device__ __forceinline__ double wait_words(const CgSlot *set, unsigned long long epoch, unsigned spins, int lane,
                                             bool &late) {
    constexpr int PER = CG_MAX_GRID / 32;
    double got[PER];
    unsigned need = 0;  // words still to come
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        got[i] = 0.0;
        if (lane + 32 * i < (int)gridDim.x) need |= 1u << i;
    }
    for (unsigned spin = 0; need && spin < spins; ++spin) {
        double w[PER];
        unsigned long long e[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            e[i] = 0;
            if (need >> i & 1) ld_slot(set + lane + 32 * i, w[i], e[i]);
        }
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if ((need >> i & 1) && e[i] == epoch) {
                got[i] = w[i];
                need &= ~(1u << i);
            }
    }
    late = __any_sync(0xffffffffu, need != 0);
    return ((got[0] + got[1]) + (got[2] + got[3])) + got[4];
}

// The sum warps: r.z, r.r and at first b.b of every iteration, and beta.
__device__ void sum_warps(const CgArgs &a, CgShared &sh, int me, int work, int all) {
    const int lane = threadIdx.x & 31;
    double rz = 0.0;
    for (unsigned long long epoch = a.epoch + 1;; ++epoch) {
        named_sync(BAR_PARTS, all);
        if (sh.quit) return;
        const int nv = epoch == a.epoch + 1 ? 3 : 2;
        for (int k = me; k < nv; k += CG_SUMS) {
            const double t = sum_parts(sh.part[k], work, lane);
            if (lane == 0) st_slot(a.slots + k * CG_MAX_GRID + blockIdx.x, t, epoch);
        }
        for (int k = me; k < nv; k += CG_SUMS) {
            bool late;
            const double t = warp_sum(wait_words(a.slots + k * CG_MAX_GRID, epoch, a.spins, lane, late));
            if (lane == 0) {
                sh.sum[k] = t;
                sh.late[k] = late;
                if (k == W_RZ) sh.beta = rz == 0.0 ? 0.0 : t / rz;
            }
            if (k == W_RZ) rz = t;
        }
        named_arrive(BAR_SUMS, all);
    }
}

// Value loads of the part of the matrix that is not kept in shared memory: read once an iteration,
// so kept out of L1, where the gathered z lives.
__device__ __forceinline__ double ld_stream(const double *p) {
    double v;
    asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// Brings memory to the L2 cache (16-byte aligned address and size).
__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// Steps from HBM to L2 ahead of the loads (with the first slices brought there while the sums wait: a
// step of the 341,000-DOF block 1.155 -> 1.114 ms; 4 to 10: the same within 1%).
constexpr int CG_AHEAD = 6;

// The B values of a node in y, a vector of YS values a node; 0 where not `on` (same in all lanes; a
// branch around the one wide load was faster than the load predicated).
template <int B, int YS>
__device__ __forceinline__ void gather(const double *y, int32_t node, bool on, double (&w)[B]) {
    const double *p = y + YS * (int64_t)node;
    if constexpr (YS == 4) {
#pragma unroll
        for (int j = 0; j < B; ++j) w[j] = 0.0;
        double pad;
        if (on)
            asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                         : "=d"(w[0]), "=d"(w[1]), "=d"(w[2]), "=d"(pad)
                         : "l"(p));
    } else {
#pragma unroll
        for (int j = 0; j < B; ++j) w[j] = on ? p[j] : 0.0;
    }
}

// Rows of A y of the lane's node in one slice: S = 1: acc[c] is component c of the lane's node.
// S = 4: acc[0] is component (lane & 3) of the quad's node.
template <int B, int S, bool RES, int YS>
__device__ __forceinline__ void slice_rows(const double *val, const int32_t *col, int steps, int lane,
                                           const double *y, double (&acc)[S == 1 ? B : 1]) {
    double s[B];
#pragma unroll
    for (int i = 0; i < B; ++i) s[i] = 0.0;
    const double *vp = val + lane;
    const int32_t *cp = col + lane;
    // U steps at a time: the values and gathered z of the next U are on their way while these are
    // multiplied, and the columns of the U after them.  The last warp of a CTA works alone on its
    // longest slice, so a step's two dependent loads must not stand in a row.
    constexpr int U = B == 1 ? 4 : 2;
    int32_t c[U];
    double m[U][B * B], w[U][B];
    auto cols = [&](int t) {
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = t + u < steps ? cp[32 * (t + u)] : -1;
    };
    auto load = [&](int t, double (&mm)[U][B * B], double (&ww)[U][B]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool on = t + u < steps;
#pragma unroll
            for (int e = 0; e < B * B; ++e) {
                const double *q = vp + 32 * ((t + u) * (B * B) + e);
                mm[u][e] = !on ? 0.0 : RES ? *q : ld_stream(q);
            }
            gather<B, YS>(y, c[u], on, ww[u]);
        }
    };
    cols(0);
    load(0, m, w);
    cols(U);
    for (int t = 0; t < steps; t += U) {
        double mn[U][B * B], wn[U][B];
        if (!RES && lane == 0 && t + CG_AHEAD < steps)
            prefetch_l2(val + (int64_t)(32 * B * B) * (t + CG_AHEAD),
                        256 * B * B * (steps - t - CG_AHEAD < U ? steps - t - CG_AHEAD : U));
        load(t + U, mn, wn);
        cols(t + 2 * U);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < B; ++j)
#pragma unroll
                for (int i = 0; i < B; ++i) s[i] = __fma_rn(m[u][B * i + j], w[u][j], s[i]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int e = 0; e < B * B; ++e) m[u][e] = mn[u][e];
#pragma unroll
            for (int j = 0; j < B; ++j) w[u][j] = wn[u][j];
        }
    }
    if constexpr (S == 1) {
#pragma unroll
        for (int i = 0; i < B; ++i) acc[i] = s[i];
    } else if constexpr (B == 1) {
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
        acc[0] = (lane & 3) == 0 ? s[0] : 0.0;  // the quad's first lane has the row
    } else {
        // the quad's 4 x 3 partial sums to component (lane & 3) in 3 additions: lanes of even
        // number keep components 0 and 2, odd ones 1 (and nothing), then pairs exchange
        const bool odd = lane & 1, hi = lane & 2;
        const double a = __shfl_xor_sync(0xffffffffu, odd ? s[0] : s[1], 1);
        const double d = __shfl_xor_sync(0xffffffffu, odd ? s[2] : 0.0, 1);
        const double k0 = (odd ? s[1] : s[0]) + a;  // component lane & 1 over the pair
        const double k2 = (odd ? 0.0 : s[2]) + d;   // component 2 over the pair (even lanes)
        const double o = __shfl_xor_sync(0xffffffffu, hi ? k0 : k2, 2);
        acc[0] = (hi ? k2 : k0) + o;
    }
}

// 8-byte words of a plan of ns slices in shared memory (even: the matrix behind it is copied 16 bytes
// at a time).
__host__ __device__ constexpr int plan_words(int ns) { return (33 * ns + 1 + 3) / 4 * 2; }

template <int B, int S, bool RES>
__global__ void __launch_bounds__((CG_WARPS + CG_SUMS) * 32, 1) k_cg_solve(CgArgs a, int warps) {
    constexpr int NR = S == 1 ? B : 1;  // rows of a lane
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ CgShared sh;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int work = 32 * warps, all = blockDim.x;  // threads that work; with the sum warps
    const int s0 = a.cta[blockIdx.x], ns = a.cta[blockIdx.x + 1] - s0;
    const int step0 = a.sbase[s0];
    // vectors of the CTA's rows, in slice order
    const bool in_shared = RES || !a.vec;
    const int64_t own = (int64_t)ns * NR * 32, len = in_shared ? own : a.vec_len;
    double *vec = in_shared ? reinterpret_cast<double *>(dyn) : a.vec + (int64_t)s0 * NR * 32;
    double *X = vec, *R = X + len, *Pv = R + len, *Q = Pv + len, *D = Q + len;
    const double *val = a.val + (int64_t)step0 * (32 * B * B);
    const int32_t *col = a.col + (int64_t)step0 * 32;
    // first steps and nodes of the CTA's slices, behind the vectors: every fence empties the L1 cache
    double *behind = reinterpret_cast<double *>(dyn) + 5 * own;
    const int32_t *snode = a.snode + 32 * s0, *sbase = a.sbase + s0;
    if (a.plan_shared) {
        int32_t *plan = reinterpret_cast<int32_t *>(behind);
        for (int i = threadIdx.x; i < 32 * ns; i += blockDim.x) plan[i] = snode[i];
        for (int i = threadIdx.x; i <= ns; i += blockDim.x) plan[32 * ns + i] = sbase[i];
        snode = plan;
        sbase = plan + 32 * ns;
        behind += plan_words(ns);
    }
    if constexpr (RES) {  // the CTA's part of the matrix
        const int steps = a.sbase[s0 + ns] - step0;
        double *sv = behind;
        int32_t *sc = reinterpret_cast<int32_t *>(sv + (int64_t)steps * (32 * B * B));
        for (int i = threadIdx.x; i < steps * (16 * B * B); i += blockDim.x)
            reinterpret_cast<double2 *>(sv)[i] = __ldg(reinterpret_cast<const double2 *>(val) + i);
        for (int i = threadIdx.x; i < steps * 32; i += blockDim.x) sc[i] = __ldg(col + i);
        val = sv;
        col = sc;
    }
    if (threadIdx.x == 0) sh.quit = 0;
    __syncthreads();
    if (wid >= warps) {
        sum_warps(a, sh, wid - warps, work, all);
        return;
    }
    // r = b - A x, z = D^-1 r, p = q = 0 (with beta = 0 the first step forms p = z, q = A z)
    double v0 = 0.0, v1 = 0.0, v2 = 0.0;
    for (int sl = wid; sl < ns; sl += warps) {
        const int t0 = sbase[sl] - step0, t1 = sbase[sl + 1] - step0;
        const int32_t node = snode[32 * sl + lane];
        double acc[NR];
        slice_rows<B, S, RES, B>(val + (int64_t)t0 * (32 * B * B), col + (int64_t)t0 * 32, t1 - t0, lane,
                                 a.x, acc);
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            const int k = (sl * NR + c) * 32 + lane;
            const int comp = S == 1 ? c : lane & 3;
            double xi = 0.0, ri = 0.0, di = 0.0;
            if (node >= 0 && comp < B) {
                const int64_t i = B * (int64_t)node + comp;
                const double bi = a.b[i];
                xi = a.x[i];
                di = a.dinv[i];
                ri = bi - acc[c];
                const double zi = di * ri;
                a.z[z_stride<B> * (int64_t)node + comp] = zi;
                v0 = __fma_rn(ri, zi, v0);
                v1 = __fma_rn(ri, ri, v1);
                v2 = __fma_rn(bi, bi, v2);
            }
            X[k] = xi;
            R[k] = ri;
            D[k] = di;
            Pv[k] = 0.0;
            Q[k] = 0.0;
        }
    }
    sh.part[W_RZ][threadIdx.x] = v0;
    sh.part[W_RR][threadIdx.x] = v1;
    sh.part[W_BB][threadIdx.x] = v2;
    named_arrive(BAR_PARTS, all);
    // Whether a product starts before it is known that the iteration takes place: the last one, for
    // nothing, then costs a product (30 us at 750 nodes an SM, where the sums wait 1 us for it).
    constexpr bool EARLY = S == 4 || B == 1;
    double rz = 0.0, rr = 0.0, bb = 0.0, beta = 0.0, best = -1.0;
    int iters = 0, best_it = 0;
    bool ok = true, first = true;
    for (unsigned long long epoch = a.epoch + 1;; ++epoch) {
        // every CTA's z is visible
        named_sync(BAR_WORK, work);
        if (wid == 0) {
            if (lane == 0) {
                __threadfence();  // the CTA's z
                st_slot(a.slots + W_Z * CG_MAX_GRID + blockIdx.x, 0.0, epoch);
            }
            bool late;
            wait_words(a.slots + W_Z * CG_MAX_GRID, epoch, a.spins, lane, late);
            __threadfence();
            if (lane == 0) sh.failed = late;
        }
        named_sync(BAR_WORK, work);
        ok = !sh.failed;
        bool stop = false, taken = false;
        auto take = [&]() {  // the sums of the residual: the end, or beta
            named_sync(BAR_SUMS, all);
            taken = true;
            rz = sh.sum[W_RZ];
            rr = sh.sum[W_RR];
            beta = sh.beta;
            ok = ok && !sh.late[W_RZ] && !sh.late[W_RR];
            if (first) {
                bb = sh.sum[W_BB];
                ok = ok && !sh.late[W_BB];
            } else {
                ++iters;
            }
            const bool done = rr <= a.tol2 * bb;
            stop = !ok || done || iters >= a.max_iter;
            if (!first && a.stagnate && iters % CG_CHECK == 0 && !done) {
                if (best < 0.0 || rr < 0.25 * best) {
                    best = rr;
                    best_it = iters;
                } else if (iters - best_it > 1000) {
                    stop = true;
                }
            }
            first = false;
        };
        if (!EARLY || !ok) take();
        double pq = 0.0;
        for (int sl = wid; sl < ns && !stop; sl += warps) {
            const int t0 = sbase[sl] - step0, t1 = sbase[sl + 1] - step0;
            const int32_t node = snode[32 * sl + lane];
            double acc[NR], zi[NR];
#pragma unroll
            for (int c = 0; c < NR; ++c) {
                const int comp = S == 1 ? c : lane & 3;
                zi[c] = node >= 0 && comp < B ? a.z[z_stride<B> * (int64_t)node + comp] : 0.0;
            }
            slice_rows<B, S, RES, z_stride<B>>(val + (int64_t)t0 * (32 * B * B), col + (int64_t)t0 * 32,
                                               t1 - t0, lane, a.z, acc);
            if (!taken) take();
            if (stop) break;
#pragma unroll
            for (int c = 0; c < NR; ++c) {
                const int k = (sl * NR + c) * 32 + lane;
                const double pi = __fma_rn(beta, Pv[k], zi[c]), qi = __fma_rn(beta, Q[k], acc[c]);
                Pv[k] = pi;
                Q[k] = qi;
                pq = __fma_rn(pi, qi, pq);
            }
        }
        if (!taken) take();
        if (stop) break;
        if (!RES && lane == 0 && wid < ns) {  // the warp's next slice, while HBM is idle
            const int t0 = sbase[wid] - step0, t1 = sbase[wid + 1] - step0;
            if (t1 > t0) prefetch_l2(val + (int64_t)t0 * (32 * B * B), (t1 - t0) * (256 * B * B));
        }
        sh.part[0][threadIdx.x] = pq;
        named_sync(BAR_WORK, work);
        if (wid == 0) {
            CgSlot *set = a.slots + W_PQ * CG_MAX_GRID;
            double t = sum_parts(sh.part[0], work, lane);
            if (lane == 0) st_slot(set + blockIdx.x, t, epoch);
            bool late;
            t = warp_sum(wait_words(set, epoch, a.spins, lane, late));
            if (lane == 0) {
                sh.pq = t;
                sh.alpha = rz / t;  // by one warp: a division is a dozen dependent FP64 instructions
                sh.failed = late;
            }
        }
        named_sync(BAR_WORK, work);
        if (!(ok = !sh.failed)) break;
        // breakdown: p = 0 (already converged) or A not positive definite
        if (!(sh.pq > 0.0)) break;
        const double alpha = sh.alpha;
        v0 = v1 = 0.0;
        for (int sl = wid; sl < ns; sl += warps) {
            const int32_t node = snode[32 * sl + lane];
#pragma unroll
            for (int c = 0; c < NR; ++c) {
                const int k = (sl * NR + c) * 32 + lane;
                const int comp = S == 1 ? c : lane & 3;
                X[k] = __fma_rn(alpha, Pv[k], X[k]);
                const double ri = __fma_rn(-alpha, Q[k], R[k]), zi = D[k] * ri;
                R[k] = ri;
                if (node >= 0 && comp < B) a.z[z_stride<B> * (int64_t)node + comp] = zi;
                v0 = __fma_rn(ri, zi, v0);
                v1 = __fma_rn(ri, ri, v1);
            }
        }
        sh.part[W_RZ][threadIdx.x] = v0;
        sh.part[W_RR][threadIdx.x] = v1;
        named_arrive(BAR_PARTS, all);
    }
    // (on every way out of the loop the sum warps wait for partial sums)
    if (threadIdx.x == 0) sh.quit = 1;
    named_arrive(BAR_PARTS, all);
    // (ok: the sums of the first residual are complete, so no CTA reads x any more)
    for (int sl = wid; sl < ns && ok; sl += warps) {
        const int32_t node = snode[32 * sl + lane];
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            const int comp = S == 1 ? c : lane & 3;
            if (node >= 0 && comp < B) a.x[B * (int64_t)node + comp] = X[(sl * NR + c) * 32 + lane];
        }
    }
    if (threadIdx.x == 0 && (blockIdx.x == 0 || !ok)) {
        if (ok) {
            a.out->iters = iters;
            a.out->rr = rr;
            a.out->bb = bb;
        } else {
            a.out->failed = 1;
            a.slots[CG_FAILED].epoch = a.epoch + 1;
        }
    }
}

// The solution of a solve that no CTA has given up to the caller (xout), or the state advanced: free
// rows u = x, v = (x - u) / h; a clamped row is held at 0, a row without mass keeps u.
__global__ void k_cg_finish(int64_t n3, const double *x, const CgSlot *slots, unsigned long long epoch,
                            double *__restrict__ xout, double *__restrict__ u, double *__restrict__ v,
                            const uint8_t *__restrict__ fr, const uint8_t *__restrict__ clamped, double h) {
    dependency_wait();
    if (slots[CG_FAILED].epoch == epoch) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (xout) {
            xout[i] = x[i];
        } else if (fr[i]) {
            v[i] = (x[i] - u[i]) / h;
            u[i] = x[i];
        } else {
            v[i] = 0.0;
            if (clamped[i / 3]) u[i] = 0.0;
        }
    }
}

// Column nodes of the slices, once per context: block part + S t of the lane's node, the node
// itself past its end.
__global__ void k_cg_cols(int32_t nslices, int S, const int32_t *__restrict__ snode,
                          const int32_t *__restrict__ sbase, const int32_t *__restrict__ adj_ptr,
                          const int32_t *__restrict__ adj, int32_t *__restrict__ col) {
    const int lane = threadIdx.x & 31, part = lane % S;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t sl = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; sl < nslices; sl += nw) {
        const int32_t a = snode[32 * sl + lane];
        const int32_t p0 = a >= 0 ? adj_ptr[a] : 0, deg = a >= 0 ? adj_ptr[a + 1] - p0 : 0;
        for (int32_t t = sbase[sl]; t < sbase[sl + 1]; ++t) {
            const int32_t p = part + S * (t - sbase[sl]);
            col[32 * (int64_t)t + lane] = p < deg ? adj[p0 + p] : (a >= 0 ? a : 0);
        }
    }
}

// The matrix of the solve in slice order: h2 K + mass on the diagonal, rows that are not solved
// for zero (so that their q, hence r, stays zero).  One CTA per slice and FILL_STEPS steps: the
// rows' contiguous pieces are read into shared memory, 3 * FILL_STEPS * S doubles at a time, and
// written out by value and lane.  Bound by memory: reads and writes the matrix once (240 MB for
// 14 M entries).
constexpr int FILL_STEPS = 8;

template <int B, int S>
__global__ void __launch_bounds__(256)
k_cg_fill(const int32_t *__restrict__ snode, const int32_t *__restrict__ sbase,
          const int32_t *__restrict__ adj_ptr, const int32_t *__restrict__ adj,
          const double *__restrict__ val, const double *__restrict__ mass, double h2,
          const uint8_t *__restrict__ fr, double *__restrict__ out) {
    constexpr int NODES = 32 / S, RUN = B * S * FILL_STEPS;  // entries of a row per chunk
    __shared__ double buf[NODES * B][RUN + 1];
    const int64_t sl = blockIdx.x;
    const int32_t b0 = sbase[sl], steps = sbase[sl + 1] - b0;
    for (int32_t t0 = 0; t0 < steps; t0 += FILL_STEPS) {
        for (int i = threadIdx.x; i < NODES * B * RUN; i += blockDim.x) {
            const int row = i / RUN, e = i - row * RUN, m = row / B, c = row - m * B;
            const int32_t a = snode[32 * sl + S * m];
            double v = 0.0;
            if (a >= 0) {
                const int32_t p0 = adj_ptr[a], deg = adj_ptr[a + 1] - p0;
                const int32_t k = B * S * t0 + e;  // entry of the row
                if (k < B * deg && fr[B * (int64_t)a + c]) {
                    v = val[(int64_t)B * B * p0 + (int64_t)c * B * deg + k];
                    if (mass) {
                        v *= h2;
                        const int32_t p = k / B;
                        if (k - B * p == c && adj[p0 + p] == a)
                            v = __fma_rn(h2, val[(int64_t)B * B * p0 + (int64_t)c * B * deg + k], mass[a]);
                    }
                }
            }
            buf[row][e] = v;
        }
        __syncthreads();
        const int nst = steps - t0 < FILL_STEPS ? steps - t0 : FILL_STEPS;
        for (int i = threadIdx.x; i < nst * B * B * 32; i += blockDim.x) {
            const int lane = i & 31, e = (i >> 5) % (B * B), t = (i >> 5) / (B * B);
            const int row = (lane / S) * B + e / B, k = B * (S * t + lane % S) + e % B;
            out[((int64_t)(b0 + t0 + t) * (B * B) + e) * 32 + lane] = buf[row][k];
        }
        __syncthreads();
    }
}

template <int B, int S>
int launch_fill(Ctx *c, const double *val, const double *mass, double h2, cudaStream_t s) {
    k_cg_fill<B, S><<<(unsigned)c->cg_slices, 256, 0, s>>>(c->cg_snode, c->cg_sbase, c->adj_ptr, c->adj,
                                                           val, mass, h2, c->cg_free, c->cg_val);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

template <int B, int S, bool RES> int launch_solve(Ctx *c, CgArgs &a, cudaStream_t s) {
    void *args[] = {&a, &c->cg_warps};
    const void *kern = (const void *)k_cg_solve<B, S, RES>;
    STA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CG_SMEM));
    STA_CUDA_TRY(cudaLaunchCooperativeKernel(kern, dim3(c->cg_grid), dim3(32 * (c->cg_warps + CG_SUMS)), args,
                                             c->cg_smem, s));
    return STA_OK;
}

template <int B, int S> int launch_solve(Ctx *c, CgArgs &a, cudaStream_t s) {
    return c->cg_resident ? launch_solve<B, S, true>(c, a, s) : launch_solve<B, S, false>(c, a, s);
}

}  // namespace

// The buffers and the slice plan of a context's solves, once.
int cg_alloc(Ctx *c) {
    if (c->cg) return STA_OK;
    const int64_t n = c->n, n3 = c->nrows;  // DOFs
    const int B = c->op == STA_OP_PROXY ? 1 : 3;
    std::vector<int32_t> ap(n + 1, 0);
    if (n > 0)
        STA_CUDA_TRY(cudaMemcpy(ap.data(), c->adj_ptr, sizeof(int32_t) * (n + 1), cudaMemcpyDeviceToHost));
    // a quad per node while 32 nodes a warp would leave an SM's quadrants without a warp each: a
    // lane's blocks follow one another in time, a quad's are four at a time but cost 3 more
    // instructions a slice.  Measured, cycles of a product: 61 nodes an SM, 3 x 3 blocks: 6,400
    // with quads, 13,600 with lanes; 750 nodes an SM: 68,700 with quads, 62,400 with lanes
    // (scalar operator: 18,200 and 8,700).
    const int64_t per_sm = (n + c->num_sms - 1) / c->num_sms;
    int S = per_sm < 384 ? 4 : 1;
    // A warp works alone on a row far longer than the rest, 970 cycles a step (scalar: 110); where a lane's
    // steps of it take longer than a CTA's whole product with quads (64 cycles an FP64 instruction of a
    // quadrant), quads, which take a quarter of them.  Iterations, us, with lanes / quads, by the longest
    // row: 453 nodes an SM, 30 blocks 33 / 35, 60: 42 / 40, 300: 152 / 66; 774 an SM, 60: 51 / 59, 100:
    // 69 / 64, 300: 167 / 89; scalar, 774 an SM, 100: 16 / 22, 200: 24 / 24, 1000: 74 / 36.
    if (S == 1) {
        const int maxg = std::min(c->num_sms, CG_MAX_GRID);
        int64_t longest = 0, quads = 0;
        for (int64_t a = 0; a < n; ++a) {
            longest = std::max<int64_t>(longest, ap[a + 1] - ap[a]);
            quads += B * B * (int64_t)((ap[a + 1] - ap[a] + 3) / 4) + 10;
        }
        if (longest * (B == 3 ? 970 : 110) > quads / 8 / maxg / 4 * 64) S = 4;
    }
    const int per = 32 / S;
    const int64_t want = (n + per - 1) / per;
    const int maxg = std::min(c->num_sms, CG_MAX_GRID);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, maxg));
    // contiguous node ranges of equal work, in FP64 instructions of a slice: B * B a step, and
    // about 10 a row for the vectors
    const int rows = S == 1 ? B : 1;
    auto steps_of = [&](int64_t a) { return (int64_t)(ap[a + 1] - ap[a] + S - 1) / S; };
    auto weight = [&](int64_t a) { return B * B * steps_of(a) + 10 * rows; };
    int64_t total = 0;
    for (int64_t a = 0; a < n; ++a) total += weight(a);
    std::vector<int32_t> snode, sbase{0}, cta{0}, order;
    std::vector<int64_t> range(grid + 1, 0);
    int64_t most = 0, sum = 0;
    for (int g = 0; g < grid; ++g) {
        int64_t a1 = range[g];
        const int64_t lim = total * (g + 1) / grid;
        while (a1 < n && (g == grid - 1 || sum + weight(a1) <= lim)) sum += weight(a1++);
        range[g + 1] = a1;
        most = std::max(most, (a1 - range[g] + per - 1) / per);
    }
    // warps in fours (one per SM quadrant), no more than slices
    const int warps = (int)std::max<int64_t>(4, std::min<int64_t>(CG_WARPS, (most + 3) / 4 * 4));
    int max_slices = 0;
    int64_t max_steps = 0;
    for (int g = 0; g < grid; ++g) {
        order.clear();
        for (int64_t a = range[g]; a < range[g + 1]; ++a) order.push_back((int32_t)a);
        std::stable_sort(order.begin(), order.end(), [&](int32_t p, int32_t q) {
            return ap[p + 1] - ap[p] > ap[q + 1] - ap[q];
        });
        // the slices, longest first, each to the warp with the least work so far (among equals to
        // the SM quadrant with the least: a quadrant has its own FP64 pipe, which a warp
        // instruction holds for 64 cycles, and warp w runs on quadrant w % 4); warp w's slices
        // take the positions w, w + warps, ...  Dealt in plain order the first quadrant got the
        // longest slice of every four, 20% over the mean, and warps left alone on a long slice
        // waited for every load.
        const size_t cnt = (order.size() + per - 1) / per;
        std::vector<std::vector<int>> of(warps);
        std::vector<int64_t> load(warps, 0);
        int64_t quad[4] = {0, 0, 0, 0};
        for (size_t i = 0; i < cnt; ++i) {
            int k = 0;
            for (int w = 1; w < warps; ++w)
                if (load[w] < load[k] || (load[w] == load[k] && quad[w % 4] < quad[k % 4])) k = w;
            of[k].push_back((int)i);
            load[k] += weight(order[i * per]);
            quad[k % 4] += weight(order[i * per]);
        }
        const int32_t first = sbase.back();
        // the warps of a quadrant in descending number of slices, and no places past the last slice: an
        // empty one costs a warp its turn and shared memory (36 places for 32 slices: solves of the
        // scalar operator of 113,800 rows 4.15 ms, now 3.99; steps of 341,000 DOFs 1.10, now 1.08)
        for (int w = 0; w < warps; ++w)
            for (int v = w + 4; v < warps; v += 4)
                if (of[v].size() > of[w].size()) std::swap(of[v], of[w]);
        size_t places = 0;
        for (int w = 0; w < warps; ++w)
            if (!of[w].empty()) places = std::max(places, w + 1 + warps * (of[w].size() - 1));
        for (size_t i = 0; i < places; ++i) {
            const auto &q = of[i % warps];
            const bool has = i / warps < q.size();  // else an empty slice
            const size_t at = has ? (size_t)q[i / warps] * per : 0;
            for (int l = 0; l < 32; ++l)
                snode.push_back(has && at + l / S < order.size() ? order[at + l / S] : -1);
            sbase.push_back(sbase.back() + (has ? (int32_t)steps_of(order[at]) : 0));
        }
        cta.push_back((int32_t)sbase.size() - 1);
        max_slices = std::max(max_slices, cta[g + 1] - cta[g]);
        max_steps = std::max<int64_t>(max_steps, sbase.back() - first);
    }
    const int64_t slices = (int64_t)sbase.size() - 1, steps = sbase.back();
    const size_t vec_bytes = 5 * sizeof(double) * 32 * rows * (size_t)max_slices;
    const size_t mat_bytes = (size_t)max_steps * 32 * (B * B * sizeof(double) + sizeof(int32_t));
    const size_t plan_bytes = sizeof(double) * plan_words(max_slices);
    const bool vec_shared = vec_bytes <= CG_SMEM, resident = vec_bytes + mat_bytes <= CG_SMEM;
    size_t smem = resident ? vec_bytes + mat_bytes : (vec_shared ? vec_bytes : 0);
    // The plan goes to shared memory unless the cache would pay for it with the next one of the sizes
    // that shared memory is set aside in (scalar operator of 113,800 rows: 182 KB without the plan,
    // 196 set aside; with it 228, and a frame's solve takes 4.3 ms instead of 4.15).
    auto set_aside = [](size_t used) {
        for (size_t kb : {32, 64, 100, 132, 164, 196})
            if (used + sizeof(CgShared) + 1024 <= kb * 1024) return kb;
        return (size_t)228;
    };
    c->cg_plan_shared = vec_shared && smem + plan_bytes <= CG_SMEM && set_aside(smem + plan_bytes) == set_aside(smem);
    if (c->cg_plan_shared) smem += plan_bytes;
    STA_TRY(dev_alloc(c, &c->cg_free, n3));
    STA_TRY(dev_alloc(c, &c->cg_snode, 32 * slices));
    STA_TRY(dev_alloc(c, &c->cg_sbase, slices + 1));
    STA_TRY(dev_alloc(c, &c->cg_cta, grid + 1));
    STA_TRY(dev_alloc(c, &c->cg_col, 32 * steps));
    STA_TRY(dev_alloc(c, &c->cg_val, 32 * steps * B * B));
    c->cg_vec = nullptr;
    if (!vec_shared) STA_TRY(dev_alloc(c, &c->cg_vec, 5 * 32 * rows * slices));
    CgSlot *slots = nullptr;
    STA_TRY(dev_alloc(c, &slots, CG_FAILED + 1));
    c->cg_slots = slots;
    STA_CUDA_TRY(cudaMemset(slots, 0, sizeof(CgSlot) * (CG_FAILED + 1)));
    if (!c->h_cg) {
        STA_CUDA_TRY(cudaHostAlloc((void **)&c->h_cg, sizeof(CgResult), cudaHostAllocMapped));
        STA_CUDA_TRY(cudaHostGetDevicePointer((void **)&c->d_cg, c->h_cg, 0));
    }
    STA_CUDA_TRY(cudaMemcpy(c->cg_snode, snode.data(), sizeof(int32_t) * snode.size(), cudaMemcpyHostToDevice));
    STA_CUDA_TRY(cudaMemcpy(c->cg_sbase, sbase.data(), sizeof(int32_t) * sbase.size(), cudaMemcpyHostToDevice));
    STA_CUDA_TRY(cudaMemcpy(c->cg_cta, cta.data(), sizeof(int32_t) * cta.size(), cudaMemcpyHostToDevice));
    if (slices > 0) {
        const int64_t want_ctas = (slices * 32 + 255) / 256;
        k_cg_cols<<<(unsigned)std::min<int64_t>(want_ctas, c->num_sms * 8), 256>>>(
            (int32_t)slices, S, c->cg_snode, c->cg_sbase, c->adj_ptr, c->adj, c->cg_col);
        STA_CUDA_TRY(cudaGetLastError());
        STA_CUDA_TRY(cudaStreamSynchronize(0));
    }
    c->cg_grid = grid;
    c->cg_S = S;
    c->cg_slices = slices;
    c->cg_steps = steps;
    c->cg_warps = warps;
    c->cg_resident = resident;
    c->cg_smem = smem;
    // x, b, D^-1, z (whole 32-byte words); last: marks the plan as complete
    STA_TRY(dev_alloc(c, &c->cg, (3 * n3 + 3) / 4 * 4 + (B == 3 ? 4 : 1) * n));
    return STA_OK;
}

// Solves (h2 K(val) + mass) x = b on the rows with cg_free set, from the x, b and D^-1 in the
// context's buffers, into xout, or (null) into the state of the implicit-Euler loop, which it advances;
// waits for the result.  A solve that fails changes neither.  mass null: none (h2 = 1).
int launch_cg_solve(Ctx *c, const double *val, const double *mass, double h2, double tol,
                    int32_t max_iter, bool stagnate, double *xout, cudaStream_t s,
                    CgResult *res) {
    const int64_t n3 = c->nrows;
    *res = CgResult{};
    if (n3 == 0) return STA_OK;
    const bool scalar = c->op == STA_OP_PROXY;
    CgArgs a{};
    a.snode = c->cg_snode;
    a.sbase = c->cg_sbase;
    a.cta = c->cg_cta;
    a.col = c->cg_col;
    a.val = c->cg_val;
    a.x = c->cg;
    a.b = c->cg + n3;
    a.dinv = c->cg + 2 * n3;
    a.z = c->cg + (3 * n3 + 3) / 4 * 4;
    a.vec = c->cg_vec;
    a.vec_len = (int64_t)c->cg_slices * 32 * (c->cg_S == 1 && !scalar ? 3 : 1);
    a.plan_shared = c->cg_plan_shared;
    a.slots = static_cast<CgSlot *>(c->cg_slots);
    a.epoch = c->cg_epoch;
    c->cg_epoch += (unsigned long long)max_iter + 2;  // past every exchange of this solve
    a.out = c->d_cg;
    a.tol2 = tol * tol;
    a.max_iter = max_iter;
    a.stagnate = stagnate;
    a.spins = c->cg_spins;
    *c->h_cg = CgResult{};
    if (scalar) {
        STA_TRY((c->cg_S == 1 ? launch_fill<1, 1>(c, val, mass, h2, s) : launch_fill<1, 4>(c, val, mass, h2, s)));
        STA_TRY((c->cg_S == 1 ? launch_solve<1, 1>(c, a, s) : launch_solve<1, 4>(c, a, s)));
    } else {
        STA_TRY((c->cg_S == 1 ? launch_fill<3, 1>(c, val, mass, h2, s) : launch_fill<3, 4>(c, val, mass, h2, s)));
        STA_TRY((c->cg_S == 1 ? launch_solve<3, 1>(c, a, s) : launch_solve<3, 4>(c, a, s)));
    }
    const int64_t ctas = std::min<int64_t>((n3 + 255) / 256, 8 * (int64_t)c->num_sms);
    STA_TRY(launch_overlapped(k_cg_finish, (unsigned)ctas, 256, 0, s, n3, (const double *)a.x, (const CgSlot *)a.slots,
                              a.epoch + 1, xout, c->du, c->dv, c->cg_free, c->clamped, c->dyn_h));
    STA_CUDA_TRY(cudaStreamSynchronize(s));
    *res = *c->h_cg;
    if (res->failed) return fail(STA_ECUDA, "the solve's grid-wide sum did not complete");
    return STA_OK;
}

}  // namespace sta
