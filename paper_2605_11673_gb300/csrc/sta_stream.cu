// Streaming update (Sec. 3.2, Algorithm 1; the local_recompute policy of Sec. 3.5 made
// bitwise): apply a frame's mask changes, collect the fold units its edits touch, and re-fold
// exactly those with the rebuild's operands, order and operations.  Also the mask-to-activity
// pass of a full rebuild with a new mask.  Fold definition and shared device code:
// sta_fold.cuh.
#include <cstring>

#include "sta_bulk.cuh"
#include "sta_claim.cuh"
#include "sta_fold.cuh"

namespace sta {
namespace {

// ------------------------------------------------------------------------------------------
// Entry-parallel fold of a list of units (streaming).  A frame's touched list is short and its
// longest folds (diagonal units, ~24 contributions) set the latency, so here each lane folds ONE
// matrix entry, and one FP64 instruction per step advances a whole warp of folds.  The claim
// kernel lists the two kinds of unit apart (diagonal units from the front of the list, pair
// units from the back), so that a warp folds units of one kind: 5 diagonal units (lanes
// 6g .. 6g+5 fold the 6 entries i <= j of unit g) or 3 pair units (lanes 9g .. 9g+8 fold the
// 9 entries (i, j)).  A warp's step count is its longest fold, and on GB300 an FP64 warp
// instruction holds its SM quadrant's FP64 pipe for 64 cycles: mixing a ~24-contribution diagonal
// unit with ~6-contribution pair units would leave most of those steps idle.
// A lane's operands are one double of each active contributor's run, whose addresses follow from
// the unit record and its activity bits: it copies up to ENT_DEPTH of them into its column of
// shared memory with 8-byte cp.async, all in flight at once and none in a register, then adds them
// in order; only the lane itself reads its column, so no barrier is needed.
// Operands, order and operations are those of k_fold_flat, so the values are the same bits.
// ------------------------------------------------------------------------------------------
constexpr int ENT_DG = 5;      // diagonal units per warp round (6 lanes each: 30 lanes)
constexpr int ENT_PG = 3;      // pair units per warp round (9 lanes each: 27 lanes)
constexpr int ENT_DEPTH = 24;  // operands of a lane in flight
constexpr int ENT_WARPS = 4;

// One warp round over units first .. first+NG-1 of one kind of the n_units that unit(k) names;
// `col`: the lane's column of the warp's shared buffer.
template <bool DIAG, typename F>
__device__ __forceinline__ void fold_units(const FoldArgs &A, UnitState *ustate, F unit,
                                           int64_t first, int64_t n_units, double *col, int lane,
                                           bool has_eps) {
    constexpr int GW = DIAG ? RUN_DIAG : RUN_PAIR;   // lanes (entries) per unit
    constexpr int NG = DIAG ? ENT_DG : ENT_PG;       // units per warp round
    const int g = lane / GW, q = lane % GW;          // g == NG: idle lanes
    const int64_t k = first + g;
    const bool valid = g < NG && k < n_units;
    int4 bm = make_int4(0, 0, 0, 0);
    int2 mir = make_int2(0, 0);
    uint4 st = make_uint4(0, 0, 0, 0);
    int32_t u = 0;
    if (valid) {
        u = unit(k);
        bm = __ldg(A.bmeta + u);
        if (!DIAG) mir = __ldg(A.bmirror + u);
        st = __ldcg(reinterpret_cast<const uint4 *>(ustate + u));  // (claimed in this very kernel, or before)
    }
    ActiveRuns it(valid, st, bm.w, bm.z + q, GW, A.uext);
    const int n = it.count();
    const int maxn = __reduce_max_sync(0xffffffffu, n);
    double acc = 0.0;
    for (int j0 = 0; j0 < maxn; j0 += ENT_DEPTH) {  // warp-uniform
        const int c = n - j0 < ENT_DEPTH ? n - j0 : ENT_DEPTH;  // this lane's operands (may be < 0)
        const int cm = maxn - j0 < ENT_DEPTH ? maxn - j0 : ENT_DEPTH;
        for (int j = 0; j < c; ++j) cp_async<8>(col + 32 * j, A.Ke + it.next());
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        for (int j = 0; j < cm; ++j)
            if (j < c) acc = j0 + j == 0 ? plus_zero(col[0]) : acc + col[32 * j];
        __syncwarp();
    }
    if (!valid) return;
    // release the claim: all claims are done, and the other lanes of the unit do not read it
    if (q == 0) ustate[u].claims = 0;
    if (DIAG) {
        // 6-run entry q = (i, j), i <= j
        const int i = q < 3 ? 0 : (q < 5 ? 1 : 2), j = q < 3 ? q : (q < 5 ? q - 2 : 2);
        double a = acc;
        if (i == j && has_eps) a += A.eps;
        double *out = A.val + bm.x;
        const int rs = bm.y >> 1;
        out[i * rs + j] = a;
        if (i != j) out[j * rs + i] = a;
    } else {
        const int qi = q / 3, qj = q % 3;
        A.val[bm.x + qi * (bm.y >> 1) + qj] = acc;
        A.val[mir.x + qj * mir.y + qi] = acc;
    }
}

// count[0]: diagonal units | pair units << 32 (the claim kernel's); count[2] gets the frame's
// touched CSR entries (9 per diagonal unit, 18 = both blocks per pair unit), also stored into
// the host-mapped word `host_count` when given.  `cap`: the list's length.  `next_count`, when
// given, is the count pair of the next frame (graph mode alternates two), zeroed here so that
// the captured frame needs no memset node of its own.
__global__ void __launch_bounds__(ENT_WARPS * 32)
k_fold_entries(FoldArgs A, UnitState *ustate, const int32_t *list,
               unsigned long long *count, int64_t cap, unsigned long long *host_count,
               unsigned long long *next_count) {
    __shared__ double stage[ENT_WARPS][ENT_DEPTH * 32];
    const int lane = threadIdx.x & 31;
    double *col = stage[threadIdx.x >> 5] + lane;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    dependency_wait();
    const unsigned long long packed = *count;  // final: the claim kernel has ended
    const int64_t nd = (int64_t)(packed & 0xffffffffull), np = (int64_t)(packed >> 32);
    const int64_t gd = (nd + ENT_DG - 1) / ENT_DG, gp = (np + ENT_PG - 1) / ENT_PG;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long entries = 9ull * (unsigned long long)nd + 18ull * (unsigned long long)np;
        count[2] = entries;
        if (host_count) *host_count = entries;
        if (next_count) {
            next_count[0] = 0;
            next_count[2] = 0;
        }
    }
    const bool has_eps = A.eps != 0.0;
    for (int64_t item = warp; item < gd + gp; item += nwarps) {  // warp-uniform
        if (item < gd)
            fold_units<true>(A, ustate, [&](int64_t k) { return list[k]; }, item * ENT_DG, nd,
                             col, lane, has_eps);
        else
            fold_units<false>(A, ustate, [&](int64_t k) { return list[cap - 1 - k]; },
                              (item - gd) * ENT_PG, np, col, lane, has_eps);
    }
}

// Streaming, phase 1: apply the frame's mask changes and collect the touched fold units.  One
// thread per (edited tet k, unit slot s): it moves the contributor's activity bit and claims the
// slot's unit (claim_unit); the thread that wins appends the unit to the fold list, a diagonal
// unit (slots 0-3) at the front and a pair unit at the back of the `cap` entries, both counted by
// one CTA-aggregated atomic on counters[1] = diagonal units | pair units << 32 (a large frame's
// warps all appending to that one word serialise at the L2; per CTA there are 8 times fewer).
// The fold releases the claims and counts the touched entries.  The list order depends on
// scheduling, the values do not (each unit folds independently).  edited[k] = tet id | (new
// state << 31); the edited count is *m_dev if m_dev, else m; counters[1] starts at zero; a frame
// lists at most 10 units per edited tet and at most every unit once, so the two ends never meet
// when cap >= min(10 m, units).
constexpr int CLAIM_THREADS = 256;

template <bool REPLAY>
__global__ void __launch_bounds__(CLAIM_THREADS)
k_stream_claim(const int32_t *__restrict__ edited, int64_t m,
                               const int64_t *__restrict__ m_dev,
                               const int32_t *__restrict__ tunit,
                               const int32_t *__restrict__ tpos, UnitState *__restrict__ ustate,
                               uint32_t *__restrict__ uext, uint8_t *__restrict__ mask,
                               int32_t *__restrict__ list, int64_t cap,
                               unsigned long long *counters) {
    // per warp of the CTA: its packed winner counts, then its offset; the CTA's base
    __shared__ unsigned long long s_cnt[CLAIM_THREADS / 32];
    __shared__ unsigned long long s_base;
    const int64_t n = 10 * (m_dev ? *m_dev : m);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // the thread's first edit and its unit, which no kernel writes, before the wait: while the frame before
    // this one ends (direct launches of 600 edits back to back: 18.5-20 us -> 10.4, with the edits
    // read from host memory instead of copied)
    uint32_t w1 = 0;
    int32_t u1 = 0, p1 = 0;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x;
    if (first + threadIdx.x < n) {
        const int64_t i = first + threadIdx.x;
        w1 = (uint32_t)edited[i / 10];
        const int64_t k = 10 * (int64_t)(w1 & 0x7fffffffu) + i % 10;
        u1 = __ldg(tunit + k);
        p1 = __ldg(tpos + k);
    }
    dependency_wait();
    for (int64_t i0 = first; i0 < n; i0 += stride) {  // CTA-uniform
        const int64_t i = i0 + threadIdx.x;
        bool won = false, diag = false;
        int32_t u = 0;
        if (i < n) {
            const bool again = i0 != first;
            const uint32_t w = again ? (uint32_t)edited[i / 10] : w1;
            const int32_t t = (int32_t)(w & 0x7fffffffu);
            const uint32_t on = w >> 31;
            const int s = (int)(i % 10);
            if (s == 0) mask[t] = (uint8_t)on;
            u = again ? __ldg(tunit + 10 * (int64_t)t + s) : u1;
            diag = s < 4;
            won = claim_unit<REPLAY>(ustate, uext, u, again ? __ldg(tpos + 10 * (int64_t)t + s) : p1, on != 0u);
        }
        const unsigned dball = __ballot_sync(0xffffffffu, won && diag);
        const unsigned pball = __ballot_sync(0xffffffffu, won && !diag);
        // packed counts add without carries: each half stays below 2^32
        if (lane == 0)
            s_cnt[wid] = (unsigned long long)__popc(dball) | ((unsigned long long)__popc(pball) << 32);
        __syncthreads();
        if (threadIdx.x == 0) {  // exclusive prefix over the CTA's warps, one atomic for all
            unsigned long long tot = 0;
            for (int w = 0; w < CLAIM_THREADS / 32; ++w) {
                const unsigned long long v = s_cnt[w];
                s_cnt[w] = tot;
                tot += v;
            }
            s_base = tot ? atomicAdd(&counters[1], tot) : 0ull;
        }
        __syncthreads();
        const unsigned long long base = s_base + s_cnt[wid];
        __syncthreads();  // s_cnt and s_base are rewritten in the next round
        const unsigned below = (1u << lane) - 1u;
        if (won && diag) list[(base & 0xffffffffull) + __popc(dball & below)] = u;
        if (won && !diag) list[cap - 1 - (int64_t)((base >> 32) + __popc(pball & below))] = u;
    }
    launch_dependents();
}

// A small frame in one launch: a cluster of SF_CTAS CTAs, one an SM, claims the units of the frame's edits, which
// come by value with the launch, and after a cluster barrier each CTA folds the units that its own
// threads won, listed in its shared memory (diagonal units from the front, pair units from the
// back).  Such a frame is all latency: launch, drain and dependent round trips (edit count, edits,
// list, list count), which this kernel does not make or overlaps with the frame before.  Frames of 4
// edits back to back: 10.9 us as two kernels of a graph, 5.4 here; of 32 edits: 11.3 and 5.8 (7.4 with
// 8 CTAs, whose warps fold two rounds one after the other; 7.1 with 16 of 4 warps).
constexpr int SF_CTAS = 16;
constexpr int SF_WARPS = 7;  // (their operand columns: 42 KB)
constexpr int SF_THREADS = 32 * SF_WARPS;
constexpr int SF_ROUNDS = (10 * SMALL_FRAME + SF_CTAS * SF_THREADS - 1) / (SF_CTAS * SF_THREADS);

// Every thread of the cluster, whose earlier writes are visible afterwards.  The aligned forms want whole
// warps: each is brought together first, as it may come from a branch of one lane.
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct SmallFrame {
    int32_t m;
    int32_t edited[SMALL_FRAME];
};

template <bool REPLAY>
__global__ void __cluster_dims__(SF_CTAS, 1, 1) __launch_bounds__(SF_THREADS)
k_frame_small(const __grid_constant__ SmallFrame F, FoldArgs A, const int32_t *__restrict__ tunit,
              const int32_t *__restrict__ tpos, UnitState *ustate, uint32_t *uext,
              uint8_t *__restrict__ mask, unsigned long long *counters,
              unsigned long long *host_count) {  // (the folds read ustate's and uext's words through A)
    constexpr int CAP = SF_ROUNDS * SF_THREADS;
    __shared__ double stage[SF_WARPS][ENT_DEPTH * 32];
    __shared__ int32_t won[CAP];
    __shared__ int n_won[2];        // diagonal, pair units of this CTA
    __shared__ unsigned touched;    // of the cluster, in CTA 0
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < 2) n_won[threadIdx.x] = 0;
    if (threadIdx.x == 2) touched = 0u;
    // items are dealt to the CTAs in turn, so that each gets its share of a short frame; their edits
    // and units, which no kernel writes, are read before the wait, while the frame before ends
    uint32_t w[SF_ROUNDS];
    int32_t u[SF_ROUNDS], pos[SF_ROUNDS];
#pragma unroll
    for (int r = 0; r < SF_ROUNDS; ++r) {
        const int i = (int)((r * SF_THREADS + threadIdx.x) * SF_CTAS + blockIdx.x);
        if (i < 10 * F.m) {
            w[r] = (uint32_t)F.edited[i / 10];
            const int64_t k = 10 * (int64_t)(w[r] & 0x7fffffffu) + i % 10;
            u[r] = __ldg(tunit + k);
            pos[r] = __ldg(tpos + k);
        }
    }
    cluster_sync();
    dependency_wait();
#pragma unroll
    for (int r = 0; r < SF_ROUNDS; ++r) {
        const int i = (int)((r * SF_THREADS + threadIdx.x) * SF_CTAS + blockIdx.x);
        if (i < 10 * F.m) {
            const int s = i % 10;
            if (s == 0) mask[w[r] & 0x7fffffffu] = (uint8_t)(w[r] >> 31);
            if (claim_unit<REPLAY>(ustate, uext, u[r], pos[r], (w[r] >> 31) != 0u)) {
                if (s < 4) won[atomicAdd(&n_won[0], 1)] = u[r];
                else won[CAP - 1 - atomicAdd(&n_won[1], 1)] = u[r];
            }
        }
    }
    __syncthreads();
    const int nd = n_won[0], np = n_won[1];
    if (threadIdx.x == 0) {  // the touched entries of the frame, summed in CTA 0
        unsigned a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_addr(&touched)));
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a),
                     "r"((unsigned)(9 * nd + 18 * np)) : "memory");
    }
    // every claim and activity change of the frame is done and visible
    cluster_sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counters[3] = touched;
        *host_count = touched;
    }
    const bool has_eps = A.eps != 0.0;
    double *col = stage[wid] + lane;
    const int gd = (nd + ENT_DG - 1) / ENT_DG, gp = (np + ENT_PG - 1) / ENT_PG;
    for (int item = wid; item < gd + gp; item += SF_WARPS) {  // warp-uniform
        if (item < gd)
            fold_units<true>(A, ustate, [&](int64_t k) { return won[k]; }, item * ENT_DG, nd, col, lane, has_eps);
        else
            fold_units<false>(A, ustate, [&](int64_t k) { return won[CAP - 1 - k]; }, (item - gd) * ENT_PG, np,
                              col, lane, has_eps);
    }
}

// Activity bits of every unit from the mask (full rebuild with a new mask).  A CTA takes as many
// consecutive units as it has threads; their contributors stand side by side, so it reads them
// coalesced, BITS_WINDOW at a time, keeps one bit each in shared memory (a ballot per warp load), and
// then every thread cuts its unit's words out of the bits.  Bound by the gathers of the mask and
// their latency; a lane per unit over its own list needed a request per lane for the list as well.
// Pre-fractured block of 577,000 tetrahedra (5.8 M contributors, 0.9 M units): 33 -> 17 us.
constexpr int BITS_THREADS = 256, BITS_LOADS = 8;
constexpr int BITS_WINDOW = BITS_THREADS * BITS_LOADS;

__global__ void __launch_bounds__(BITS_THREADS, 8)
k_mask_bits(int64_t nunits, const int32_t *__restrict__ uc0, const int32_t *__restrict__ ctet,
            const uint8_t *__restrict__ mask, uint4 *__restrict__ ustate,
            uint32_t *__restrict__ uext) {
    __shared__ uint32_t bits[BITS_WINDOW / 32 + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t u0 = (int64_t)blockIdx.x * BITS_THREADS, u = u0 + threadIdx.x;
    const bool valid = u < nunits;
    const int32_t lo = __ldg(uc0 + u0);
    const int32_t hi = __ldg(uc0 + (u0 + BITS_THREADS < nunits ? u0 + BITS_THREADS : nunits));
    const int32_t b = valid ? __ldg(uc0 + u) : hi, e = valid ? __ldg(uc0 + u + 1) : hi;
    launch_dependents();  // (the fold's CTAs set up while the last of these run)
    dependency_wait();
    uint4 st = valid ? ustate[u] : make_uint4(0, 0, 0, 0);
    st.x = st.z = 0u;
    uint32_t word = 0;
    int32_t j = b;  // the unit's next contributor
    for (int32_t w0 = lo; w0 < hi; w0 += BITS_WINDOW) {
        int32_t t[BITS_LOADS];
#pragma unroll
        for (int k = 0; k < BITS_LOADS; ++k) {
            const int32_t i = w0 + k * BITS_THREADS + (int)threadIdx.x;
            t[k] = i < hi ? __ldg(ctet + i) : -1;
        }
        bool on[BITS_LOADS];
#pragma unroll
        for (int k = 0; k < BITS_LOADS; ++k) on[k] = t[k] >= 0 && __ldg(mask + t[k]);
#pragma unroll
        for (int k = 0; k < BITS_LOADS; ++k) {
            const uint32_t m = __ballot_sync(0xffffffffu, on[k]);
            if (lane == 0) bits[k * (BITS_THREADS / 32) + wid] = m;
        }
        __syncthreads();
        const int32_t end = e < w0 + BITS_WINDOW ? e : w0 + BITS_WINDOW;
        while (j < end) {  // the rest of one of the unit's words, as far as it is in the window
            const int at = (j - b) & 31, f = j - w0;
            const int n = 32 - at < end - j ? 32 - at : end - j;
            const uint32_t v = __funnelshift_r(bits[f >> 5], bits[(f >> 5) + 1], f & 31);
            word |= (n == 32 ? v : v & ((1u << n) - 1u)) << at;
            j += n;
            if (at + n == 32 || j == e) {
                const int w = (j - 1 - b) >> 5;
                if (w == 0) st.x = word;
                else if (w == 1) st.z = word;
                else uext[st.w + w - 2] = word;
                word = 0;
            }
        }
        __syncthreads();
    }
    if (valid) ustate[u] = st;
}

}  // namespace

int persistent_grid(const Ctx *c, const void *kernel, int threads, int64_t items, bool tuned) {
    int per_sm = tuned ? c->blocks_per_sm : 0;
    if (per_sm <= 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
    }
    int64_t need = (items + threads - 1) / threads;
    int64_t cap = (int64_t)per_sm * c->num_sms;
    int64_t g = need < cap ? need : cap;
    return (int)(g < 1 ? 1 : g);
}

int launch_fold_list(Ctx *c, const int32_t *list, int64_t cap, unsigned long long *count,
                     int64_t max_items, cudaStream_t s, unsigned long long *host_count,
                     unsigned long long *next_count) {
    const int threads = ENT_WARPS * 32;
    // a warp round per 3 units for the largest possible list (all pair units), at most the
    // resident CTAs
    const int grid = persistent_grid(c, (const void *)k_fold_entries, threads,
                                     (max_items + ENT_PG - 1) / ENT_PG * 32);
    return launch_overlapped(k_fold_entries, (unsigned)grid, threads, 0, s, fold_args(c), c->ustate, list,
                             count, cap, host_count, next_count);
}

int launch_mask_bits(Ctx *c, cudaStream_t s) {
    if (c->T == 0 || c->op == STA_OP_PROXY) return STA_OK;  // the proxy reads the mask itself
    const int64_t grid = (c->nunits + BITS_THREADS - 1) / BITS_THREADS;
    return launch_overlapped(k_mask_bits, (unsigned)grid, BITS_THREADS, 0, s, c->nunits, c->uc0, c->ctet,
                             c->mask, reinterpret_cast<uint4 *>(c->ustate), c->uext);
}

// Every value from the current mask: the operator's full rebuild.
int launch_values(Ctx *c, cudaStream_t s) {
    if (c->op == STA_OP_PROXY) return launch_proxy_rebuild(c, s);
    STA_TRY(launch_rebuild(c, s));
    return launch_dyn_mass_all(c, s);  // the lumped mass, when the dynamics are set up
}

// One streaming frame: claim kernel, then the fold of the touched units.  The edited count is *m_dev
// if given (a sequence captured once and replayed for any frame up to `cap`, for which the grids are
// sized), else m.  `next_cnt`: the counters of the next frame, which the frame's last kernel zeroes,
// or nullptr.  `replay`: see claim_unit.
int launch_stream_frame(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev,
                        unsigned long long *cnt, int64_t cap, cudaStream_t s,
                        unsigned long long *next_cnt, bool replay) {
    if (c->op == STA_OP_PROXY)
        return launch_proxy_frame(c, edited, m, m_dev, cap, c->plist, cnt, s, next_cnt);
    if (c->policy == STA_POLICY_FIXED) {
        STA_TRY(launch_fx_frame(c, edited, m, m_dev, cap, c->touched, cnt, s, next_cnt, replay));
        return launch_dyn_mass_edited(c, edited, m, m_dev, cap, s);
    }
    const int threads = CLAIM_THREADS;
    int64_t g = (10 * cap + threads - 1) / threads;
    const int64_t gmax = (int64_t)c->num_sms * 16;
    g = g < 1 ? 1 : (g > gmax ? gmax : g);
    STA_TRY(launch_overlapped(replay ? k_stream_claim<true> : k_stream_claim<false>, (unsigned)g, threads, 0, s,
                              edited, m, m_dev, c->tunit,
                              c->tpos, c->ustate, c->uext, c->mask, c->touched, c->nunits, cnt));
    STA_TRY(launch_fold_list(c, c->touched, c->nunits, cnt + 1, 10 * (cap > 0 ? cap : 1), s,
                             c->d_count_mapped, next_cnt ? next_cnt + 1 : nullptr));
    return launch_dyn_mass_edited(c, edited, m, m_dev, cap, s);
}

// Whether the device can run k_frame_small's cluster (more than 8 CTAs is not a size every one has).
bool small_frames_fit() {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SF_CTAS);
    cfg.blockDim = dim3(SF_THREADS);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = SF_CTAS;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    bool fits = true;
    for (auto kern : {k_frame_small<false>, k_frame_small<true>})
        fits = fits && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
               cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0;
    if (!fits) cudaGetLastError();
    return fits;
}

// A frame of m <= SMALL_FRAME edited tetrahedra (tet id | new state << 31, host memory) in one launch.
int launch_small_frame(Ctx *c, const int32_t *edited, int m, bool replay, cudaStream_t s) {
    SmallFrame F;
    F.m = m;
    std::memcpy(F.edited, edited, sizeof(int32_t) * m);
    return launch_overlapped(replay ? k_frame_small<true> : k_frame_small<false>, SF_CTAS, SF_THREADS, 0, s, F, fold_args(c), c->tunit, c->tpos,
                             c->ustate, c->uext, c->mask, c->counters, c->d_count_mapped);
}

bool frame_counts_to_host(const Ctx *c) {
    return c->op == STA_OP_ELASTICITY && c->policy == STA_POLICY_REFOLD && c->d_count_mapped;
}

// Streaming update with caller-chosen scratch (the allocation-free entry point): the same two
// kernels, with the edited-tet list, the touched-unit list and the counters at the given
// addresses; the touched counts are copied to the context's counters afterwards so that
// sta_last_touched reports them.
int launch_stream_scratch(Ctx *c, int64_t m, const int32_t *d_edited, int32_t *touched,
                          unsigned long long *counters, cudaStream_t s) {
    const bool replay = capturing(s);
    STA_CUDA_TRY(cudaMemsetAsync(counters + 1, 0, 3 * sizeof(unsigned long long), s));
    if (m > 0 && c->op == STA_OP_PROXY) {
        STA_TRY(launch_proxy_frame(c, d_edited, m, nullptr, m, touched, counters, s, nullptr));
    } else if (m > 0 && c->policy == STA_POLICY_FIXED) {
        STA_TRY(launch_fx_frame(c, d_edited, m, nullptr, m, touched, counters, s, nullptr, replay));
    } else if (m > 0) {
        const int threads = CLAIM_THREADS;
        const int64_t g = (10 * m + threads - 1) / threads;
        // the touched list holds 10 m units (at most 10 per edited tet)
        // (the claim reads d_edited before its dependency_wait: it was copied there before the
        // memset above, and a kernel that follows a memset starts when that is done)
        STA_TRY(launch_overlapped(replay ? k_stream_claim<true> : k_stream_claim<false>, (unsigned)g, threads, 0, s,
                                  d_edited, m, (const int64_t *)nullptr,
                                  c->tunit, c->tpos, c->ustate, c->uext, c->mask, touched, 10 * m,
                                  counters));
        STA_TRY(launch_fold_list(c, touched, 10 * m, counters + 1, 10 * m, s, nullptr, nullptr));
    }
    if (m > 0) STA_TRY(launch_dyn_mass_edited(c, d_edited, m, nullptr, m, s));
    // touched units and touched entries, for sta_last_touched
    STA_CUDA_TRY(cudaMemcpyAsync(c->counters + 1, counters + 1, 3 * sizeof(unsigned long long),
                                 cudaMemcpyDeviceToDevice, s));
    c->last_counters = c->counters;
    c->count_on_host = false;  // read back from the device counters
    return STA_OK;
}

}  // namespace sta
