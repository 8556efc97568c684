// Full rebuild (the full_rebuild policy of Sec. 3.5): every value of the superset pattern folded
// from the element cache over the active mask, in FP64 or, under STA_POLICY_FIXED, as the
// fixed-point integer sum.  Fold definition and shared device code: sta_fold.cuh.
#include <type_traits>

#include "sta_bulk.cuh"
#include "sta_fold.cuh"

namespace sta {
namespace {

// ------------------------------------------------------------------------------------------
// The fold kernel.  A chunk is up to 28 consecutive pair units or 16 consecutive diagonal units
// whose runs are at most CHUNK_BYTES together (chunk records built at create).  Its operands are
// its units' runs of the element cache, which lie one unit after the other in memory: one copy
// brings them to shared memory, from the first active contributor's to the last one's; only a
// stretch of more than FOLD_GAP without an active contributor splits it (a copy costs the producer
// 80 cycles, the time of 3 KB at an SM's share of the bandwidth).
//
// One producer warp of a CTA walks the CTA's chunks (c, c + grid, ...): lane l reads unit l's
// record and activity (FOLD_AHEAD chunks ahead, by cp.async: with one chunk ahead in registers the
// producer's load latency was the kernel's time), leaves what the fold needs in the next stage of a
// ring of FOLD_STAGES and issues the chunk's copies.  The other FOLD_CONS warps fold, each a round
// of 32 fold entries of the chunk (6 per diagonal unit, 9 per pair unit): every lane folds one entry
// over its unit's active contributors from shared memory and writes it and its mirror.
// Where the active contributors of all the round's units stand side by side (most of a mesh: all of
// them, or the originals without the inactive copies behind them) operand j is at a fixed offset;
// else the lane walks its activity bits.  A unit of more than 64 contributors is a chunk of its
// own, folded from global memory.
//
// What bounds it: the FP64 pipe and HBM are close.  A fully active block of 384,000 tetrahedra: 1.0 M
// FP64 warp instructions, 50 us at one per quadrant and 64 cycles; 330 MB, 49 us at copy rate.  The
// kernel before held operands in registers, 4 to 8 loads of a lane at a time, after a list of run
// offsets compacted from per-contributor words (315 instructions a round): every tile waited for its
// loads, memory and FP64 pipe both at 45%.  Copies in flight cost no registers.  Measured, before ->
// now (L2 flushed, launch included): that block 101 -> 68 us, 48 blocks of 0.8 M tetrahedra 199 ->
// 138 us, pre-fractured block (384,000 of 577,000 active) 127 -> 102 us, the same in fixed point 197
// -> 164 us.  Two producers, 12 or 15 consumers, 2 or 4 CTAs an SM, chunks of 5 to 18 KB: within 5%,
// or slower.
// ------------------------------------------------------------------------------------------
constexpr int FOLD_CONS = 8;      // consumer warps: a round of a full pair chunk each
constexpr int FOLD_THREADS = 32 * (FOLD_CONS + 1);
constexpr int FOLD_STAGES = 5;
constexpr int FOLD_AHEAD = 4;     // chunks whose unit records are on their way
constexpr int FOLD_CTAS = 3;      // per SM: 15 chunks in the rings, up to 180 KB
static_assert(CHUNK_PAIR * RUN_PAIR <= 32 * FOLD_CONS && CHUNK_DIAG * RUN_DIAG <= 32 * FOLD_CONS,
              "a round per consumer warp");
constexpr int FOLD_GAP = 256;                      // doubles

// What a consumer lane needs of its unit.
struct __align__(16) UnitMeta {
    int32_t out, rs, out2, rs2;  // value offset and row stride of (a, b), of (b, a)
    uint32_t w0, w1;             // activity of contributors 0 .. 63
    int32_t base;                // run j starts at double base + stride * j of the stage
    int32_t info;                // active contributors | side by side << 8 | in global memory << 9 |
                                 //   the first active one << 16
};

struct FoldStage {
    double data[CHUNK_BYTES / 8];
    UnitMeta meta[CHUNK_PAIR];
    int32_t first, n, diag, pad;  // units of the chunk; n = 0: no more chunks
};

struct FoldShared {
    FoldStage stage[FOLD_STAGES];
    int4 bm[FOLD_AHEAD][32];
    uint4 st[FOLD_AHEAD][32];
    int2 mir[FOLD_AHEAD][32];
    uint64_t full[FOLD_STAGES], empty[FOLD_STAGES];
};

// Fixed-point operands of the fold (policy STA_POLICY_FIXED, sta_fixed.cu): the quantised
// contributions at the element-cache offsets, the exponent of each entry and the integer sums,
// keyed by the value index of the entry's upper block.
struct FxArgs {
    const long long *Kq;
    const int16_t *e;
    long long *S;
};

// The zero-fill form's chunks of one producer: the positions k = 0, 1, ... of its stripe (chunk
// b + k G) whose flag is set.  The flags of 32 positions are read at once (one per lane), those of
// the next 32 one step ahead, and handed out from a ballot.
struct FlagStream {
    int32_t base;    // stripe position of bit 0 of `mask`
    unsigned mask;   // set flags of positions base .. base+31 not yet handed out
    uint8_t ahead;   // this lane's flag of position base + 32 + lane
    __device__ __forceinline__ void load_ahead(const uint8_t *flags, int32_t b, int32_t G,
                                               int32_t n, int lane) {
        const int64_t t = b + (int64_t)(base + 32 + lane) * G;
        ahead = t < n ? __ldcg(flags + t) : 0;
    }
    // the next flagged chunk, or n past the end of the stripe
    __device__ __forceinline__ int32_t next(const uint8_t *flags, int32_t b, int32_t G,
                                            int32_t n, int lane) {
        while (mask == 0) {  // warp-uniform
            base += 32;
            if (b + (int64_t)base * G >= n) return n;
            mask = __ballot_sync(0xffffffffu, ahead != 0);
            load_ahead(flags, b, G, n, lane);
        }
        const int k = __ffs(mask) - 1;
        mask &= mask - 1;
        return b + (base + k) * G;
    }
};

// The place of a lane in round r of a chunk: entry q = (ei, ej) of the chunk's unit ul.
template <bool DIAG> struct Place {
    int ul, q, ei, ej, e;
    __device__ __forceinline__ Place(int r, int lane) {
        constexpr int W = DIAG ? RUN_DIAG : RUN_PAIR;
        e = 32 * r + lane;
        ul = e / W;
        q = e - W * ul;
        // 6-run entry q = (i, j), i <= j, of a diagonal unit; 3x3 row-major of a pair unit
        ei = DIAG ? (q < 3 ? 0 : (q < 5 ? 1 : 2)) : q / 3;
        ej = DIAG ? (q < 3 ? q : (q < 5 ? q - 2 : 2)) : q - 3 * (q / 3);
    }
};

// One lane's fold over its unit's active contributors from global memory, four loads in flight.
template <bool FX, typename V>
__device__ __forceinline__ V fold_global(const V *__restrict__ src, ActiveRuns run) {
    const int c = run.count();
    V acc = V(0);
    for (int j = 0; j < c; j += 4) {
        V v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = j + k < c ? __ldg(src + run.next()) : V(0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (j + k < c) {
                if constexpr (FX) acc += v[k];
                else acc = j + k == 0 ? plus_zero(v[k]) : acc + v[k];  // +0.0 + the first one
            }
    }
    return acc;
}

// An entry's value (and integer sum) to the entry and to its mirror.
template <bool FX, bool DIAG, typename V>
__device__ __forceinline__ void write_entry(const FoldArgs &A, const FxArgs &X, const Place<DIAG> &P,
                                            int32_t out, int32_t rs, int32_t out2, int32_t rs2,
                                            int32_t key, V acc, int ex) {
    double a;
    if constexpr (FX) {
        X.S[key] = acc;
        a = __ll2double_rn(acc) * pow2i(ex);
    } else {
        a = acc;
    }
    if (DIAG) {  // mirrored inside the block; eps on the diagonal
        if (P.ei == P.ej && A.eps != 0.0) a += A.eps;
        A.val[key] = a;
        if (P.ei != P.ej) A.val[out + P.ej * rs + P.ei] = a;
    } else {
        A.val[key] = a;
        A.val[out2 + P.ej * rs2 + P.ei] = a;
    }
}

// One round of a chunk of n units: 32 fold entries, one per lane.  Releases the stage (`empty`) once
// its operands are read.
template <bool FX, bool DIAG, typename V>
__device__ __forceinline__ void fold_round(const FoldArgs &A, const FxArgs &X, const V *src,
                                           const FoldStage &S, uint64_t *empty, int n,
                                           const Place<DIAG> &P, int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int W = DIAG ? RUN_DIAG : RUN_PAIR;
    const bool valid = P.e < n * W;
    const int ul = valid ? P.ul : 0, q = P.q, ei = P.ei, ej = P.ej;
    const UnitMeta m = S.meta[ul];
    const int32_t first = S.first;
    const int32_t key = m.out + ei * m.rs + ej;
    int ex = 0;  // the entry's fixed-point exponent, loaded before the fold
    if constexpr (FX) ex = valid ? (int)__ldg(X.e + key) : 0;
    const bool direct = valid && (m.info >> 9 & 1);
    const int cnt = valid && !direct ? m.info & 255 : 0;
    const int most = __reduce_max_sync(FULL, cnt);
    V acc = V(0);
    const V *d = reinterpret_cast<const V *>(S.data) + (m.base + q);
    if (__all_sync(FULL, cnt == 0 || (m.info >> 8 & 1))) {
        d += W * (m.info >> 16);
        if (cnt > 0) {
            if constexpr (FX) acc = d[0];
            else acc = plus_zero(d[0]);  // +0.0 + the first contribution, no FP64 add
        }
        // a warp's adds wait for one another, 64 cycles each; the next operand is read meanwhile
        // (one add per turn of the loop: an FP64 instruction holds its pipe also when no lane
        // takes part, so none may be issued past the round's longest fold)
        V v = cnt > 1 ? d[W] : V(0), x;
        for (int j = 1; j < most; j += 2) {
            x = j + 1 < cnt ? d[2 * W] : V(0);
            if (j < cnt) acc += v;
            if (j + 1 >= most) break;
            v = j + 2 < cnt ? d[3 * W] : V(0);
            if (j + 1 < cnt) acc += x;
            d += 2 * W;
        }
    } else {
        ActiveRuns run(cnt > 0, make_uint4(m.w0, 0u, m.w1, 0u), 0, 0, W, nullptr);
        if (cnt > 0) {
            if constexpr (FX) acc = d[run.next()];
            else acc = plus_zero(d[run.next()]);
        }
        V v = cnt > 1 ? d[run.next()] : V(0);
        for (int j = 1; j < most; ++j) {
            const V x = j + 1 < cnt ? d[run.next()] : V(0);
            if (j < cnt) acc += v;
            v = x;
        }
    }
    __syncwarp();
    if (lane == 0) bar_arrive(empty);
    if (direct) {
        const int4 bm = __ldg(A.bmeta + first + ul);
        const uint4 st = __ldcg(reinterpret_cast<const uint4 *>(A.ustate) + first + ul);
        acc = fold_global<FX, V>(src, ActiveRuns(true, st, bm.w, bm.z + q, W, A.uext));
    }
    if (valid) write_entry<FX, DIAG, V>(A, X, P, m.out, m.rs, m.out2, m.rs2, key, acc, ex);
}

// FX = false: the canonical FP64 fold.  FX = true: the same over the quantised contributions with
// int64 adds (integer pipe), then S_k stored and converted once, val = double(S_k) 2^e_k (+ eps on
// the diagonal).  ZF = false (fused form): every chunk, +0.0 for the units without an active
// contributor.  ZF = true (zero-fill form): the values were set to zero and the chunks to fold flagged
// by k_zero_fill; the producer visits only the flagged ones of its stripe.
template <bool FX, bool ZF>
__global__ void __launch_bounds__(FOLD_THREADS, FOLD_CTAS)
k_fold_flat(FoldArgs A, const int2 *__restrict__ chunks, int32_t nchunks,
            const uint8_t *cflag, FxArgs X, unsigned int *__restrict__ fault) {
    using V = typename std::conditional<FX, long long, double>::type;
    const V *src;
    if constexpr (FX) src = X.Kq; else src = A.Ke;
    extern __shared__ __align__(128) unsigned char smem[];
    FoldShared &sh = *reinterpret_cast<FoldShared *>(smem);
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < FOLD_STAGES; ++s) {
            bar_init(&sh.full[s], 1);
            bar_init(&sh.empty[s], FOLD_CONS);
        }
        bar_init_fence();
    }
    __syncthreads();
    dependency_wait();

    if (wid == FOLD_CONS) {  // producer
        const int32_t G = (int32_t)gridDim.x, b = (int32_t)blockIdx.x;
        FlagStream fs{-32, 0u, 0};
        if constexpr (ZF) fs.load_ahead(cflag, b, G, nchunks, lane);
        int32_t c = b - G;
        auto record = [&]() {  // of the CTA's next chunk, empty past the end
            int32_t k;
            if constexpr (ZF) k = fs.next(cflag, b, G, nchunks, lane);
            else k = c = c < nchunks - G ? c + G : nchunks;
            return k < nchunks ? __ldg(chunks + k) : make_int2(0, 0);
        };
        // one commit group per chunk; a lane reads back only what it copied
        auto fetch = [&](int2 r, int k) {
            if (lane < (r.y & 255)) {
                cp_async<16>(&sh.bm[k][lane], A.bmeta + r.x + lane);
                cp_async<16>(&sh.st[k][lane], A.ustate + r.x + lane);
                cp_async<8>(&sh.mir[k][lane], A.bmirror + r.x + lane);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        int2 recs[FOLD_AHEAD], last;  // of the chunks on their way; of the one after them
#pragma unroll
        for (int k = 0; k < FOLD_AHEAD; ++k) recs[k] = record();
        last = record();
#pragma unroll
        for (int k = 0; k < FOLD_AHEAD; ++k) fetch(recs[k], k);
        bool more = true;
        unsigned it = 0;
        while (more) {
#pragma unroll
            for (int k = 0; k < FOLD_AHEAD; ++k) {  // (unrolled: recs stays in registers)
                if (!more) break;
                const int2 rec = recs[k];
                asm volatile("cp.async.wait_group %0;" ::"n"(FOLD_AHEAD - 1) : "memory");
                const int n = rec.y & 255, dg = rec.y >> 8, W = dg ? RUN_DIAG : RUN_PAIR;
                more = n > 0;
                int4 bm = make_int4(0, 0, 0, 0);
                uint4 st = make_uint4(0, 0, 0, 0);
                int2 mir = make_int2(0, 0);
                if (lane < n) {
                    bm = sh.bm[k][lane];
                    st = sh.st[k][lane];
                    mir = sh.mir[k][lane];
                }
                recs[k] = last;
                last = record();
                fetch(recs[k], k);
                FoldStage &S = sh.stage[it % FOLD_STAGES];
                uint64_t *full = &sh.full[it % FOLD_STAGES];
                if (it >= FOLD_STAGES &&
                    !bar_wait(&sh.empty[it % FOLD_STAGES], ((it / FOLD_STAGES) - 1) & 1)) {
                    *fault = 1u;
                    more = false;
                    break;
                }
                // the unit's active runs: doubles s0 (even) .. s1 of the cache
                const bool wide = bm.w > 64, act = !wide && (st.x | st.z) != 0u;
                const int j0 = st.x ? __ffs(st.x) - 1 : 31 + __ffs(st.z);
                const int j1 = st.z ? 63 - __clz(st.z) : 31 - __clz(st.x);
                const int na = __popc(st.x) + __popc(st.z);
                const int s0 = act ? bm.z + ((W * j0) & ~1) : 0;
                const int s1 = act ? bm.z + ((W * (j1 + 1) + 1) & ~1) : 0;
                // units stand in address order: one piece from the first active run to the last
                const unsigned am = __ballot_sync(FULL, act);
                const int lo = __shfl_sync(FULL, s0, am ? __ffs(am) - 1 : 0);
                const int hi = __shfl_sync(FULL, s1, am ? 31 - __clz(am) : 0);
                int skip = lo;           // what precedes the unit in the cache and not in the stage
                bool head = act && s0 == lo;  // the lane copies the piece that starts at its unit
                int send = hi, total = hi - lo;
                if (total - (int)__reduce_add_sync(FULL, (unsigned)(s1 - s0)) > FOLD_GAP) {
                    // leave out the long stretches between active units
                    int before = s1;  // the end of the active units before this one
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(FULL, before, o);
                        if (lane >= o && y > before) before = y;
                    }
                    before = __shfl_up_sync(FULL, before, 1);
                    if (lane == 0) before = 0;
                    const bool gap = act && before > 0 && s0 - before > FOLD_GAP;
                    head = head || gap;
                    int left = gap ? s0 - before : 0;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(FULL, left, o);
                        if (lane >= o) left += y;
                    }
                    skip += left;
                    total -= __shfl_sync(FULL, left, 31);
                    const unsigned hm = __ballot_sync(FULL, head);
                    const unsigned later = lane < 31 ? hm >> (lane + 1) << (lane + 1) : 0u;
                    const int e2 = __shfl_sync(FULL, before, later ? __ffs(later) - 1 : 0);
                    if (later) send = e2;
                }
                const unsigned bytes = 8u * (unsigned)total;
                if (lane < n) {
                    UnitMeta m;
                    m.out = bm.x;
                    m.rs = bm.y >> 1;
                    m.out2 = mir.x;
                    m.rs2 = mir.y;
                    m.w0 = st.x;
                    m.w1 = st.z;
                    m.base = bm.z - skip;
                    m.info = wide ? 1 << 9 : (na | (act && j1 - j0 + 1 == na) << 8 | (act ? j0 : 0) << 16);
                    S.meta[lane] = m;
                }
                if (lane == 0) {
                    S.first = rec.x;
                    S.n = n;
                    S.diag = dg;
                }
                __syncwarp();
                if (lane == 0) bar_arrive_expect(full, bytes);
                __syncwarp();
                if (head) bulk_load(S.data + (s0 - skip), src + s0, 8u * (unsigned)(send - s0), full);
                ++it;
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }

    // consumers
    const Place<false> mine(wid, lane);  // a pair chunk's round is the warp of its number's
    int rot = 0;                         // the warp that takes the next diagonal chunk's first round
    for (unsigned it = 0;; ++it) {
        FoldStage &S = sh.stage[it % FOLD_STAGES];
        if (!bar_wait(&sh.full[it % FOLD_STAGES], (it / FOLD_STAGES) & 1)) {
            *fault = 1u;
            bar_wait(&sh.full[it % FOLD_STAGES], (it / FOLD_STAGES) & 1);  // copies still in flight
            break;
        }
        const int n = S.n;
        if (n == 0) break;
        uint64_t *empty = &sh.empty[it % FOLD_STAGES];
        if (S.diag) {
            const int rounds = (n * RUN_DIAG + 31) / 32;
            const int r = wid >= rot ? wid - rot : wid - rot + FOLD_CONS;
            rot += rounds;
            if (rot >= FOLD_CONS) rot -= FOLD_CONS;
            if (r < rounds)
                fold_round<FX, true, V>(A, X, src, S, empty, n, Place<true>(r, lane), lane);
            else if (lane == 0)
                bar_arrive(empty);
        } else if (32 * wid < n * RUN_PAIR) {
            fold_round<FX, false, V>(A, X, src, S, empty, n, mine, lane);
        } else if (lane == 0) {
            bar_arrive(empty);
        }
    }
}

// Zero-fill form, first pass.  Flags the chunks the fold must visit -- those with an active
// contributor, and with eps != 0 the diagonal ones -- from the units' activity (a warp per chunk,
// 512 contiguous bytes), and sets every value (and, for the fixed-point fold, every integer sum) to
// zero with 16-byte stores.
__global__ void k_zero_fill(const int2 *__restrict__ chunks, int32_t nchunks,
                            const UnitState *ustate, bool eps, uint8_t *__restrict__ cflag, double *__restrict__ val,
                            long long *__restrict__ S, int64_t nnz) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    launch_dependents();
    dependency_wait();
    for (int64_t c = tid >> 5; c < nchunks; c += nthreads >> 5) {  // warp-uniform
        const int2 r = __ldg(chunks + c);
        bool on = eps && r.y >> 8;
        if (lane < (r.y & 255)) {
            const uint4 st = __ldcg(reinterpret_cast<const uint4 *>(ustate) + r.x + lane);
            on = on || (st.x | st.z) != 0u || st.w != UNIT_NARROW;
        }
        on = __any_sync(0xffffffffu, on);
        if (lane == 0) cflag[c] = on;
    }
    // (both arrays are cudaMalloc'd, 256-byte aligned; an odd last word alone)
    const int64_t pairs = nnz >> 1;
    auto fill = [&](void *p) {
        int4 *q = reinterpret_cast<int4 *>(p);
        int64_t i = tid;
        for (; i + 3 * nthreads < pairs; i += 4 * nthreads) {
#pragma unroll
            for (int k = 0; k < 4; ++k) q[i + k * nthreads] = make_int4(0, 0, 0, 0);
        }
        for (; i < pairs; i += nthreads) q[i] = make_int4(0, 0, 0, 0);
    };
    fill(val);
    if (S) fill(S);
    if (tid == 0 && (nnz & 1)) {
        val[nnz - 1] = 0.0;
        if (S) S[nnz - 1] = 0;
    }
}

// The fold of a small pattern: a warp per round, operands straight from global memory.  With one or
// two chunks per resident CTA of k_fold_flat its pipeline has little to overlap and its start-up
// costs more than it gives; the integer fold, whose adds are short, and a pattern that would be
// zero-filled first (this writes every value) gain longer.  Measured, this / the ring, back to back:
// blocks of 1,296 tetrahedra 6.4 / 8.4 us, 16,464: 9.5 / 9.5, 48,000: 16.5 / 14.4, that in fixed
// point 12.4 / 14.4; refinement hierarchy of 27,600 tetrahedra 10.3 / 13.7 (zero-fill form).
constexpr int SMALL_CHUNKS = 2, SMALL_CHUNKS_LONG = 8;  // per resident CTA of k_fold_flat

template <bool FX, bool DIAG>
__device__ __forceinline__ void small_round(const FoldArgs &A, const FxArgs &X, int2 rec, int r, int lane) {
    using V = typename std::conditional<FX, long long, double>::type;
    constexpr int W = DIAG ? RUN_DIAG : RUN_PAIR;
    const V *src;
    if constexpr (FX) src = X.Kq; else src = A.Ke;
    const Place<DIAG> P(r, lane);
    if (P.e >= (rec.y & 255) * W) return;
    const int32_t u = rec.x + P.ul;
    const int4 bm = __ldg(A.bmeta + u);
    const int2 mir = __ldg(A.bmirror + u);
    const uint4 st = reinterpret_cast<const uint4 *>(A.ustate)[u];
    const int32_t key = bm.x + P.ei * (bm.y >> 1) + P.ej;
    int ex = 0;
    if constexpr (FX) ex = (int)__ldg(X.e + key);
    const V acc = fold_global<FX, V>(src, ActiveRuns(true, st, bm.w, bm.z + P.q, W, A.uext));
    write_entry<FX, DIAG, V>(A, X, P, bm.x, bm.y >> 1, mir.x, mir.y, key, acc, ex);
}

template <bool FX>
__global__ void __launch_bounds__(32 * FOLD_CONS)
k_fold_small(FoldArgs A, const int2 *__restrict__ chunks, FxArgs X) {
    const int2 rec = __ldg(chunks + blockIdx.x);
    const int r = threadIdx.x >> 5, lane = threadIdx.x & 31;
    dependency_wait();
    if (rec.y >> 8) small_round<FX, true>(A, X, rec, r, lane);
    else small_round<FX, false>(A, X, rec, r, lane);
}

template <bool FX, bool ZF>
int launch_fold(Ctx *c, cudaStream_t s) {
    const FxArgs X{c->fx_q, c->fx_e, c->fx_s};
    const FoldArgs A = fold_args(c);
    if (c->nchunks <= (int64_t)(FX || ZF ? SMALL_CHUNKS_LONG : SMALL_CHUNKS) * FOLD_CTAS * c->num_sms) {
        return launch_overlapped(k_fold_small<FX>, (unsigned)c->nchunks, 32 * FOLD_CONS, 0, s, A,
                                 (const int2 *)c->chunks, X);
    }
    if (ZF)
        STA_TRY(launch_overlapped(k_zero_fill, c->num_sms * 8, 256, 0, s, (const int2 *)c->chunks,
                                  (int32_t)c->nchunks, (const UnitState *)c->ustate, c->eps != 0.0, c->cflag,
                                  c->val, FX ? c->fx_s : nullptr, c->nnz));
    STA_CUDA_TRY(cudaFuncSetAttribute(k_fold_flat<FX, ZF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(FoldShared)));
    int per_sm = c->blocks_per_sm;
    if (per_sm <= 0 || per_sm > FOLD_CTAS) per_sm = FOLD_CTAS;
    const int64_t cap = (int64_t)per_sm * c->num_sms;
    const unsigned grid = (unsigned)(c->nchunks < cap ? c->nchunks : cap);
    return launch_overlapped(k_fold_flat<FX, ZF>, grid, FOLD_THREADS, sizeof(FoldShared), s, A,
                             (const int2 *)c->chunks, (int32_t)c->nchunks, (const uint8_t *)c->cflag, X,
                             c->d_fault);
}

}  // namespace

// AUTO: the zero-fill form while fewer than 40% of the tetrahedra are active.  Measured on
// GB300: a refinement hierarchy with 12% of its superset active rebuilds in about a third of
// the fused form's time; a pre-fractured block with 66% active is faster fused.
int rebuild_form_of(const Ctx *c) {
    if (c->rebuild_form != STA_REBUILD_AUTO) return c->rebuild_form;
    return c->n_active * 5 < c->T * 2 ? STA_REBUILD_ZERO_FILL : STA_REBUILD_FUSED;
}

// Full rebuild in the context's form (rebuild_form_of: fused, or zero fill + fold of the chunks
// with an active contributor).
int launch_rebuild(Ctx *c, cudaStream_t s) {
    if (c->nchunks == 0) return STA_OK;
    const bool fx = c->policy == STA_POLICY_FIXED;
    if (rebuild_form_of(c) == STA_REBUILD_ZERO_FILL)
        return fx ? launch_fold<true, true>(c, s) : launch_fold<false, true>(c, s);
    return fx ? launch_fold<true, false>(c, s) : launch_fold<false, false>(c, s);
}

}  // namespace sta
