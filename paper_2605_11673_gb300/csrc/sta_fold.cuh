// Fold kernels: the full rebuild and the streaming update.
//
// Both evaluate, for a node-pair block (a, b) of the superset pattern, the 9 CSR values
//   A[3a+i][3b+j] = fold_{tau active, ascending id} K^(tau)[3 la + i][3 lb + j]   (+ eps)
// i.e. Eq. 8 of STA-FEM restricted to one block, with the fold starting at +0.0 and eps
// added afterwards on the diagonal.  The work unit is an unordered node pair {a <= b}: the
// element matrices are stored exactly symmetric, so block (b, a) folds the same operands in
// the same order as (a, b) and one fold writes both.  The streaming pass (Sec. 3.2,
// Algorithm 1; the local_recompute policy of Sec. 3.5) folds the units touched by the frame's
// edits only, with the same operands, order and operations, so its values are bit-identical
// to the rebuild's.
//
// No atomics touch values: each entry is folded by exactly one lane, and the summation order
// is the order of the unit's contributor list (ascending tetrahedron id), independent of the
// kernel and the launch configuration.  Every fold starts with (+0.0 + c1) formed without an
// FP64 operation (plus_zero) and continues with one FP64 add per further contribution.
//
// This header holds what both folds share: the arguments, the +0.0 start, and the walk over a
// unit's active contributors.
#pragma once

#include "sta_internal.cuh"

namespace sta {
namespace {

struct FoldArgs {
    const int4 *__restrict__ bmeta;     // per unit: value offset of (a,b), rs_a << 1 | diag, first run, count
    const int2 *__restrict__ bmirror;   // per unit: value offset of (b,a), rs_b
    const UnitState *ustate;            // per unit: activity bits
    const uint32_t *uext;               // activity words of contributors 64 and up
    const double *__restrict__ Ke;
    double *__restrict__ val;
    double eps;
};

// 2^x for x in [-1022, 1023], exact (the fixed-point scale of an entry)
__device__ __forceinline__ double pow2i(int x) {
    return __longlong_as_double((long long)(x + 1023) << 52);
}

// +0.0 + v without an FP64 operation: identical except that -0.0 becomes +0.0.
__device__ __forceinline__ double plus_zero(double v) {
    long long bits = __double_as_longlong(v);
    return __longlong_as_double(bits == (long long)0x8000000000000000ULL ? 0LL : bits);
}

// The active contributors of one unit in list order, as offsets of their runs.  Every lane of a
// unit walks the same bits: no list is built, and the offset of the next operand is known without
// a load (but for the words of contributors 64 and up, plain loads: claims of the same kernel, or of
// one that still ran when this one started, change them).
struct ActiveRuns {
    uint32_t w, w1;       // bits left in the current word; word 1
    int32_t run, stride;  // offset of the current word's first run; doubles per run
    int32_t k, words;     // words passed; words after the first two
    const uint32_t *ext;
    __device__ __forceinline__ ActiveRuns(bool valid, const uint4 &st, int cnt, int32_t first,
                                          int32_t run_len, const uint32_t *uext)
        : w(valid ? st.x : 0u), w1(valid ? st.z : 0u), run(first), stride(run_len), k(0),
          words(valid && cnt > 64 ? (cnt + 31) / 32 - 2 : 0),
          ext(words > 0 ? uext + st.w : nullptr) {}
    // active contributors in all words (call before next)
    __device__ __forceinline__ int count() const {
        int n = __popc(w) + __popc(w1);
        for (int i = 0; i < words; ++i) n += __popc(ext[i]);
        return n;
    }
    // offset of the next active contributor's run; called at most count() times
    __device__ __forceinline__ int32_t next() {
        while (w == 0 && k <= words) {
            run += 32 * stride;
            w = k == 0 ? w1 : ext[k - 1];
            ++k;
        }
        const int j = __ffs(w) - 1;
        w &= w - 1;
        return run + stride * j;
    }
};

inline FoldArgs fold_args(const Ctx *c) {
    return FoldArgs{c->bmeta, c->bmirror, c->ustate, c->uext, c->Ke, c->val, c->eps};
}

}  // namespace
}  // namespace sta
