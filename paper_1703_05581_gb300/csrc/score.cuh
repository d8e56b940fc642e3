// Shared by the two profile scorers (Algorithm 1 and Algorithm 2): the group
// of base periods one launch scores, the profile's layout in shared memory
// and small device helpers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace ffa {

// The base periods scored by one launch: records [t0[i], t0[i + 1]) belong
// to entry i, whose profiles have p0[i] bins and whose plane starts at
// element off[i] of `prof` with rows ld[i] elements apart (all share m_rows
// and the widths); record it of entry i goes to rec[i][it - t0[i]].  A
// single base period is a group of one.  Entries may come from different
// series (a batch): each has its own records.
struct ScoreGroup {
    int32_t n;
    int64_t t0[FOLD_GROUP_MAX + 1];
    int32_t p0[FOLD_GROUP_MAX];
    int64_t off[FOLD_GROUP_MAX];
    int64_t ld[FOLD_GROUP_MAX];
    ffa_record* rec[FOLD_GROUP_MAX];
};

__device__ __forceinline__ int score_entry(const ScoreGroup& g, int64_t it) {
    int lo = 0, hi = g.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.t0[mid] <= it) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// One base period (or `count` ready profiles of p0 bins), and a group of n
// base periods sharing m_rows (*p0max: the longest profile).
ScoreGroup score_single(int64_t p0, int64_t ld, int64_t count, ffa_record* d_rec);
ScoreGroup score_group(int n, const int64_t* p0, const int64_t* off, int64_t m_rows, ffa_record* const* recs,
                       int64_t* p0max);

constexpr double KMAD = 1.4826;  // printed after Eq. 4

// ---- float-float ------------------------------------------------------------
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (h, l) += (bh, bl), h not renormalised (the low parts accumulate)
__device__ __forceinline__ void ff_acc(float& h, float& l, float bh, float bl) {
    float s, e;
    two_sum(h, bh, s, e);
    h = s;
    l = __fadd_rn(l, __fadd_rn(e, bl));
}
// h = fl(h + l), l = the rest: the canonical pair of the sum
__device__ __forceinline__ void ff_norm(float& h, float& l) {
    const float s = __fadd_rn(h, l);
    l = __fsub_rn(l, __fsub_rn(s, h));
    h = s;
}

__device__ __forceinline__ int as_bits(float v) { return __float_as_int(v); }
__device__ __forceinline__ int as_bits(int32_t v) { return v; }

// Three-input maximum in one instruction (sm_100 family); NaN is ignored as by fmaxf.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ int max3(int a, int b, int c) { return max(max(a, b), c); }

// Warp maximum in one instruction (redux.sync; the .f32 form is new with the
// sm_100 family).
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }

// ---- the profile in shared memory ----------------------------------------------
// The profile is cut into blocks of R bins (R = 8, 16 or 32).  Quads of four
// bins are XOR-swizzled inside their block so that both access patterns are
// free of bank conflicts without padding: consecutive bins (loading), and
// quad s of consecutive blocks (lanes of a warp on consecutive blocks).
template <int R>
__device__ __forceinline__ uint32_t blk_addr(uint32_t b) {  // byte address of block b's quad 0
    constexpr uint32_t QB = R / 4;
    return b * (R * 4) + ((((b * QB) >> 3) & (QB - 1)) << 4);
}
// quad s of the block at address a is at a ^ (s << 4)
template <int R>
__device__ __forceinline__ uint32_t bin_addr(uint32_t j) {  // byte address of bin j
    constexpr uint32_t QB = R / 4;
    return (((j << 2) & ~15u) ^ (((j >> 5) & (QB - 1)) << 4)) | ((j & 3) << 2);
}

}  // namespace ffa
