// Shared by the two profile scorers (Algorithm 1 and Algorithm 2): the group
// of base periods one launch scores, the profile's layout in shared memory
// and small device helpers.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

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
    return (j << 2) ^ ((j >> 1) & ((R / 4 - 1) << 4));
}

// The block offsets' element: float-float (a float2) or wrapping int32.
template <class V>
struct Offset {
    using type = float2;
};
template <>
struct Offset<int32_t> {
    using type = int32_t;
};
// Difference of two block offsets, box sums of prefixes: wrapping for int
// profiles (exact for box sums below 2^31), rounded to nearest for float.
__device__ __forceinline__ float off_diff(float2 b, float2 a) {
    return __fadd_rn(__fsub_rn(b.x, a.x), __fsub_rn(b.y, a.y));
}
__device__ __forceinline__ int32_t off_diff(int32_t b, int32_t a) { return (int32_t)((uint32_t)b - (uint32_t)a); }
__device__ __forceinline__ float box_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ int32_t box_sub(int32_t a, int32_t b) { return (int32_t)((uint32_t)a - (uint32_t)b); }
__device__ __forceinline__ float box_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ int32_t box_add(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }
__device__ __forceinline__ float box_lowest(float) { return -INFINITY; }
__device__ __forceinline__ int32_t box_lowest(int32_t) { return INT32_MIN; }

template <bool ONE>
__device__ __forceinline__ void cta_sync() {
    if (ONE) __syncwarp();
    else __syncthreads();
}

template <class V>
__device__ __forceinline__ void load_quad(const unsigned char* smem, uint32_t a, V (&v)[4]) {
    *reinterpret_cast<int4*>(v) = *reinterpret_cast<const int4*>(smem + a);
}
template <class V, int R>
__device__ __forceinline__ V load_bin(const unsigned char* smem, uint32_t j) {
    return *reinterpret_cast<const V*>(smem + bin_addr<R>(j));
}

// Load a profile into shared memory: hrow's p0 bins, plus (two) trow's read
// sft bins further on, four bins at a time; acc(v) sees every bin once (and
// the quad that straddles the wrap a second time, with other tail bins: it
// only takes statistics that guide a search).  Four quads' loads are issued
// before any is used, without a branch between them -- one quad in flight per
// thread took 8.9k of 29.7k SM cycles per profile of 19977 bins.
template <class V, int R, class Acc>
__device__ __forceinline__ void load_profile(unsigned char* smem, const V* __restrict__ hrow, const V* __restrict__ trow,
                                             int sft, bool two, int p0, int tid, int T, Acc acc) {
    constexpr int U = 4;
    auto store_quad = [&](int q, const V (&v)[4]) {
        *reinterpret_cast<int4*>(smem + (((uint32_t)q ^ (((uint32_t)q >> 3) & (R / 4 - 1))) << 4)) =
            *reinterpret_cast<const int4*>(v);
    };
    const int nq4 = p0 >> 2;
    auto tail_at = [&](int j) { return trow[j + sft < p0 ? j + sft : j + sft - p0]; };
    // AL: hrow is 16-byte aligned.  q < nq4; the tail's quad is read from the
    // last position that lies inside the row if it wraps.
    auto load_quads = [&](auto al, auto tw, int q0, int n) {
        constexpr bool AL = decltype(al)::value, TW = decltype(tw)::value;
        V h[U][4], t[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (u >= n) break;
            const int q = q0 + u * T;
            if (AL) {
                *reinterpret_cast<int4*>(h[u]) = *reinterpret_cast<const int4*>(hrow + 4 * q);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) h[u][i] = hrow[4 * q + i];
            }
            if (TW) {
                int o = 4 * q + sft;
                o = o >= p0 ? o - p0 : o;
                o = min(o, p0 - 4);
#pragma unroll
                for (int i = 0; i < 4; ++i) t[u][i] = trow[o + i];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (u >= n) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (TW) h[u][i] = h[u][i] + t[u][i];
                acc(h[u][i]);
            }
            store_quad(q0 + u * T, h[u]);
        }
    };
    auto load_all = [&](auto al, auto tw) {
        int q = tid;
        for (; q + (U - 1) * T < nq4; q += U * T) load_quads(al, tw, q, U);
        for (; q < nq4; q += T) load_quads(al, tw, q, 1);
    };
    const bool al = (reinterpret_cast<uintptr_t>(hrow) & 15) == 0;
    if (two) {
        if (al) load_all(std::true_type{}, std::true_type{});
        else load_all(std::false_type{}, std::true_type{});
        // the quad whose tail wraps, by the thread that stored it
        const int qw = (p0 - sft) >> 2;
        if (sft != 0 && ((p0 - sft) & 3) && qw < nq4 && tid == qw % T) {
            V v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                v[i] = hrow[4 * qw + i] + tail_at(4 * qw + i);
                acc(v[i]);
            }
            store_quad(qw, v);
        }
    } else {
        if (al) load_all(std::true_type{}, std::false_type{});
        else load_all(std::false_type{}, std::false_type{});
    }
    if (tid < (p0 & 3)) {
        const int j = 4 * nq4 + tid;
        V v = hrow[j];
        if (two) v = v + tail_at(j);
        *reinterpret_cast<V*>(smem + bin_addr<R>(j)) = v;
        acc(v);
    }
}

// Cyclic extension: bins p0 .. nbx * R - 1 repeat the profile.  A quad of the
// extension is four consecutive bins of the profile from a start of one
// residue mod 4: two quads read, one written.
template <class V, int R>
__device__ __forceinline__ void extend_profile(unsigned char* smem, int p0, int nbx, int first, int step) {
    const int ext = nbx * R - p0;
    if (ext > p0 - 4) {  // wraps again (short profiles): bin by bin
        for (int j = first; j < ext; j += step) {
            int s = j;
            while (s >= p0) s -= p0;
            *reinterpret_cast<V*>(smem + bin_addr<R>(p0 + j)) = load_bin<V, R>(smem, s);
        }
        return;
    }
    const int lead = (4 - (p0 & 3)) & 3;  // bins up to the first whole quad
    if (first < lead) *reinterpret_cast<V*>(smem + bin_addr<R>(p0 + first)) = load_bin<V, R>(smem, first);
    auto quad_addr = [](uint32_t q) { return (q ^ ((q >> 3) & (R / 4 - 1))) << 4; };
    const int q0 = (p0 + lead) >> 2, nq = (ext - lead) >> 2;  // nbx * R is a multiple of 4
    const bool b0 = lead & 1, b1 = lead & 2;
    for (int q = first; q < nq; q += step) {
        V r[8], t[6], v[4];
        load_quad(smem, quad_addr((uint32_t)q), *reinterpret_cast<V(*)[4]>(&r[0]));
        load_quad(smem, quad_addr((uint32_t)q + 1), *reinterpret_cast<V(*)[4]>(&r[4]));
#pragma unroll
        for (int i = 0; i < 6; ++i) t[i] = b0 ? r[i + 1] : r[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = b1 ? t[i + 2] : t[i];
        *reinterpret_cast<int4*>(smem + quad_addr((uint32_t)(q0 + q))) = *reinterpret_cast<const int4*>(v);
    }
}

// Sum of two float-float pairs, as a canonical pair.
__device__ __forceinline__ void ff_add(float& ah, float& al, float bh, float bl) {
    float s, e;
    two_sum(ah, bh, s, e);
    e = __fadd_rn(e, __fadd_rn(al, bl));
    ah = __fadd_rn(s, e);
    al = __fsub_rn(e, __fsub_rn(ah, s));
}
// The same on two pairs at once, in packed FP32 instructions.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tsub.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ void ff_add2(float2& ah, float2& al, float2 bh, float2 bl) {
    const float2 s = add2(ah, bh), bb = sub2(s, ah);
    float2 e = add2(sub2(ah, sub2(s, bb)), sub2(bh, bb));
    e = add2(e, add2(al, bl));
    ah = add2(s, e);
    al = sub2(e, sub2(ah, s));
}
// Inclusive scan over the lanes [0, n) of a warp (n <= 32).
__device__ __forceinline__ void ff_warp_scan(float& h, float& l, int n) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        if (o >= n) break;
        const float uh = __shfl_up_sync(0xffffffffu, h, o), ul = __shfl_up_sync(0xffffffffu, l, o);
        if (lane >= o) ff_add(h, l, uh, ul);
    }
}
// Two scans over 32 lanes at once (h and l per scan in x and y).  A lane with
// no neighbour adds zero, which leaves a canonical pair as it is.
__device__ __forceinline__ void ff_warp_scan2(float2& h, float2& l) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        float2 uh, ul;
        uh.x = __shfl_up_sync(0xffffffffu, h.x, o);
        uh.y = __shfl_up_sync(0xffffffffu, h.y, o);
        ul.x = __shfl_up_sync(0xffffffffu, l.x, o);
        ul.y = __shfl_up_sync(0xffffffffu, l.y, o);
        if (lane < o) uh = ul = make_float2(0.0f, 0.0f);
        ff_add2(h, l, uh, ul);
    }
}

constexpr int SCORE_MAXSEG = 64;  // segments of 32 blocks of the longest profile with its extension

// Block offsets: the exclusive scan of the block totals that offs holds (a
// float2's x).  Float sums have one tree whatever the CTA's size: a scan over
// 32 blocks, a scan over the segments' totals within `group` blocks (1024 /
// 512 / 256 by profile length), and the groups one after another.  Ends with
// a barrier.
template <class V, bool ONE>
__device__ __forceinline__ void scan_offsets(typename Offset<V>::type* offs, float2* seg, int nbx, int group) {
    constexpr bool INT = !std::is_same<V, float>::value;
    const int lane = threadIdx.x & 31, warp = ONE ? 0 : threadIdx.x >> 5, NW = ONE ? 1 : blockDim.x >> 5;
    if constexpr (INT) {
        // wrapping sums have no order: 128 blocks a segment, four per lane
        const int nseg = (nbx + 127) >> 7;
        uint32_t ci = 0;  // ONE: carry
        for (int sgm = warp; sgm < nseg; sgm += NW) {
            const int b0 = (sgm << 7) + 4 * lane;
            uint32_t v[4], s = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = b0 + i < nbx ? (uint32_t)offs[b0 + i] : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t u = v[i];
                v[i] = s;
                s += u;
            }
            uint32_t x = s;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += u;
            }
            const uint32_t ex = x - s + ci;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (b0 + i < nbx) offs[b0 + i] = (int)(ex + v[i]);
            const uint32_t tot = __shfl_sync(0xffffffffu, x, 31);
            if (ONE) ci += tot;
            else if (lane == 0) seg[sgm].x = __uint_as_float(tot);
        }
        cta_sync<ONE>();
        if (!ONE && nseg > 1) {
            for (int sgm = warp ? warp : NW; sgm < nseg; sgm += NW) {
                uint32_t base = 0;
                for (int i = 0; i < sgm; ++i) base += __float_as_uint(seg[i].x);
                for (int b = (sgm << 7) + lane; b < nbx && b < (sgm + 1) << 7; b += 32)
                    offs[b] = (int)((uint32_t)offs[b] + base);
            }
            __syncthreads();
        }
    } else {
        const int nseg = (nbx + 31) >> 5, per = group >> 5;  // segments, segments a group
        for (int pair = warp; 2 * pair < nseg; pair += NW) {  // two segments at a time
            const int b = (pair << 6) + lane;
            float2 h, l = make_float2(0.0f, 0.0f);
            h.x = b < nbx ? offs[b].x : 0.0f;
            h.y = b + 32 < nbx ? offs[b + 32].x : 0.0f;
            ff_warp_scan2(h, l);
            if (lane == 31) {
                seg[2 * pair] = make_float2(h.x, l.x);
                seg[2 * pair + 1] = make_float2(h.y, l.y);
            }
            float2 p, r;
            p.x = __shfl_up_sync(0xffffffffu, h.x, 1);
            p.y = __shfl_up_sync(0xffffffffu, l.x, 1);
            r.x = __shfl_up_sync(0xffffffffu, h.y, 1);
            r.y = __shfl_up_sync(0xffffffffu, l.y, 1);
            if (lane == 0) p = r = make_float2(0.0f, 0.0f);
            if (b < nbx) offs[b] = p;
            if (b + 32 < nbx) offs[b + 32] = r;
        }
        cta_sync<ONE>();
        float th = 0.0f, tl = 0.0f;  // total of the group before
        for (int g0 = 0; g0 < nseg; g0 += per) {
            const int ng = nseg - g0 < per ? nseg - g0 : per;
            float h = 0.0f, l = 0.0f;
            if (lane < ng) {
                const float2 t = seg[g0 + lane];
                h = t.x;
                l = t.y;
            }
            ff_warp_scan(h, l, ng);
            // segments of this group dealt out as above
            const int first = g0 + (warp + NW - g0 % NW) % NW;
            for (int sgm = first; sgm < g0 + ng; sgm += NW) {
                float bh = __shfl_sync(0xffffffffu, h, sgm - g0 - 1), bl = __shfl_sync(0xffffffffu, l, sgm - g0 - 1);
                if (sgm == g0) bh = bl = 0.0f;
                const int b = (sgm << 5) + lane;
                if (b < nbx) {
                    const float2 p = offs[b];
                    ff_add(bh, bl, p.x, p.y);
                    if (g0) {
                        float rh = th, rl = tl;
                        ff_add(rh, rl, bh, bl);
                        bh = rh;
                        bl = rl;
                    }
                    offs[b] = make_float2(bh, bl);
                }
            }
            th = __shfl_sync(0xffffffffu, h, ng - 1);  // one extension group at most follows
            tl = __shfl_sync(0xffffffffu, l, ng - 1);
        }
        cta_sync<ONE>();
    }
}

// Widths 2^n of wmask: M[n] = the largest box of width 2^n that starts in
// this thread's items (first, first + step, ... < nitem; an item is min(R, 16)
// bins of a block).  A block's largest box is its offset difference plus its
// largest difference of in-block prefixes (rounding is monotone).
template <class V, int R, int NS>
__device__ __forceinline__ void width_maxima(const unsigned char* smem, const typename Offset<V>::type* offs,
                                             uint32_t wmask, int first, int step, int nitem, V (&M)[NS]) {
    constexpr int P = R < 16 ? R : 16;
    constexpr int PARTS = R / P;
    constexpr int LR = R == 8 ? 3 : (R == 16 ? 4 : 5);
    const V lowest = box_lowest((V)0);
#pragma unroll
    for (int n = 0; n < NS; ++n) M[n] = lowest;
    for (int im = first; im < nitem; im += step) {
        const int b = im / PARTS, hf = im % PARTS;
        const uint32_t a = blk_addr<R>((uint32_t)b) ^ (uint32_t)(hf * (P * 4));
        const auto o1 = offs[b];
        V c[P];
#pragma unroll
        for (int s = 0; s < P / 4; ++s) load_quad(smem, a ^ (s << 4), *reinterpret_cast<V(*)[4]>(&c[4 * s]));
        // the next part: the same block's (offset 0), or the next block's
        const bool last = hf == PARTS - 1;
        const uint32_t an = last ? blk_addr<R>((uint32_t)b + 1) : a ^ (uint32_t)(P * 4);
        V xd = 0;
        if (last) xd = off_diff(offs[b + 1], o1);
        if (wmask & 15u) {
            V nx[8];
            load_quad(smem, an, *reinterpret_cast<V(*)[4]>(&nx[0]));
            if (R > 8) load_quad(smem, an ^ 16, *reinterpret_cast<V(*)[4]>(&nx[4]));
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                if ((1 << n) >= R || !(wmask >> n & 1u)) continue;
                const int w = 1 << n;
                V m = lowest, mx = lowest;
#pragma unroll
                for (int r = 0; r + w < P; r += 2) {
                    if (r + 1 + w < P) m = max3(m, box_sub(c[r + w], c[r]), box_sub(c[r + 1 + w], c[r + 1]));
                    else m = max3(m, m, box_sub(c[r + w], c[r]));
                }
#pragma unroll
                for (int i = 0; i < w; i += 2) {
                    if (i + 1 < w) mx = max3(mx, box_sub(nx[i], c[P - w + i]), box_sub(nx[i + 1], c[P - w + i + 1]));
                    else mx = max3(mx, mx, box_sub(nx[i], c[P - w + i]));
                }
                M[n] = max3(M[n], m, box_add(xd, mx));
            }
        }
        if (R == 32 && (wmask >> 4 & 1u)) {  // width 16 = one part further on
            V m = lowest;
#pragma unroll
            for (int s = 0; s < P / 4; ++s) {
                V v[4];
                load_quad(smem, an ^ (s << 4), v);
                m = max3(m, box_sub(v[0], c[4 * s]), box_sub(v[1], c[4 * s + 1]));
                m = max3(m, box_sub(v[2], c[4 * s + 2]), box_sub(v[3], c[4 * s + 3]));
            }
            M[4] = max3(M[4], M[4], box_add(xd, m));
        }
#pragma unroll
        for (int n = LR; n < NS; ++n) {
            if (!(wmask >> n & 1u)) continue;
            const int d = 1 << (n - LR);
            // eight or more blocks on, the swizzle is the same
            const uint32_t a2 =
                d >= 8 ? a + (uint32_t)(d * R * 4) : blk_addr<R>((uint32_t)(b + d)) ^ (uint32_t)(hf * (P * 4));
            const V D = off_diff(offs[b + d], o1);
            V m = lowest;
#pragma unroll
            for (int s = 0; s < P / 4; ++s) {
                V v[4];
                load_quad(smem, d >= 8 ? (a ^ (s << 4)) + (uint32_t)(d * R * 4) : a2 ^ (s << 4), v);
                if constexpr (!std::is_same<V, float>::value) {
                    m = max3(m, box_sub(v[0], c[4 * s]), box_sub(v[1], c[4 * s + 1]));
                    m = max3(m, box_sub(v[2], c[4 * s + 2]), box_sub(v[3], c[4 * s + 3]));
                } else {
                    float d0, d1, d2, d3;
                    asm("{\n\t.reg .b64 x, y, z;\n\t"
                        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tsub.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
                        : "=f"(d0), "=f"(d1)
                        : "f"(v[0]), "f"(v[1]), "f"(c[4 * s]), "f"(c[4 * s + 1]));
                    asm("{\n\t.reg .b64 x, y, z;\n\t"
                        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tsub.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
                        : "=f"(d2), "=f"(d3)
                        : "f"(v[2]), "f"(v[3]), "f"(c[4 * s + 2]), "f"(c[4 * s + 3]));
                    m = max3(m, d0, d1);
                    m = max3(m, d2, d3);
                }
            }
            M[n] = max3(M[n], M[n], box_add(D, m));
        }
    }
}

// The box of width w that starts at bin j (of the extension's index space),
// as width_maxima forms it.
template <class V, int R>
__device__ __forceinline__ V box_at(const unsigned char* smem, const typename Offset<V>::type* offs, int j, int w) {
    const int b = j / R, b2 = (j + w) / R;
    V bx = box_sub(load_bin<V, R>(smem, j + w), load_bin<V, R>(smem, j));
    if (b2 != b) bx = box_add(off_diff(offs[b2], offs[b]), bx);
    return bx;
}

}  // namespace ffa
