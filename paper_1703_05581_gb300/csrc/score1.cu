// Algorithm 1 (Section 2.2.1, Eq. 3-4) on the GPU, one CTA per folded
// profile at a time (persistent over a run of consecutive trials), with the
// last FFA stage (Section 2.1) fused into the load.
//
// The profile lives in shared memory only (score.cuh's swizzled layout, no
// padding, nothing held in registers between steps), so a CTA is as small as
// the profile's length asks for -- one warp for the shortest ones -- and
// several profiles share an SM: one's serial steps (selections, reductions,
// barriers) run under the others' arithmetic.
//
// Median and MAD (exact).  The profile's mean and standard deviation, taken
// while it is loaded, and the offset and ratio that the CTA's previous trial
// showed, predict the median (then the MAD) to within a few sigma / sqrt(N).
// One pass over the profile counts the samples below a window of that width
// and lists those inside it; if the wanted ranks lie in the window, one warp
// finds the order statistics in the list (a few counting passes at
// interpolated pivots), otherwise the window is moved and the pass repeated,
// and after a few attempts an exact radix select over the profile takes over.
// A window's bounds are monotone functions of the value, so the counts are
// exact whatever the prediction was.  Float profiles with gaps or many equal
// values, whose windows hold no sample or too many, go on with pivots that are
// samples themselves.  Int profiles need no list: their window holds one bucket
// per integer.
//
// Box sums.  With the in-block exclusive prefix c_b[o] (blocks of R bins, the
// cyclic extension included) and the block offsets C[b] = sum of earlier
// blocks (float-float, or wrapping int32), the box of width w = R * d at bin
// R b + o is (C[b + d] - C[b]) + (c_{b+d}[o] - c_b[o]); widths below R
// use the block itself and the next one.  Rounding is monotone, so a block's
// largest box is D + max_o (c_{b+d}[o] - c_b[o]): the offset D is added once
// per block and width, not per bin.  Only the maximum of each width is kept;
// the winning width's first argmax is found afterwards by recomputing that
// width in the threads that hold its maximum.  The block that runs past p0
// scores all its bins (its extra boxes are cyclic boxes of the first bins
// again).
//
// What bounds it.  Long profiles: the width pass's shared-memory reads (one
// per bin and width) and the load of two rows; short ones: instructions, about
// 4 per bin and width in all.  A fused launch of 4096 x 19977 takes 0.39 ms at
// 95 thread-instructions a bin (0.82 ms at 195 with the profile in the
// registers of one 1024-thread CTA per SM and a histogram per profile).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "score.cuh"

namespace ffa {

namespace {

template <class V>
struct IsInt {
    static constexpr bool value = std::is_integral<V>::value;
};

// Where a CTA's regions start in dynamic shared memory (bytes); the profile
// is at 0.  `offs` (block offsets) and `list` (window members, `cap` slots
// per thread) share a region: the list is dead before the offsets are formed.
// `aux`: the window's members packed (float), its histogram (int), or the
// radix select's.
struct ScoreLay {
    uint32_t offs, list, aux;
    int32_t cap;
    int32_t group;  // blocks of one group of the offset scan
};

constexpr int score_pack(int r) { return r == 8 ? 256 : 768; }  // members a float window may have
constexpr int score_nb(int r) { return r == 8 ? 256 : 512; }    // buckets of an int window

struct S1Sh {
    unsigned long long key[2];
    float fa[32], fb[32], fc[32];
    uint2 wc[2][32];          // per-warp counts of a window pass (two slots, alternating)
    alignas(16) float2 seg[SCORE_MAXSEG];  // segment totals of the offset scan
    uint32_t wkey[16];        // per-width maxima as order-preserving keys
    uint32_t npack;
    int bin_a, bin_b;
    uint32_t below_a;
    int ok;
    uint32_t pos, tail;  // first argmax: in the whole blocks, in the one that runs past p0
    float best;
    int bw;
};

__device__ __forceinline__ unsigned long long ff_key(float h, float l) {
    return ((unsigned long long)fkey(h) << 32) | fkey(l);
}

// |x - (mh + ml)| as a canonical float-float pair
__device__ __forceinline__ void ff_dev(float x, float mh, float ml, float& h, float& l) {
    two_sum(x, -mh, h, l);
    l = __fsub_rn(l, ml);
    ff_norm(h, l);
    if (h < 0.0f || (h == 0.0f && l < 0.0f)) {
        h = -h;
        l = -l;
    }
}

// 2^(n/2) as the correctly rounded square root of 2^n
__device__ __forceinline__ float sqrt_pow2(int n) {
    return __int_as_float((127 + (n >> 1)) << 23) * ((n & 1) ? 1.41421356237309515f : 1.0f);
}

// Warp 0: the buckets of hist[0, n) (n a multiple of 128) that hold ranks
// ta <= tb (both below the total), and the count before the first one.
template <bool ONE>
__device__ __forceinline__ void hist_find(const uint32_t* hist, int n, uint32_t ta, uint32_t tb, S1Sh& sh) {
    const int lane = threadIdx.x & 31;
    if (ONE || threadIdx.x < 32) {
        const int per = n >> 5, b0 = lane * per;
        uint32_t s = 0;
        for (int t = 0; t < per; t += 4) {
            const uint4 h = *reinterpret_cast<const uint4*>(hist + b0 + t);
            s += (h.x + h.y) + (h.z + h.w);
        }
        uint32_t x = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        uint32_t c = x - s;
        if (tb >= c && ta < x) {
            for (int t = 0; t < per; ++t) {
                const uint32_t h = hist[b0 + t];
                if (ta >= c && ta < c + h) {
                    sh.bin_a = b0 + t;
                    sh.below_a = c;
                }
                if (tb >= c && tb < c + h) sh.bin_b = b0 + t;
                c += h;
            }
        }
    }
    cta_sync<ONE>();
}

// Exact rank-`rank` key over the whole profile by an 8-bit radix select (the
// rare case: no spread, or a window that could not be placed).  Keys: the
// value, or with MAD its deviation from the median (float: from mh + ml;
// int: 2|x - med| with s2 = 2 med).
template <class V, int R, bool ONE, bool MAD>
__device__ __noinline__ unsigned long long radix_rank(const unsigned char* smem, uint32_t* hist, S1Sh& sh, int p0,
                                                      uint32_t rank, float mh, float ml, long long s2) {
    const int T = ONE ? 32 : (int)blockDim.x, tid = threadIdx.x;
    unsigned long long prefix = 0, mask = 0;
    for (int shift = 56; shift >= 0; shift -= 8) {
        cta_sync<ONE>();
        for (int b = tid; b < 256; b += T) hist[b] = 0;
        cta_sync<ONE>();
        for (int j = tid; j < p0; j += T) {
            const V v = load_bin<V, R>(smem, j);
            unsigned long long kk;
            if constexpr (std::is_integral<V>::value) {
                const long long e = 2 * (long long)v - s2;
                kk = MAD ? (unsigned long long)(e < 0 ? -e : e) : (unsigned long long)ikey((int32_t)v);
            } else {
                float h = (float)v, l = 0.0f;
                if (MAD) ff_dev((float)v, mh, ml, h, l);
                kk = ff_key(h, l);
            }
            if ((kk & mask) == prefix) atomicAdd(&hist[(kk >> shift) & 0xff], 1u);
        }
        cta_sync<ONE>();
        hist_find<ONE>(hist, 256, rank, rank, sh);
        rank -= sh.below_a;
        prefix |= (unsigned long long)sh.bin_a << shift;
        mask |= 0xffull << shift;
    }
    cta_sync<ONE>();
    return prefix;
}

__device__ __forceinline__ unsigned long long warp_extreme(unsigned long long k, bool largest) {
    uint32_t h = (uint32_t)(k >> 32), l = (uint32_t)k;
    const uint32_t top = largest ? __reduce_max_sync(0xffffffffu, h) : __reduce_min_sync(0xffffffffu, h);
    if (h != top) l = largest ? 0u : ~0u;
    l = largest ? __reduce_max_sync(0xffffffffu, l) : __reduce_min_sync(0xffffffffu, l);
    return ((unsigned long long)top << 32) | l;
}

// The keys of the two middle ranks of a whole float profile (MAD: of its
// deviations from mh + ml), for profiles with few distinct values or gaps,
// where a window holds no sample or too many.  A pass counts the samples below
// and up to a pivot and finds its neighbours on both sides; the next pivot is
// the neighbour on the wanted side, then a value interpolated inside the
// bounds -- two or three passes settle a profile of few levels, which a radix
// select takes eight or sixteen for (3000 profiles of 1100 bins and 16 levels:
// 49 us, 144 with windows and a radix select only; 150 of 64 bins and 2 levels:
// 7.4 and 32).  False if the ranks were not found.
template <int R, bool ONE, bool MAD>
__device__ __forceinline__ bool member_ranks(const unsigned char* smem, S1Sh& sh, int p0, float mh, float ml,
                                             float guess, float sig, unsigned long long& ka,
                                             unsigned long long& kb) {
    const uint32_t r1 = (uint32_t)((p0 - 1) / 2), r2 = (uint32_t)(p0 / 2);
    const int T = ONE ? 32 : (int)blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = T >> 5;
    uint4* part = reinterpret_cast<uint4*>(sh.seg);  // a warp's neighbours
    unsigned long long lo = 0, hi = ~0ull;           // the wanted keys are in [lo, hi]
    uint32_t cl = 0, ch = (uint32_t)p0;              // keys below lo, up to hi
    unsigned long long p = ff_key(guess, 0.0f);
    bool member = false;
    auto found = [&](unsigned long long a, unsigned long long b) {
        ka = a;
        kb = b;
        return true;
    };
    auto value = [](unsigned long long k) { return fkey_inv((uint32_t)(k >> 32)); };
    for (int a = 0; a < 12; ++a) {
        uint32_t lt = 0, le = 0;
        unsigned long long dn = 0, up = ~0ull;
        for (int j = tid; j < p0; j += T) {
            float h = load_bin<float, R>(smem, j), l = 0.0f;
            if (MAD) ff_dev(h, mh, ml, h, l);
            const unsigned long long k = ff_key(h, l);
            lt += k < p;
            le += k <= p;
            if (k < p && k > dn) dn = k;
            if (k > p && k < up) up = k;
        }
        lt = __reduce_add_sync(0xffffffffu, lt);
        le = __reduce_add_sync(0xffffffffu, le);
        dn = warp_extreme(dn, true);
        up = warp_extreme(up, false);
        if (!ONE) {
            if (lane == 0) {
                sh.wc[0][warp] = make_uint2(lt, le);
                part[warp] = make_uint4((uint32_t)(dn >> 32), (uint32_t)dn, (uint32_t)(up >> 32), (uint32_t)up);
            }
            __syncthreads();
            uint2 c = make_uint2(0u, 0u);
            uint4 n = make_uint4(0u, 0u, ~0u, ~0u);
            if (lane < NW) {
                c = sh.wc[0][lane];
                n = part[lane];
            }
            __syncthreads();
            lt = __reduce_add_sync(0xffffffffu, c.x);
            le = __reduce_add_sync(0xffffffffu, c.y);
            dn = warp_extreme(((unsigned long long)n.x << 32) | n.y, true);
            up = warp_extreme(((unsigned long long)n.z << 32) | n.w, false);
        }
        if (r1 < lt) {
            if (r2 >= lt) return found(dn, le > lt ? p : up);
            if (r1 == lt - 1) return found(dn, dn);
            hi = dn;
            ch = lt;
        } else if (r1 < le) {
            return found(p, r2 < le ? p : up);
        } else {
            if (r1 == le && r2 == r1) return found(up, up);
            lo = up;
            cl = le;
        }
        const bool down = r1 < lt;
        if (member) {
            float x;
            if (lo != 0 && hi != ~0ull)
                x = fmaf((float)(2 * (r1 - cl) + 1) / (float)(2 * (ch - cl)), value(hi) - value(lo), value(lo));
            else {
                // about the ranks' distance near a normal median
                const float step = sig / (0.3f * (float)p0);
                x = down ? value(dn) - step * (float)(lt - r1) : value(up) + step * (float)(r1 + 1 - le);
            }
            p = ff_key(x, 0.0f);
            member = !(p > lo && p < hi);
            if (member) p = down ? dn : up;
        } else {
            p = down ? dn : up;
            member = true;
        }
    }
    return false;
}

// The median's and the MAD's float pairs from their two middle ranks' keys
// (the median (a + b) / 2 exactly).
__device__ __forceinline__ void pair_median(unsigned long long ka, unsigned long long kb, bool two, float& h, float& l) {
    const float a = fkey_inv((uint32_t)(ka >> 32)), b = fkey_inv((uint32_t)(kb >> 32));
    h = a;
    l = 0.0f;
    if (two) {
        two_sum(a, b, h, l);
        h *= 0.5f;
        l *= 0.5f;
    }
}
__device__ __forceinline__ void pair_mad(unsigned long long ka, unsigned long long kb, bool two, float& h, float& l) {
    h = fkey_inv((uint32_t)(ka >> 32));
    l = fkey_inv((uint32_t)ka);
    if (two) {
        ff_acc(h, l, fkey_inv((uint32_t)(kb >> 32)), fkey_inv((uint32_t)kb));
        ff_norm(h, l);
        h *= 0.5f;
        l *= 0.5f;
    }
}

// Median and MAD of any float profile, as the pairs sh.fa[0..1] and
// sh.fa[2..3]: by pivots if the profile has a spread (sig; 0: none, or not
// finite), else, and where they fail, by a radix select.  One call for all of
// it: the scorer keeps its registers.
template <int R, bool ONE>
__device__ __noinline__ void profile_ranks(unsigned char* smem, uint32_t* hist, S1Sh& sh, int p0, float mean,
                                           float sig) {
    const uint32_t r1 = (uint32_t)((p0 - 1) / 2), r2 = (uint32_t)(p0 / 2);
    float mh = 0.0f, ml = 0.0f, kh, kl;
    unsigned long long ka, kb;
    if (!(sig > 0.0f)) {
        // Squares that are all 0: float pairs lose their low part near the
        // smallest numbers (as FP64 does not), so the profile is scored 2^64
        // times as large, which leaves its S/N as it is.
        const int T = ONE ? 32 : (int)blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        float top = 0.0f;
        for (int j = threadIdx.x; j < p0; j += T) top = fmaxf(top, fabsf(load_bin<float, R>(smem, j)));
        top = warp_max(top);
        if (!ONE) {
            if (lane == 0) sh.fa[warp] = top;
            __syncthreads();
            top = warp_max(lane < (T >> 5) ? sh.fa[lane] : 0.0f);
            __syncthreads();
        }
        if (top < 1e-12f) {
            for (int j = threadIdx.x; j < p0; j += T) {
                float* x = reinterpret_cast<float*>(smem + bin_addr<R>(j));
                *x *= 18446744073709551616.0f;
            }
            cta_sync<ONE>();
        }
    }
    if (!(sig > 0.0f && member_ranks<R, ONE, false>(smem, sh, p0, mh, ml, mean, sig, ka, kb))) {
        ka = radix_rank<float, R, ONE, false>(smem, hist, sh, p0, r1, mh, ml, 0);
        kb = r1 == r2 ? ka : radix_rank<float, R, ONE, false>(smem, hist, sh, p0, r2, mh, ml, 0);
    }
    pair_median(ka, kb, r1 != r2, mh, ml);
    if (!(sig > 0.0f && member_ranks<R, ONE, true>(smem, sh, p0, mh, ml, 0.6745f * sig, sig, ka, kb))) {
        ka = radix_rank<float, R, ONE, true>(smem, hist, sh, p0, r1, mh, ml, 0);
        kb = r1 == r2 ? ka : radix_rank<float, R, ONE, true>(smem, hist, sh, p0, r2, mh, ml, 0);
    }
    pair_mad(ka, kb, r1 != r2, kh, kl);
    if (threadIdx.x == 0) {
        sh.fa[0] = mh;
        sh.fa[1] = ml;
        sh.fa[2] = kh;
        sh.fa[3] = kl;
    }
    cta_sync<ONE>();
}

// One warp: the values of ranks t1 <= t2 <= t1 + 1 among the n <= 128 KQ
// members v of a window (in registers, member 128 k + 4 lane + e in v[4 k + e],
// +inf beyond n), all between lo and hi.  MAD: of |x - mh|.  Counting passes
// at interpolated pivots; each pass also yields the pivot's neighbours on both
// sides, and the interval closes in on members, so that clusters of nearly
// equal values (folds of quantised series) cost no more passes.
template <bool MAD, int KQ>
__device__ __forceinline__ bool pick2(const float (&v)[4 * KQ], uint32_t n, uint32_t t1, uint32_t t2, float lo, float hi,
                                      float mh, float& va, float& vb) {
    uint32_t cl = 0, ch = n;  // members < lo, <= hi
    bool step = false;        // next pivot: the first member from lo on
    for (int a = 0; a < 32; ++a) {
        float p = lo;
        if (!step) {
            p = fmaf(__fdividef((float)(2 * (t1 - cl) + 1), (float)(2 * (ch - cl))), hi - lo, lo);
            if (!(p < hi)) p = lo;
        }
        uint32_t c = 0;
        float ab[4], up[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            ab[e] = INFINITY;
            up[e] = -INFINITY;
        }
#pragma unroll
        for (int k = 0; k < KQ; ++k) {
            if (128u * k >= n) break;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d = MAD ? fabsf(__fsub_rn(v[4 * k + e], mh)) : v[4 * k + e];
                const bool in = d <= p;
                c += in;
                up[e] = fmaxf(up[e], in ? d : -INFINITY);
                ab[e] = fminf(ab[e], in ? INFINITY : d);
            }
        }
        c = __reduce_add_sync(0xffffffffu, c);
        const float above = -warp_max(-fminf(fminf(ab[0], ab[1]), fminf(ab[2], ab[3])));
        const float upto = warp_max(fmaxf(max3(up[0], up[1], up[2]), up[3]));
        if (c <= t1) {
            if (c == t1 && t2 == t1) {
                va = vb = above;
                return true;
            }
            lo = above;
            cl = c;
            step = t1 - c <= 1;
        } else {
            // fewer than t1 + 1 members are below lo
            if (p == lo || c == t1 + 1) {
                va = upto;
                vb = c > t2 ? upto : above;
                return true;
            }
            hi = upto;
            ch = c;
            step = false;
        }
    }
    return false;
}

// One warp: the exact deviations |x - (mh + ml)| of ranks t1 <= t2 among the
// m values at `pack` (near-ties of the FP32 deviation), as keys.  Up to 32 by
// comparison in registers, more by a quickselect.
__device__ __forceinline__ void rank_deviations(const float* pack, uint32_t m, uint32_t t1, uint32_t t2, float mh,
                                                float ml, unsigned long long& ka, unsigned long long& kb) {
    const int lane = threadIdx.x & 31;
    auto key_of = [&](float x) {
        float h, l;
        ff_dev(x, mh, ml, h, l);
        return ff_key(h, l);
    };
    if (m <= 32) {
        const unsigned long long ki = lane < m ? key_of(pack[lane]) : ~0ull;
        uint32_t rk = 0;
        for (uint32_t j = 0; j < m; ++j) {
            const unsigned long long kj = __shfl_sync(0xffffffffu, ki, j);
            rk += (kj < ki) || (kj == ki && j < (uint32_t)lane);
        }
        ka = __shfl_sync(0xffffffffu, ki, __ffs(__ballot_sync(0xffffffffu, lane < m && rk == t1)) - 1);
        kb = __shfl_sync(0xffffffffu, ki, __ffs(__ballot_sync(0xffffffffu, lane < m && rk == t2)) - 1);
        return;
    }
    for (int want = 0; want < 2; ++want) {
        const uint32_t t = want ? t2 : t1;
        unsigned long long klo = 0, khi = ~0ull, kp = 0;  // the wanted key is in [klo, khi]
        uint32_t at = 0;
        for (uint32_t a = 0; a <= m; ++a) {
            // the next member in the interval is the pivot
            for (uint32_t scan = 0; scan <= m; scan += 32) {
                const uint32_t i = at + lane < m ? at + lane : at + lane - m;
                const unsigned long long k = i < m ? key_of(pack[i]) : 0ull;
                const unsigned in = __ballot_sync(0xffffffffu, i < m && k >= klo && k <= khi);
                if (in) {
                    const int src = __ffs(in) - 1;
                    kp = __shfl_sync(0xffffffffu, k, src);
                    at = (at + src + 1) % m;
                    break;
                }
                at = (at + 32) % m;
            }
            uint32_t less = 0, upto = 0;
            for (uint32_t i = lane; i < m; i += 32) {
                const unsigned long long k = key_of(pack[i]);
                less += k < kp;
                upto += k <= kp;
            }
            less = __reduce_add_sync(0xffffffffu, less);
            upto = __reduce_add_sync(0xffffffffu, upto);
            if (t < less) khi = kp - 1;
            else if (t >= upto) klo = kp + 1;
            else break;
        }
        (want ? kb : ka) = kp;
        if (t1 == t2) {
            kb = kp;
            break;
        }
    }
}

// R: bins per block.  ONE: the CTA is one warp.
template <class V, int R, bool ONE, bool FUSED, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    k_score1(const V* __restrict__ prof_all, const ScoreGroup sg, int64_t m_rows, int64_t trial0, int64_t count,
             uint32_t wmask, int wtop, const ScoreLay lay, int32_t* d_status) {
    constexpr bool INT = IsInt<V>::value;
    constexpr int P = R < 16 ? R : 16;  // bins per item of the width pass
    constexpr int PARTS = R / P;
    constexpr int NS = R == 8 ? 12 : 16;  // widths 2^0 .. 2^(NS-1)
    constexpr int NB = score_nb(R);
    constexpr int NP = score_pack(R);
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ S1Sh sh;
    const int T = ONE ? 32 : (int)blockDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = ONE ? 0 : tid >> 5;
    const int NW = T >> 5;
    using Off = typename Offset<V>::type;
    Off* offs = reinterpret_cast<Off*>(smem + lay.offs);
    uint32_t* hist = reinterpret_cast<uint32_t*>(smem + lay.aux);
    float* pack = reinterpret_cast<float*>(smem + lay.aux);
    auto sync = [&]() { cta_sync<ONE>(); };
    // block sums of two counts per thread (one barrier); slot alternates
    auto sum2 = [&](uint32_t a, uint32_t b, int slot) -> uint2 {
        a = __reduce_add_sync(0xffffffffu, a);
        b = __reduce_add_sync(0xffffffffu, b);
        if (ONE) {
            __syncwarp();
            return make_uint2(a, b);
        }
        if (lane == 0) sh.wc[slot][warp] = make_uint2(a, b);
        __syncthreads();
        if (NW <= 4) {  // few warps: read them all
            uint2 t = sh.wc[slot][0];
            for (int i = 1; i < NW; ++i) {
                const uint2 v = sh.wc[slot][i];
                t.x += v.x;
                t.y += v.y;
            }
            return t;
        }
        const uint2 v = lane < NW ? sh.wc[slot][lane] : make_uint2(0u, 0u);
        return make_uint2(__reduce_add_sync(0xffffffffu, v.x), __reduce_add_sync(0xffffffffu, v.y));
    };
    // this CTA's run of consecutive trials
    const int64_t it_end = count * (int64_t)(blockIdx.x + 1) / gridDim.x;
    int64_t it = count * (int64_t)blockIdx.x / gridDim.x;
    float hint_med = 0.0f, hint_mad = 0.6745f;  // (median - mean) / sigma, MAD / sigma of the trials before
    int ei = it < it_end ? score_entry(sg, it) : 0;
    for (; it < it_end; ++it) {
        if (it >= sg.t0[ei + 1]) ++ei;
        const int p0 = sg.p0[ei];
        const int64_t ld = sg.ld[ei];
        const V* __restrict__ prof = prof_all + sg.off[ei];
        const int64_t k = trial0 + (it - sg.t0[ei]);
        const int nblk = (p0 + R - 1) / R;
        const int next = (1 << wtop) > R ? (1 << wtop) / R : 1;  // extension blocks
        const int nbx = nblk + next;

        // The in-block prefixes, in place (exclusive within each block) with
        // the block totals in `offs`: threads first, first + step, ...
        auto prefix = [&](int first, int step) {
            for (int b = first; b < nbx; b += step) {
                const uint32_t a = blk_addr<R>((uint32_t)b);
                V t = 0;
#pragma unroll
                for (int s = 0; s < R / 4; ++s) {
                    V v[4], c[4];
                    load_quad(smem, a ^ (s << 4), v);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        c[i] = t;
                        t = t + v[i];
                    }
                    *reinterpret_cast<int4*>(smem + (a ^ (s << 4))) = *reinterpret_cast<const int4*>(c);
                }
                if constexpr (INT) offs[b] = t;
                else offs[b].x = t;
            }
        };
        bool prefixed = false;
        float mh = 0.0f, ml = 0.0f;    // float: median = mh + ml
        float kmh = 0.0f, kml = 0.0f;  // float: MAD = kmh + kml
        long long s2 = 0, e2 = 0;      // int: 2 * median; 4 * MAD
        // A second round only if the MAD's pick failed after the prefixes had
        // replaced the profile (`redo`: the profile again, no windows).
        for (bool redo = false;; redo = true) {
        // ---- load; fused last FFA stage: head row k>>1 plus tail row M/2 +
        // (k>>1) read ceil(k/2) bins further on, four bins at a time.  The
        // sum, sum of squares and (int) largest |x| accumulate meanwhile.
        float fs = 0.0f, fq = 0.0f, fm = 0.0f;
        auto acc = [&](V v) {
            const float f = (float)v;
            fs += f;
            fq = fmaf(f, f, fq);
            if (INT) fm = fmaxf(fm, fabsf(f));
        };
        const bool two = FUSED && m_rows > 1;
        const V* __restrict__ hrow = prof + (FUSED ? (k >> 1) * ld : k * ld);
        const V* __restrict__ trow = prof + ((m_rows >> 1) + (k >> 1)) * ld;  // two only
        const int sft = two ? (int)((uint32_t)((k + 1) >> 1) % (uint32_t)p0) : 0;
        // pull the next rows towards L2 while this profile is scored (an even
        // trial's partner reads the same two rows)
        if (it + 1 < it_end && (FUSED ? (k & 1) && k + 1 < m_rows : true)) {
            const int lines = (int)((p0 * (int64_t)sizeof(V) + 127) / 128);
            for (int l = tid; l < lines; l += T) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(hrow + ld + l * (128 / sizeof(V))));
                if (FUSED) asm volatile("prefetch.global.L2 [%0];" ::"l"(trow + ld + l * (128 / sizeof(V))));
            }
        }
        load_profile<V, R>(smem, hrow, trow, sft, two, p0, tid, T, acc);
        if (INT)
            for (int b = 4 * tid; b < NB; b += 4 * T) *reinterpret_cast<int4*>(hist + b) = make_int4(0, 0, 0, 0);
        if (tid < 16) sh.wkey[tid] = 0u;
        if (tid == 16) sh.pos = sh.tail = 0x7fffffffu;
        if (tid == 17) sh.npack = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fs += __shfl_xor_sync(0xffffffffu, fs, o);
            fq += __shfl_xor_sync(0xffffffffu, fq, o);
        }
        if (INT) fm = warp_max(fm);
        if (!ONE) {
            if (lane == 0) {
                sh.fa[warp] = fs;
                sh.fb[warp] = fq;
                if (INT) sh.fc[warp] = fm;
            }
            __syncthreads();
            if (NW <= 4) {
                fs = sh.fa[0];
                fq = sh.fb[0];
                if (INT) fm = sh.fc[0];
                for (int i = 1; i < NW; ++i) {
                    fs += sh.fa[i];
                    fq += sh.fb[i];
                    if (INT) fm = fmaxf(fm, sh.fc[i]);
                }
            } else {
                fs = lane < NW ? sh.fa[lane] : 0.0f;
                fq = lane < NW ? sh.fb[lane] : 0.0f;
                if (INT) fm = warp_max(lane < NW ? sh.fc[lane] : 0.0f);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    fs += __shfl_xor_sync(0xffffffffu, fs, o);
                    fq += __shfl_xor_sync(0xffffffffu, fq, o);
                }
            }
        } else {
            __syncwarp();
        }
        const float rn = 1.0f / (float)p0;
        const float mean = fs * rn;
        const float sig = sqrtf(fmaxf(fmaf(fq, rn, -mean * mean), 0.0f));
        const float rsn = sqrtf(rn) * sig;  // sigma / sqrt(N)
        // cyclic extension: bins past p0 repeat the profile
        bool extended = false;
        auto extend = [&](int first, int step) { extend_profile<V, R>(smem, p0, nbx, first, step); };

        // ---- median and MAD (Eq. 3), exact ----
        const uint32_t r1 = (uint32_t)((p0 - 1) / 2), r2 = (uint32_t)(p0 / 2);
        // quads entirely inside groups of 32 bins need no bound check
        const int nq = (p0 >> 5) << 3, jt = (p0 & ~31) + tid;
        bool spread = sig > 0.0f && sig < 1e30f;  // a prediction makes sense (block-uniform)
        if (INT) spread = spread && fm < 5e8f;    // 2 |x| and window sums stay in int32
        if constexpr (!INT) {
            mh = ml = 0.0f;
            // One window [g - r, g + r] after another.  MAD: on |x - mh|.
            auto select = [&](auto mad_tag, float g, float r, unsigned long long& ka, unsigned long long& kb) -> bool {
                constexpr bool MAD = decltype(mad_tag)::value;
                const uint32_t lbase = (uint32_t)__cvta_generic_to_shared(smem) + lay.list + (uint32_t)(tid * lay.cap) * 4u;
                const uint32_t lim = lbase + (uint32_t)(lay.cap - 1) * 4u;
                const float* mine = reinterpret_cast<const float*>(smem + lay.list) + tid * lay.cap;
                for (int a = 0; a < 5; ++a) {
                    const float lo = g - r, hi = g + r;
                    uint32_t ptr = lbase, below = 0;
                    auto take = [&](float v) {
                        const float d = MAD ? fabsf(__fsub_rn(v, mh)) : v;
                        asm volatile(
                            "{\n\t.reg .pred p, q;\n\t"
                            "setp.lt.f32 p, %2, %3;\n\t"
                            "setp.le.and.f32 q, %2, %4, !p;\n\t"
                            "@p add.u32 %1, %1, 1;\n\t"
                            "@q st.shared.f32 [%0], %5;\n\t"
                            "@q add.u32 %0, %0, 4;\n\t"
                            "@q min.u32 %0, %0, %6;\n\t}"
                            : "+r"(ptr), "+r"(below)
                            : "f"(d), "f"(lo), "f"(hi), "f"(v), "r"(lim)
                            : "memory");
                    };
                    for (int q = tid; q < nq; q += T) {
                        V v[4];
                        load_quad(smem, (uint32_t)q << 4, v);
#pragma unroll
                        for (int i = 0; i < 4; ++i) take(v[i]);
                    }
                    for (int j = jt; j < p0; j += T) take(load_bin<V, R>(smem, j));
                    // pack the threads' lists
                    const uint32_t nl = (ptr - lbase) >> 2;
                    if (nl) {
                        const uint32_t at = atomicAdd(&sh.npack, nl);
                        if (at + nl <= NP)
                            for (uint32_t i = 0; i < nl; ++i) pack[at + i] = mine[i];
                    }
                    const uint2 c = sum2(below + (ptr == lim ? 1u << 17 : 0u), nl, a & 1);
                    const uint32_t cl = c.x & 0x1ffffu;
                    if (c.x >> 17 || c.y > NP) {  // a thread's list, or the packed one, overflowed
                        if (tid == 0) sh.npack = 0;
                        r *= 0.5f;
                        sync();
                        // (one thread's list overflows in every few normal
                        // profiles; lists half full: equal values, once more)
                        if (2 * c.y > (uint32_t)(T * (lay.cap - 1))) a += 2;
                        continue;
                    }
                    if (c.y == 0) {  // a gap
                        sync();
                        return false;
                    }
                    if (r1 < cl || r2 >= cl + c.y) {
                        const float dens = (float)c.y / (2.0f * r);
                        if (r1 < cl) g -= r + (float)(cl - r1) / dens;
                        else g += r + (float)(r2 + 1 - cl - c.y) / dens;
                        r *= 1.5f;
                        if (tid == 0) sh.npack = 0;
                        sync();
                        continue;
                    }
                    if (warp == 0) {
                        // pick, then settle near-ties exactly
                        const uint32_t n = c.y, t1 = r1 - cl, t2 = r2 - cl;
                        constexpr int KQ = NP / 128;
                        float v[4 * KQ];
#pragma unroll
                        for (int k = 0; k < KQ; ++k) {
                            const uint32_t i = 128 * k + 4 * lane;
                            float4 q = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                            if (i < n) q = *reinterpret_cast<const float4*>(pack + i);
                            v[4 * k] = q.x;
                            v[4 * k + 1] = i + 1 < n ? q.y : INFINITY;
                            v[4 * k + 2] = i + 2 < n ? q.z : INFINITY;
                            v[4 * k + 3] = i + 3 < n ? q.w : INFINITY;
                        }
                        __syncwarp();
                        float va, vb;
                        int ok = pick2<MAD, KQ>(v, n, t1, t2, lo, hi, mh, va, vb);
                        if constexpr (!MAD) {
                            if (lane == 0) {
                                sh.key[0] = ff_key(va, 0.0f);
                                sh.key[1] = ff_key(vb, 0.0f);
                            }
                        } else if (ok) {
                            // |x - mh| in FP32 is within E of the exact
                            // deviation: the wanted ranks are among the members
                            // within 2 E of va, vb; rank those exactly
                            const float E = (hi + fabsf(mh)) * 1.2e-7f;
                            const float ca = va - 3.0f * E, cb = vb + 3.0f * E;
                            uint32_t less = 0, m = 0;
#pragma unroll
                            for (int i = 0; i < 4 * KQ; ++i) {
                                if (32u * (i & ~3) >= n) break;
                                const float d = fabsf(__fsub_rn(v[i], mh));
                                less += d < ca;
                                const bool is = d >= ca && d <= cb;
                                const unsigned near = __ballot_sync(0xffffffffu, is);
                                if (near) {
                                    if (is) pack[m + __popc(near & ((1u << lane) - 1))] = v[i];
                                    m += __popc(near);
                                }
                            }
                            __syncwarp();
                            less = __reduce_add_sync(0xffffffffu, less);
                            if (ca < lo || cb > hi) {  // too near the window's edge
                                ok = 0;
                            } else {
                                unsigned long long k1, k2;
                                rank_deviations(pack, m, t1 - less, t2 - less, mh, ml, k1, k2);
                                if (lane == 0) {
                                    sh.key[0] = k1;
                                    sh.key[1] = k2;
                                }
                            }
                        }
                        if (lane == 0) {
                            sh.ok = ok;
                            sh.npack = 0;
                        }
                    } else if (!ONE) {  // meanwhile
                        if (MAD) prefix(tid - 32, T - 32);
                        else extend(tid - 32, T - 32);
                    }
                    if (!ONE) (MAD ? prefixed : extended) = true;
                    sync();
                    ka = sh.key[0];
                    kb = sh.key[1];
                    return sh.ok != 0;
                }
                return false;
            };
            unsigned long long ka = 0, kb = 0;
            bool done = false;
            if (spread && !redo && select(std::false_type{}, fmaf(hint_med, sig, mean), 3.2f * rsn, ka, kb)) {
                pair_median(ka, kb, r1 != r2, mh, ml);
                if (!extended) {  // read after the barriers of the MAD's selection
                    extend(tid, T);
                    extended = true;
                }
                done = select(std::true_type{}, hint_mad * sig, 2.6f * rsn, ka, kb);
                if (!done && prefixed) {  // the profile is gone: once more
                    prefixed = false;
                    sync();
                    continue;
                }
                pair_mad(ka, kb, r1 != r2, kmh, kml);
            }
            if (!done) {
                profile_ranks<R, ONE>(smem, hist, sh, p0, mean, spread ? sig : 0.0f);
                mh = sh.fa[0];
                ml = sh.fa[1];
                kmh = sh.fa[2];
                kml = sh.fa[3];
                if (!extended) extend(tid, T);
            }
            if (spread) {
                const float is = 1.0f / sig;
                hint_med += 0.3f * ((mh - mean) * is - hint_med);
                hint_mad += 0.3f * (kmh * is - hint_mad);
            }
        } else {
            extend(tid, T);  // read after the barriers of the selections
            extended = true;
            // Int profiles: a window of at most NB consecutive integers (of
            // the value, or of the deviation 2|x - med| in steps of two), one
            // bucket each, so that the bucket is the value.
            auto select = [&](auto mad_tag, int lo, int width, long long& va, long long& vb) -> bool {
                constexpr bool MAD = decltype(mad_tag)::value;
                const int m2 = (int)s2;
                for (int a = 0; a < 5; ++a) {
                    if (MAD || a > 0) {
                        for (int b = 4 * tid; b < NB; b += 4 * T)
                            *reinterpret_cast<int4*>(hist + b) = make_int4(0, 0, 0, 0);
                        sync();
                    }
                    uint32_t below = 0, in = 0;
                    auto take = [&](int v) {
                        const int e = MAD ? abs(2 * v - m2) : v;
                        const uint32_t t = (uint32_t)(e - lo) >> (MAD ? 1 : 0);
                        if (e < lo) ++below;
                        else if (t < (uint32_t)width) {
                            atomicAdd(&hist[t], 1u);
                            ++in;
                        }
                    };
                    for (int q = tid; q < nq; q += T) {
                        V v[4];
                        load_quad(smem, (uint32_t)q << 4, v);
#pragma unroll
                        for (int i = 0; i < 4; ++i) take((int)v[i]);
                    }
                    for (int j = jt; j < p0; j += T) take((int)load_bin<V, R>(smem, j));
                    const uint2 c = sum2(below, in, a & 1);
                    if (r1 < c.x || r2 >= c.x + c.y) {
                        const int step = MAD ? 2 : 1;
                        const float dens = fmaxf((float)c.y, 1.0f) / (float)width;
                        const float miss = r1 < c.x ? (float)(c.x - r1) : (float)(r2 + 1 - c.x - c.y);
                        const int move = step * (int)fminf((float)(width / 2) + miss / dens, 1e8f);
                        lo += r1 < c.x ? -move : move;
                        width = width + width / 2 < NB ? width + width / 2 : NB;
                        if (lo < -1000000000 || lo > 1000000000) return false;
                        sync();  // hist complete before it is cleared
                        continue;
                    }
                    hist_find<ONE>(hist, NB, r1 - c.x, r2 - c.x, sh);
                    va = lo + (MAD ? 2 : 1) * sh.bin_a;
                    vb = lo + (MAD ? 2 : 1) * sh.bin_b;
                    return true;
                }
                return false;
            };
            long long va = 0, vb = 0;
            bool done = false;
            if (spread) {
                const int r = 1 + (int)fminf(3.2f * rsn, (float)(NB / 2 - 2));
                done = select(std::false_type{}, __float2int_rn(fmaf(hint_med, sig, mean)) - r, 2 * r + 1, va, vb);
            }
            if (!done) {
                auto rank = [&](uint32_t r) -> long long {
                    return (int32_t)((uint32_t)radix_rank<V, R, ONE, false>(smem, hist, sh, p0, r, 0.0f, 0.0f, 0) ^ 0x80000000u);
                };
                va = rank(r1);
                vb = r1 == r2 ? va : rank(r2);
            }
            s2 = va + vb;
            sync();  // hist and bin_a read by all
            done = false;
            long long ea = 0, eb = 0;
            if (spread) {
                const int r = 1 + (int)fminf(2.6f * rsn, (float)(NB / 2 - 2));
                int lo = 2 * (__float2int_rn(hint_mad * sig) - r);
                if (lo < 0) lo = 0;
                lo += (int)(s2 & 1);  // deviations 2|x - med| have s2's parity
                done = select(std::true_type{}, lo, 2 * r + 1, ea, eb);
            }
            if (!done) {
                ea = (long long)radix_rank<V, R, ONE, true>(smem, hist, sh, p0, r1, 0.0f, 0.0f, s2);
                eb = r1 == r2 ? ea : (long long)radix_rank<V, R, ONE, true>(smem, hist, sh, p0, r2, 0.0f, 0.0f, s2);
            }
            e2 = ea + eb;
            if (spread) {
                const float is = 1.0f / sig;
                hint_med += 0.3f * ((0.5f * (float)s2 - mean) * is - hint_med);
                hint_mad += 0.3f * (0.25f * (float)e2 * is - hint_mad);
            }
        }
        break;
        }
        if (!prefixed) sync();  // the window list gives way to the offsets

        if (!prefixed) {
            prefix(tid, T);
            sync();
        }
        scan_offsets<V, ONE>(offs, sh.seg, nbx, lay.group);

        // ---- widths: the largest box of each, per thread ----
        V M[NS];
        const int nitem = nblk * PARTS;
        width_maxima<V, R, NS>(smem, offs, wmask, tid, T, nitem, M);
        // lane n of each warp: the warp's maximum of width 2^n; then the CTA's
        uint32_t wk = 0;
#pragma unroll
        for (int n = 0; n < NS; ++n) {
            const V m = warp_max(M[n]);  // (widths not asked for: the lowest value)
            wk = lane == n ? (uint32_t)as_bits(m) : wk;
        }
        if constexpr (INT) wk = ikey((int32_t)wk);
        else wk = fkey(__uint_as_float(wk));
        if (!ONE) {
            if (lane < 16 && (wmask >> lane & 1u)) atomicMax(&sh.wkey[lane], wk);
            __syncthreads();
        }
        // ---- S/N_w = (B_w - w*med) / (K*MAD*sqrt(w)) for w = 2^n in lane n of
        // warp 0; the best, ties to the smaller width.  sqrt(w) is 2^(n/2), or
        // 2^((n-1)/2) times the rounded sqrt(2).
        bool madpos;
        if constexpr (INT) madpos = e2 > 0;
        else madpos = kmh > 0.0f || kml > 0.0f;
        if (warp == 0) {
            if (!ONE) wk = lane < 16 ? sh.wkey[lane] : 0u;
            const bool on = lane < 16 && (wmask >> (lane & 15) & 1u);
            const int n = lane & 15;
            float key = -INFINITY;
            if constexpr (INT) {
                // 2 * (B - w * med) is an exact integer
                const long long num2 = 2 * (long long)(int32_t)(wk ^ 0x80000000u) - ((long long)s2 << n);
                // 1/sqrt(w): 2^(-n/2) for even n, else 2^(-(n-1)/2)/sqrt(2)
                const float rs = __int_as_float((127 - (n >> 1)) << 23) * ((n & 1) ? 0.70710678f : 1.0f);
                if (on) key = 0.5f * __ll2float_rn(num2) * rs;
            } else {
                // numerator in float-float (w * mh, w * ml exact: w is a power
                // of two), K * MAD in float-float rounded once, one division
                constexpr float KH = (float)KMAD, KL = (float)(KMAD - (double)KH);
                const float ph = __fmul_rn(kmh, KH);
                const float pl = __fadd_rn(__fmaf_rn(kmh, KH, -ph), __fmaf_rn(kmh, KL, __fmul_rn(kml, KH)));
                const float kf = __fadd_rn(ph, pl);
                const float w = (float)(1 << n);
                float hi, lo;
                two_sum(fkey_inv(wk), -(w * mh), hi, lo);
                const float num = __fadd_rn(hi, __fsub_rn(lo, w * ml));
                if (on) key = __fdiv_rn(num, __fmul_rn(kf, sqrt_pow2(n)));
            }
            int bw = on ? n : 31;
            float bk = key;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ok = __shfl_xor_sync(0xffffffffu, bk, o);
                const int ob = __shfl_xor_sync(0xffffffffu, bw, o);
                if (ok > bk || (ok == bk && ob < bw)) {
                    bk = ok;
                    bw = ob;
                }
            }
            if (bw > 15) bw = __ffs(wmask) - 1;  // every score NaN
            if constexpr (INT) {
                if (lane == bw) {
                    const double num = __dmul_rn(
                        0.5, (double)(2 * (long long)(int32_t)(wk ^ 0x80000000u) - ((long long)s2 << n)));
                    const double kmad = __dmul_rn(KMAD, (double)e2 * 0.25);
                    constexpr double SQRT2 = 1.4142135623730951;  // sqrt(2) rounded to nearest
                    const double sq = __dmul_rn((double)(1 << (n >> 1)), (n & 1) ? SQRT2 : 1.0);
                    sh.best = __double2float_rn(__ddiv_rn(num, __dmul_rn(kmad, sq)));
                }
            } else if (lane == bw) {
                sh.best = bk;
            }
            if (lane == 0) sh.bw = bw;
            if (ONE && lane == bw) sh.wkey[bw] = wk;
        }
        sync();
        // ---- first argmax of the winning width, recomputed bit-identically
        // in the threads whose own maximum is the CTA's: a warp takes such a
        // thread's items together, one bin per lane
        const int bw = sh.bw;
        if (madpos) {
            V target;
            if constexpr (INT) target = (V)(int32_t)(sh.wkey[bw] ^ 0x80000000u);
            else target = (V)fkey_inv(sh.wkey[bw]);
            V own = box_lowest((V)0);
#pragma unroll
            for (int n = 0; n < NS; ++n)
                if (n == bw) own = M[n];
            const int w = 1 << bw;
            unsigned who = __ballot_sync(0xffffffffu, own == target && tid < nitem);
            while (who) {
                const int src = warp * 32 + __ffs(who) - 1;
                who &= who - 1;
                const int nk = (nitem - src + T - 1) / T;
                for (int i0 = 0; i0 < nk; i0 += 32 / P) {
                    const int im = src + (i0 + lane / P) * T;
                    uint32_t f = 0x7fffffffu;
                    bool tail = false;
                    if (im < nitem) {
                        const int j = (im / PARTS) * R + (im % PARTS) * P + lane % P;
                        tail = (im / PARTS + 1) * R > p0;
                        if (box_at<V, R>(smem, offs, j, w) == target) f = (uint32_t)j;
                    }
                    const uint32_t f1 = __reduce_min_sync(0xffffffffu, tail ? 0x7fffffffu : f);
                    const uint32_t f2 = __reduce_min_sync(0xffffffffu, tail ? f : 0x7fffffffu);
                    if (lane == 0 && f1 != 0x7fffffffu) atomicMin(&sh.pos, f1);
                    if (lane == 0 && f2 != 0x7fffffffu) atomicMin(&sh.tail, f2);
                }
            }
        }
        sync();
        if (tid == 0) {
            ffa_record out;
            if (!madpos) {
                out.snr = 0.0f;
                out.width = wmask & (0u - wmask);
                out.phase = 0;
                out.flags = 1;
            } else {
                // the last block's first match counts at its cyclic position
                uint32_t pos = sh.tail;
                if (pos != 0x7fffffffu && pos >= (uint32_t)p0) pos %= (uint32_t)p0;
                pos = min(pos, sh.pos);
                out.snr = sh.best;
                out.width = 1 << bw;
                out.phase = pos == 0x7fffffffu ? 0 : (int32_t)pos;
                out.flags = 0;
                if (pos == 0x7fffffffu) dev_fail(d_status, FFA_ERR_DEVICE);
            }
            sg.rec[ei][it - sg.t0[ei]] = out;
        }
        sync();
    }
}


// ---- launches -----------------------------------------------------------------

// The CTA for profiles of up to p0 bins in blocks of R: threads, shared
// memory.  The width pass deals out items of min(R, 16) bins, so the thread
// count divides them into whole rounds.
template <class V, int R>
void score1_shape(int64_t p0, int wtop, int rounds, int tmin, int tmax, int cap, int* threads, ScoreLay* lay, size_t* smem) {
    const int64_t nblk = (p0 + R - 1) / R;
    const int64_t nbx = nblk + ((1 << wtop) > R ? (1 << wtop) / R : 1);
    const int64_t items = nblk * (R / (R < 16 ? R : 16));
    int64_t t = ((items + rounds - 1) / rounds + 31) / 32 * 32;
    t = t < tmin ? tmin : (t > tmax ? tmax : t);
    *threads = (int)t;
    size_t off = (size_t)nbx * R * 4;
    lay->cap = cap;
    lay->offs = lay->list = (uint32_t)off;
    const size_t offs = (size_t)nbx * (std::is_integral<V>::value ? 4 : 8);
    const size_t list = std::is_integral<V>::value ? 0 : (size_t)t * (size_t)lay->cap * 4;
    off += ((offs > list ? offs : list) + 15) & ~(size_t)15;
    lay->aux = (uint32_t)off;
    *smem = off + 4 * (std::is_integral<V>::value ? score_nb(R) : score_pack(R));
}

template <class V, int R, bool ONE, bool FF, int MAXT, int MINB>
ffa_status score1_launch(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t m_rows,
                         uint32_t wmask, int wtop, int threads, const ScoreLay& lay, size_t smem, int32_t* d_status,
                         cudaStream_t st) {
    const void* fn = (const void*)k_score1<V, R, ONE, FF, MAXT, MINB>;
    if (smem + sizeof(S1Sh) > 227 * 1024) return fail(FFA_ERR_UNSUPPORTED, "score: profile too long for shared memory");
    ffa_status es = ensure_smem(fn, smem);
    if (es != FFA_OK) return es;
    int64_t resident = 0;  // persistent: every CTA resident
    es = resident_ctas(fn, threads, smem, &resident);
    if (es != FFA_OK) return es;
    const unsigned grid = (unsigned)(count < resident ? count : resident);
    k_score1<V, R, ONE, FF, MAXT, MINB>
        <<<grid, threads, smem, st>>>((const V*)d_prof, sg, m_rows, trial0, count, wmask, wtop, lay, d_status);
    FFA_LAUNCH_CHECK("k_score1");
    count_launch();
    return FFA_OK;
}

// p0: the longest profile of the group
template <class V, bool FF>
ffa_status score1_t(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t p0,
                    int64_t m_rows, const ScoreWidths& wd, int32_t* d_status, cudaStream_t st) {
    uint32_t wmask = 0;
    int wtop = 0;
    for (int i = 0; i < wd.n; ++i) {
        int n = 0;
        while ((1 << n) < wd.w[i]) ++n;
        wmask |= 1u << n;
        wtop = n > wtop ? n : wtop;
    }
    int threads = 0;
    ScoreLay lay;
    size_t smem = 0;
#define FFA_SCORE1(RR, ONE, MAXT, MINB)                                                                          \
    score1_launch<V, RR, ONE, FF, MAXT, MINB>(d_prof, sg, count, trial0, m_rows, wmask, wtop, threads, lay, smem, \
                                              d_status, st)
    const int shape = score_shape(p0, wd.w[wd.n - 1]);
    lay.group = score_scan_group(shape);
    // CTA shapes, measured with ready profiles of 366..30000 bins: threads
    // against registers.  Fewer threads that hold their item in registers
    // beat more threads that spill (20000 bins: 27.7k SM cycles a profile
    // with 448 threads of 72 registers, 35.7k with 640 of 48).
    //
    // Few profiles: when no SM gets more than a few CTAs the call takes one
    // profile's latency, not its share of the SM, so a profile gets the
    // threads that its items and the SM's registers allow (records do not
    // depend on it).  `each`: CTAs of the busiest SM.
    const int64_t each = (count + sm_count() - 1) / sm_count();
    switch (shape) {
        case 0: {
            // Six bins a thread, 768 threads an SM: 150 profiles of 1100 bins
            // take 9.3 us (one warp each: 13.1), of 700 9.0 (11.2); 800 of
            // 1100 12 (14.8).  From seven an SM on the shapes below are as
            // fast (1500 of 1100: 15).
            const int64_t few = each <= 6 ? std::min<int64_t>({256, (p0 / 6 + 31) & ~31, (768 / each) & ~31}) : 0;
            if (few >= 64) {
                score1_shape<V, 8>(p0, wtop, 1, (int)few, (int)few, 10, &threads, &lay, &smem);
                return FFA_SCORE1(8, false, 256, 4);
            }
            // One warp a profile up to 1200 bins (1100 bins: 2.3k SM cycles,
            // 2.8k with two warps; 366 bins: 1.25k and 2.2k); above, two for
            // ready profiles (1489 bins: 2.8k, 3.0k with one), one in a search
            // (12 DM trials: 278 ms, 291 ms with two).
            if constexpr (!FF) {
                if (p0 > 1200) {
                    score1_shape<V, 8>(p0, wtop, 3, 64, 64, 9, &threads, &lay, &smem);
                    return FFA_SCORE1(8, false, 64, 12);
                }
            }
            // (80 registers fit 25 CTAs; a bound of 24 spills)
            score1_shape<V, 8>(p0, wtop, 1, 32, 32, 13, &threads, &lay, &smem);
            return FFA_SCORE1(8, true, 32, 22);
        }
        case 1:
        case 2: {
            score1_shape<V, 16>(p0, wtop, p0 <= 10240 ? 3 : 2, 64, 384, 9, &threads, &lay, &smem);
            // One item a thread, 512 threads of 128 registers an SM: 150
            // profiles of 3001 bins take 10.6 us (64 threads: 16.4), of 9001
            // 13.6 (16.1, 192 threads), 300 of 4201 12.3 (17.5), 500 14.5
            // of 3001 (20.6).
            const int64_t few = each <= 4 ? std::min<int64_t>(((p0 + 15) / 16 + 63) & ~63, (512 / each) & ~31) : 0;
            if (few > threads) {
                score1_shape<V, 16>(p0, wtop, 1, (int)few, (int)few, 9, &threads, &lay, &smem);
                return FFA_SCORE1(16, false, 512, 1);
            }
            return FFA_SCORE1(16, false, 384, 2);
        }
        default:
            // two profiles an SM while their shared memory fits, else one (or
            // if no SM gets a second: 150 of 20000 bins 21.7 us, 26.2 with
            // the two's threads)
            score1_shape<V, 32>(p0, wtop, 3, 320, 448, 7, &threads, &lay, &smem);
            if (each > 1 && 2 * (smem + sizeof(S1Sh) + 1024) <= 228 * 1024) return FFA_SCORE1(32, false, 448, 2);
            // (threads of the one, 4096 x 29705: float 618 us with 640, 631
            // with 768; int 692 and 678)
            if constexpr (std::is_integral<V>::value) {
                score1_shape<V, 32>(p0, wtop, 2, 512, 768, 9, &threads, &lay, &smem);
                return FFA_SCORE1(32, false, 768, 1);
            } else {
                score1_shape<V, 32>(p0, wtop, 3, 512, 640, 9, &threads, &lay, &smem);
                return FFA_SCORE1(32, false, 640, 1);
            }
    }
#undef FFA_SCORE1
}

ffa_status score1_dispatch(const void* d_prof, const ScoreGroup& sg, int32_t precision, bool fused, int64_t count,
                           int64_t trial0, int64_t p0max, int64_t m_rows, const ScoreWidths& wd, int32_t* d_status,
                           cudaStream_t st) {
    if (count <= 0) return FFA_OK;
    if (score_shape(p0max, wd.w[wd.n - 1]) < 0)
        return fail(FFA_ERR_UNSUPPORTED, "score: profile longer than 32768 bins");
    if (precision == FFA_FOLD_F32)
        return fused ? score1_t<float, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, d_status, st)
                     : score1_t<float, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, d_status, st);
    return fused ? score1_t<int32_t, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, d_status, st)
                 : score1_t<int32_t, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, d_status, st);
}

}  // namespace

int score_scan_group(int shape) { return shape == 0 ? 256 : (shape == 1 ? 512 : 1024); }

// The scorers' block length by profile length: 0: 8 bins (up to 2048), 1: 16
// (up to 8192), 2: 16, 3: 32, -1: too long; the extension by the widest box
// counts too.  Grouped launches hold one shape only, so that a profile's
// record does not depend on what it is grouped with.
int score_shape(int64_t p0, int wmax) {
    auto fits = [&](int64_t r, int64_t blocks, int64_t ext) {
        return p0 >= 1 && (p0 + r - 1) / r <= blocks && (p0 + wmax + r) / r + 1 <= ext;
    };
    return fits(8, 256, 512) ? 0 : fits(16, 512, 1024) ? 1 : fits(16, 1024, 2048) ? 2 : fits(32, 1024, 2048) ? 3 : -1;
}

ScoreGroup score_single(int64_t p0, int64_t ld, int64_t count, ffa_record* d_rec) {
    ScoreGroup sg;
    sg.n = 1;
    sg.t0[0] = 0;
    sg.t0[1] = count;
    sg.p0[0] = (int32_t)p0;
    sg.off[0] = 0;
    sg.ld[0] = ld;
    sg.rec[0] = d_rec;
    return sg;
}

ScoreGroup score_group(int n, const int64_t* p0, const int64_t* off, int64_t m_rows, ffa_record* const* recs,
                       int64_t* p0max) {
    ScoreGroup sg;
    sg.n = n;
    *p0max = 0;
    for (int i = 0; i < n; ++i) {
        sg.t0[i] = (int64_t)i * m_rows;
        sg.p0[i] = (int32_t)p0[i];
        sg.off[i] = off[i];
        sg.ld[i] = plane_pitch(p0[i]);
        sg.rec[i] = recs[i];
        *p0max = p0[i] > *p0max ? p0[i] : *p0max;
    }
    sg.t0[n] = (int64_t)n * m_rows;
    return sg;
}

ffa_status launch_score_alg1(const void* d_prof, int32_t precision, bool fused, int64_t count, int64_t trial0, int64_t p0,
                         int64_t ld, int64_t m_rows, const ScoreWidths& wd, ffa_record* d_rec, int32_t* d_status,
                         cudaStream_t st) {
    return score1_dispatch(d_prof, score_single(p0, ld, count, d_rec), precision, fused, count, trial0, p0, m_rows, wd,
                           d_status, st);
}

ffa_status launch_score_alg1_group(const void* d_plane, int32_t precision, int n, const int64_t* p0, const int64_t* off,
                               int64_t m_rows, const ScoreWidths& wd, ffa_record* const* recs, int32_t* d_status,
                               cudaStream_t st) {
    if (n < 1 || n > FOLD_GROUP_MAX) return fail(FFA_ERR_ARG, "score group: 1..FOLD_GROUP_MAX base periods");
    int64_t p0max = 0;
    const ScoreGroup sg = score_group(n, p0, off, m_rows, recs, &p0max);
    return score1_dispatch(d_plane, sg, precision, true, (int64_t)n * m_rows, 0, p0max, m_rows, wd, d_status, st);
}

}  // namespace ffa
