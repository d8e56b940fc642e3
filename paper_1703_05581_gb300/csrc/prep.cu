// Series preparation on the GPU (Section 2.3 of the paper):
//   * pre-downsampling by D0 and per-octave downsampling by 2 (FP64 sums);
//   * the dynamic running-median dereddening, exact;
//   * FP64 normalisation to FP32 z, or to the int8 code q = clip(rint(16 z)).
//
// Running median design (exact, tiled).  A CTA owns T consecutive outputs
// a..l at a time.  Their windows all contain the core C = [s_l, e_a]; window
// i is C plus |F_i| <= T-1 fringe samples left and right of it.  One pass over
// the tile's union counts the core samples below a value bracket and gathers
// the samples inside it (keyed by an order-preserving 64-bit integer,
// classified on its top 32 bits); they are sorted, and output i's order
// statistic is found by walking the few gathered fringe samples, the only
// ones whose membership depends on i.  The counts are exact, so a bracket is
// only a guess that is checked: a median outside it fails the tile's attempt
// and the next bracket is tried,
//   1. around the previous tile's medians (a CTA takes consecutive tiles;
//      a window of W samples changes by T of them from tile to tile),
//   2. wider, or exactly those medians' range if that bracket held too many
//      samples (series of few distinct values),
//   3. quantiles of a sample of the core,
//   4. the proven bracket: the rank-r element of window i lies between C's
//      order statistics r - |F_i| and r, so with rho_lo = min_i (r1_i - |F_i|)
//      and rho_hi = max_i r2_i every median of the tile lies in [C_(rho_lo),
//      C_(rho_hi)], whose 24-bit key prefixes two histogram passes over C
//      find (T <= (W+1)/4 keeps rho_lo >= 0 and rho_hi < |C|).
// A bracket that holds more equal samples than fit is settled value by value
// (rm_levels), from the proven bracket's lowest value on in the end.
// Bound by L2: the union is read once per tile, 8 (W + T) bytes for T outputs.
// 2^24 samples, W = 62501: 1.9 ms; 13.9 ms with the proven bracket alone (three
// passes, a bitonic sort of about T samples and a walk over all of them).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace ffa {

// ---------------------------------------------------------------------------
// downsampling
// ---------------------------------------------------------------------------
template <class T>
__global__ void k_downsample(const T* __restrict__ x, int64_t m, int64_t f,
                             double* __restrict__ y) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const T* p = x + f * i;
        double s = 0.0;
        for (int64_t j = 0; j < f; ++j) s += (double)p[j];
        y[i] = s;
    }
}

__global__ void k_downsample2(const double* __restrict__ x, int64_t m, double* __restrict__ y) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        double2 v = reinterpret_cast<const double2*>(x)[i];
        y[i] = (0.0 + v.x) + v.y;
    }
}

static int grid_for(int64_t m, int block) {
    int64_t g = (m + block - 1) / block;
    int64_t cap = (int64_t)sm_count() * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

ffa_status launch_downsample(const void* d_in, int32_t in_type, int64_t n, int64_t f,
                             double* d_out, cudaStream_t st) {
    int64_t m = n / f;
    if (m <= 0) return FFA_OK;
    if (in_type == FFA_IN_F64 && f == 2 && ((uintptr_t)d_in % 16) == 0) {
        k_downsample2<<<grid_for(m, 256), 256, 0, st>>>((const double*)d_in, m, d_out);
    } else if (in_type == FFA_IN_F32) {
        k_downsample<float><<<grid_for(m, 256), 256, 0, st>>>((const float*)d_in, m, f, d_out);
    } else if (in_type == FFA_IN_U8) {
        k_downsample<uint8_t><<<grid_for(m, 256), 256, 0, st>>>((const uint8_t*)d_in, m, f, d_out);
    } else if (in_type == FFA_IN_F64) {
        k_downsample<double><<<grid_for(m, 256), 256, 0, st>>>((const double*)d_in, m, f, d_out);
    } else {
        return fail(FFA_ERR_ARG, "downsample: bad input type");
    }
    FFA_LAUNCH_CHECK("k_downsample");
    count_launch();
    return FFA_OK;
}

// ---------------------------------------------------------------------------
// block-wide helpers
// ---------------------------------------------------------------------------
template <class V>
__device__ V block_reduce_min(V v, V* s_tmp) {
    for (int o = 16; o > 0; o >>= 1) {
        V u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u < v ? u : v;
    }
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) s_tmp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        v = lane < nw ? s_tmp[lane] : s_tmp[0];
        for (int o = 16; o > 0; o >>= 1) {
            V u = __shfl_xor_sync(0xffffffffu, v, o);
            v = u < v ? u : v;
        }
        if (lane == 0) s_tmp[0] = v;
    }
    __syncthreads();
    V r = s_tmp[0];
    __syncthreads();
    return r;
}

template <class V>
__device__ V block_reduce_max(V v, V* s_tmp) {
    for (int o = 16; o > 0; o >>= 1) {
        V u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u > v ? u : v;
    }
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) s_tmp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        v = lane < nw ? s_tmp[lane] : s_tmp[0];
        for (int o = 16; o > 0; o >>= 1) {
            V u = __shfl_xor_sync(0xffffffffu, v, o);
            v = u > v ? u : v;
        }
        if (lane == 0) s_tmp[0] = v;
    }
    __syncthreads();
    V r = s_tmp[0];
    __syncthreads();
    return r;
}

// Exclusive prefix sum over the block of one uint32 per thread.
__device__ uint32_t block_exscan(uint32_t v, uint32_t* s_tmp, uint32_t* total) {
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    __syncthreads();
    if (lane == 31) s_tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        uint32_t y = lane < nw ? s_tmp[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
        if (lane < nw) s_tmp[lane] = y;  // inclusive warp totals
    }
    __syncthreads();
    uint32_t base = warp > 0 ? s_tmp[warp - 1] : 0u;
    if (total) *total = s_tmp[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + x - v;
}

// Find the bin of a histogram (nbins a multiple of blockDim) that holds the
// element of 0-based rank `rank`; returns it via *bin and the count of
// elements in lower bins via *below.  Requires rank < total.
__device__ void block_find_rank(const uint32_t* hist, int nbins, uint32_t rank, uint32_t* s_tmp,
                                int* s_bin, uint32_t* s_below) {
    int per = nbins / blockDim.x;
    int b0 = threadIdx.x * per;
    uint32_t sum = 0;
    for (int t = 0; t < per; ++t) sum += hist[b0 + t];
    uint32_t ex = block_exscan(sum, s_tmp, nullptr);
    if (rank >= ex && rank < ex + sum) {
        uint32_t c = ex;
        for (int t = 0; t < per; ++t) {
            uint32_t hcount = hist[b0 + t];
            if (rank < c + hcount) {
                *s_bin = b0 + t;
                *s_below = c;
                break;
            }
            c += hcount;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// small windows (W <= 127): direct rank counting per output
// ---------------------------------------------------------------------------
__global__ void k_runmed_small(const double* __restrict__ x, int64_t n, int64_t w,
                               double* __restrict__ resid) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t h = w / 2;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        int64_t s = i - h < 0 ? 0 : i - h;
        int64_t e = i + h > n - 1 ? n - 1 : i + h;
        int64_t cnt = e - s + 1;
        int64_t r1 = (cnt - 1) / 2, r2 = cnt / 2;
        double v1 = 0.0, v2 = 0.0;
        for (int64_t j = s; j <= e; ++j) {
            double v = x[j];
            int64_t lt = 0, le = 0;
            for (int64_t t = s; t <= e; ++t) {
                double u = x[t];
                lt += (u < v);
                le += (u <= v);
            }
            if (lt <= r1 && r1 < le) v1 = v;
            if (lt <= r2 && r2 < le) v2 = v;
        }
        double med = (r1 == r2) ? v1 : (v1 + v2) / 2;
        resid[i] = x[i] - med;
    }
}

// ---------------------------------------------------------------------------
// tiled exact running median
// ---------------------------------------------------------------------------
constexpr int RM_CAP = 4096;    // gathered samples (power of two)
constexpr int RM_MAXT = 1024;   // largest tile
constexpr int RM_NT = 512;      // threads of the largest tile's CTA
constexpr int RM_NBK = 1024;    // buckets of the sort over a bracket

struct RmShared {
    union {
        struct {
            uint32_t hist1[4096], hist2a[4096], hist2b[4096];
        };
        struct {
            uint64_t ckey[RM_CAP];
            uint32_t coff[RM_CAP];
        };
    };
    uint16_t ord[RM_CAP];  // the gathered samples in key order
    union {
        // gathered fringe samples in key order: sorted place | index << 12 | right << 23
        uint32_t fringe[2 * RM_MAXT];
        uint16_t place[RM_CAP];  // while sorting: a sample's bucket, then its rank
    };
    uint32_t bkt[RM_NBK];
    uint32_t fbits[RM_CAP / 32];  // sorted places that hold fringe samples
    // fringe samples below the bracket: bits, and the counts before each word
    uint32_t lbits[RM_MAXT / 32], rbits[RM_MAXT / 32], lpre[RM_MAXT / 32 + 1], rpre[RM_MAXT / 32 + 1];
    // the same for the gathered fringe samples that precede every output's median
    uint32_t l2bits[RM_MAXT / 32], r2bits[RM_MAXT / 32], l2pre[RM_MAXT / 32 + 1], r2pre[RM_MAXT / 32 + 1];
    uint32_t tmp[64];
    int64_t tmp64[64];
    unsigned long long kmin, blo, bhi;
    float flo, finv;
    uint32_t ccount, cbelow, nf, tmin, mmin, mmax, pmin, pmax;
    int big;
    int bin_a, bin_b;
    uint32_t below_a, below_b;
};

// Sort the first cc of ckey (and coff) by key: bitonic over the next power of two.
__device__ void rm_bitonic(RmShared& sh, uint32_t cc) {
    const int T = blockDim.x, tid = threadIdx.x;
    uint32_t np2 = 1;
    while (np2 < cc) np2 <<= 1;
    for (uint32_t t = cc + tid; t < np2; t += T) {
        sh.ckey[t] = ~0ull;
        sh.coff[t] = 0xffffffffu;
    }
    __syncthreads();
    for (uint32_t kk = 2; kk <= np2; kk <<= 1) {
        for (uint32_t jj = kk >> 1; jj > 0; jj >>= 1) {
            for (uint32_t p = tid; p < np2 / 2; p += T) {
                const uint32_t t = ((p & ~(jj - 1)) << 1) | (p & (jj - 1)), u = t | jj;
                const uint64_t kt = sh.ckey[t], ku = sh.ckey[u];
                if ((kt > ku) == ((t & kk) == 0)) {
                    sh.ckey[t] = ku;
                    sh.ckey[u] = kt;
                    const uint32_t o = sh.coff[t];
                    sh.coff[t] = sh.coff[u];
                    sh.coff[u] = o;
                }
            }
            __syncthreads();
        }
    }
}

// ord = the gathered samples 0 .. cc-1 in key order: by buckets linear in the
// value across the bracket (flo, finv; a monotone map, so buckets are in
// order), then by counting inside a bucket -- one or two samples each, where
// a bitonic sort takes 55 barriers for a thousand samples.  A bucket of many
// samples needs no order if they are all equal (a series of whole numbers);
// only one of many different samples takes the bitonic sort.
constexpr uint32_t RM_BIG = 64;
__device__ void rm_sort(RmShared& sh, uint32_t cc) {
    const int T = blockDim.x, tid = threadIdx.x;
    for (int b = tid; b < RM_NBK; b += T) sh.bkt[b] = 0;
    if (tid == 0) sh.big = 0;
    __syncthreads();
    const float flo = sh.flo, finv = sh.finv;
    for (uint32_t i = tid; i < cc; i += T) {
        const float f = __fmul_rn(__fsub_rn(__double2float_rn(dkey_inv(sh.ckey[i])), flo), finv);
        const int b = min(max((int)f, 0), RM_NBK - 1);
        sh.place[i] = (uint16_t)b;
        if (atomicAdd(&sh.bkt[b], 1u) >= RM_BIG) sh.big = 1;
    }
    __syncthreads();
    {
        const int per = RM_NBK / T, b0 = tid * per;
        uint32_t s = 0;
        for (int t = 0; t < per; ++t) s += sh.bkt[b0 + t];
        uint32_t c = block_exscan(s, sh.tmp, nullptr);
        for (int t = 0; t < per; ++t) {
            const uint32_t hc = sh.bkt[b0 + t];
            sh.bkt[b0 + t] = c;
            c += hc;
        }
    }
    __syncthreads();
    for (uint32_t i = tid; i < cc; i += T) sh.ord[atomicAdd(&sh.bkt[sh.place[i]], 1u)] = (uint16_t)i;
    __syncthreads();  // bkt[b] is now the end of bucket b
    auto first = [&](int b) { return b ? sh.bkt[b - 1] : 0u; };
    const bool big = sh.big != 0;
    if (big) {
        bool mixed = false;
        for (uint32_t i = tid; i < cc; i += T) {
            const int b = sh.place[i];
            const uint32_t e0 = first(b);
            mixed |= sh.bkt[b] - e0 > RM_BIG && sh.ckey[i] != sh.ckey[sh.ord[e0]];
        }
        if (__syncthreads_or(mixed)) {
            rm_bitonic(sh, cc);
            for (uint32_t i = tid; i < cc; i += T) sh.ord[i] = (uint16_t)i;
            __syncthreads();
            return;
        }
    }
    for (uint32_t at = tid; at < cc; at += T) {
        const uint32_t i = sh.ord[at];
        const int b = sh.place[i];
        const uint32_t e0 = first(b), e1 = sh.bkt[b];
        uint32_t r = at;
        if (e1 - e0 <= RM_BIG) {
            const uint64_t k = sh.ckey[i];
            r = e0;
            for (uint32_t e = e0; e < e1; ++e) {
                const uint32_t o = sh.ord[e];
                const uint64_t ko = sh.ckey[o];
                r += ko < k || (ko == k && o < i);
            }
        }
        sh.place[i] = (uint16_t)r;
    }
    __syncthreads();
    for (uint32_t i = tid; i < cc; i += T) sh.ord[sh.place[i]] = (uint16_t)i;
    __syncthreads();
}

// Exact rank-`rank` key of x[s..e] by an 8-pass, 8-bit radix select over the
// whole CTA (slow path for tiles whose candidate set overflows).
__device__ uint64_t cta_select_key(const double* __restrict__ x, int64_t s, int64_t e, uint32_t rank,
                                   RmShared& sh) {
    uint64_t prefix = 0, mask = 0;
    for (int pass = 0; pass < 8; ++pass) {
        int shift = 56 - 8 * pass;
        for (int b = threadIdx.x; b < 256; b += blockDim.x) sh.hist1[b] = 0;
        __syncthreads();
        for (int64_t p = s + threadIdx.x; p <= e; p += blockDim.x) {
            uint64_t k = dkey(x[p]);
            if ((k & mask) == prefix) atomicAdd(&sh.hist1[(k >> shift) & 0xff], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t c = 0;
            for (int b = 0; b < 256; ++b) {
                if (rank < c + sh.hist1[b]) {
                    sh.bin_a = b;
                    sh.below_a = c;
                    break;
                }
                c += sh.hist1[b];
            }
        }
        __syncthreads();
        rank -= sh.below_a;
        prefix |= (uint64_t)sh.bin_a << shift;
        mask |= (uint64_t)0xff << shift;
        __syncthreads();
    }
    return prefix;
}

__device__ __forceinline__ uint32_t hi_key(uint64_t bits) {  // top 32 bits of dkey
    const uint32_t u = (uint32_t)(bits >> 32);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}

// One warp: the counts of set bits before each of 32 words (pre[32]: all).
__device__ __forceinline__ void rm_word_prefix(const uint32_t* bits, uint32_t* pre) {
    const int lane = threadIdx.x & 31;
    const uint32_t v = __popc(bits[lane]);
    uint32_t c = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) c += u;
    }
    pre[lane] = c - v;
    if (lane == 31) pre[32] = c;
}
// set bits below position q (<= RM_MAXT)
__device__ __forceinline__ uint32_t rm_bits_before(const uint32_t* bits, const uint32_t* pre, uint32_t q) {
    return pre[q >> 5] + ((q & 31) ? __popc(bits[q >> 5] & ((1u << (q & 31)) - 1)) : 0u);
}

// The medians of outputs a .. a + no - 1 value by value, for series with many
// equal samples: a pass over the tile's union counts the core's samples up to
// a value v, flags the fringe's and finds the next larger value; an output's
// order statistic is the first v that holds its rank.  The first pass, at
// v = start, only counts: false if a rank lies there, or after `limit` values.
// A series of two levels takes three passes where a selection for each output
// of the tile takes thousands.
__device__ __noinline__ bool rm_levels(const double* __restrict__ x, int64_t n, int64_t h, int64_t a, int no,
                                       uint64_t start, int limit, double* __restrict__ resid, RmShared& sh) {
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto win_s = [&](int64_t q) { return q - h < 0 ? (int64_t)0 : q - h; };
    auto win_e = [&](int64_t q) { return q + h > n - 1 ? n - 1 : q + h; };
    const int64_t l = a + no - 1, s_a = win_s(a), e_a = win_e(a), s_l = win_s(l), e_l = win_e(l);
    uint64_t* first = sh.ckey;   // an output's first order statistic
    uint32_t* state = sh.coff;   // how many of the two are known
    for (int o = tid; o < no; o += NT) state[o] = 0;
    if (tid == 0) {
        sh.mmin = 0xffffffffu;
        sh.mmax = 0u;
    }
    uint64_t v = start;
    for (int it = 0; it <= limit; ++it) {
        if (tid == 0) {
            sh.cbelow = 0;
            sh.kmin = ~0ull;
        }
        __syncthreads();
        uint32_t upto = 0;
        uint64_t next = ~0ull;
        auto look = [&](double d) {
            const uint64_t k = dkey(d);
            const bool in = k <= v;
            if (!in && k < next) next = k;
            return in;
        };
        {
            const int64_t step = NT;
            int64_t p = s_l + tid;
            for (; p + 3 * step <= e_a; p += 4 * step) {
                double d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) d[i] = x[p + i * step];
#pragma unroll
                for (int i = 0; i < 4; ++i) upto += look(d[i]);
            }
            for (; p <= e_a; p += step) upto += look(x[p]);
        }
        for (int side = 0; side < 2; ++side) {
            const int64_t p0 = side ? e_a + 1 : s_a;
            const int sz = (int)(side ? e_l - e_a : s_l - s_a);
            for (int q0 = warp * 32; q0 < RM_MAXT; q0 += NT) {
                bool in = false;
                if (q0 + lane < sz) in = look(x[p0 + q0 + lane]);
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (lane == 0) (side ? sh.rbits : sh.lbits)[q0 >> 5] = m;
            }
        }
        upto = __reduce_add_sync(0xffffffffu, upto);
        if (lane == 0) atomicAdd(&sh.cbelow, upto);
        if (next != ~0ull && next < *(volatile unsigned long long*)&sh.kmin) atomicMin(&sh.kmin, (unsigned long long)next);
        __syncthreads();
        if (warp == 0) {
            rm_word_prefix(sh.lbits, sh.lpre);
            rm_word_prefix(sh.rbits, sh.rpre);
        }
        __syncthreads();
        const uint32_t core = sh.cbelow;
        next = sh.kmin;
        bool bad = false, open = false;
        for (int o = tid; o < no; o += NT) {
            uint32_t st = state[o];
            if (st == 2) continue;
            const int64_t s_i = win_s(a + o), e_i = win_e(a + o), n_i = e_i - s_i + 1;
            const int64_t cnt = (int64_t)core + sh.lpre[32] - rm_bits_before(sh.lbits, sh.lpre, (uint32_t)(s_i - s_a)) +
                                rm_bits_before(sh.rbits, sh.rpre, (uint32_t)(e_i - e_a));
            if (st == 0 && (n_i - 1) / 2 < cnt) {
                if (it == 0) bad = true;
                first[o] = v;
                st = 1;
                atomicMin(&sh.mmin, (uint32_t)(v >> 32));
            }
            if (st == 1 && n_i / 2 < cnt) {
                const double v1 = dkey_inv(first[o]), v2 = dkey_inv(v);
                const double med = (n_i & 1) ? v1 : (v1 + v2) / 2;
                resid[a + o] = x[a + o] - med;
                st = 2;
                atomicMax(&sh.mmax, (uint32_t)(v >> 32));
            }
            state[o] = st;
            open |= st != 2;
        }
        if (__syncthreads_or(bad)) return false;
        if (!__syncthreads_or(open)) return true;
        if (next == ~0ull) return false;
        v = next;
    }
    return false;
}

// T outputs per tile, blockDim threads.  The CTAs take runs of `run`
// consecutive tiles in turn: long enough for one tile to predict the next,
// short enough that the CTAs' windows lie together in L2.
__global__ void __launch_bounds__(RM_NT, 3) k_runmed_tile(const double* __restrict__ x, int64_t n, int64_t w, int T,
                                                          int64_t tiles, int64_t run, double* __restrict__ resid,
                                                          int32_t* d_status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RmShared& sh = *reinterpret_cast<RmShared*>(smem_raw);
    const int NT = blockDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t h = w / 2;
    auto win_s = [&](int64_t q) { return q - h < 0 ? (int64_t)0 : q - h; };
    auto win_e = [&](int64_t q) { return q + h > n - 1 ? n - 1 : q + h; };
    bool known = false;         // pmin, pmax: the previous tile's medians (top key words)
    float wide = 0.0f;          // half-width of the bracket around them (thread 0)
    int64_t in_run = 0;
    auto learn = [&]() {
        if (tid != 0) return;
        // next tile: two ranges of this tile's medians to each side
        const float r = (float)(dkey_inv(((uint64_t)sh.mmax << 32) | 0xffffffffull) - dkey_inv((uint64_t)sh.mmin << 32));
        wide = fmaxf(2.0f * r, 0.7f * wide);
        sh.pmin = sh.mmin;
        sh.pmax = sh.mmax;
    };
    for (int64_t tile = blockIdx.x * run; tile < tiles;) {
        const int64_t a = tile * T;
        const int64_t l = (a + T < n ? a + T : n) - 1;
        const int no = (int)(l - a + 1);
        const int64_t s_a = win_s(a), e_a = win_e(a), s_l = win_s(l), e_l = win_e(l);
        const int64_t c0 = s_l, c1 = e_a, csize = c1 - c0 + 1;
        const int lsz = (int)(s_l - s_a), rsz = (int)(e_l - e_a);
        // proven core ranks; they grow with i or fall, by pieces: all outputs
        int64_t lo_need = INT64_MAX, hi_need = INT64_MIN;
        for (int o = tid; o < no; o += NT) {
            const int64_t n_i = win_e(a + o) - win_s(a + o) + 1;
            const int64_t lo = (n_i - 1) / 2 - (n_i - csize), hi = n_i / 2;
            lo_need = lo < lo_need ? lo : lo_need;
            hi_need = hi > hi_need ? hi : hi_need;
        }
        lo_need = block_reduce_min<int64_t>(lo_need, sh.tmp64);
        hi_need = block_reduce_max<int64_t>(hi_need, sh.tmp64);
        const bool bracket_ok = csize > 0 && lo_need >= 0 && hi_need < csize;
        bool done = false, over = false, levels = false;
        for (int attempt = known ? 0 : 2; bracket_ok && attempt < 4 && !done; ++attempt) {
            // ---- the bracket, as keys [blo, bhi] and as floats for the sort
            auto set_bracket = [&](double lo, double hi) {  // thread 0
                sh.blo = dkey(lo);
                sh.bhi = dkey(hi);
                sh.flo = __double2float_rn(lo);
                sh.finv = (float)RM_NBK / (__double2float_rn(hi) - sh.flo);
            };
            if (attempt < 2) {
                // 1: the tight one if too many were gathered, else a wider one
                if (tid == 0) {
                    const double lo = dkey_inv((uint64_t)sh.pmin << 32), hi = dkey_inv(((uint64_t)sh.pmax << 32) | 0xffffffffull);
                    const double d = attempt == 0 ? (double)wide : (over ? 0.0 : 4.0 * (double)wide);
                    set_bracket(lo - d, hi + d);
                }
            } else if (attempt == 2) {
                if (csize < 256) continue;
                int ns = 128;
                while (ns * 2 <= RM_CAP && ns * 2 <= csize / 2 && (ns < 1024 || (int64_t)ns * 20 < csize)) ns *= 2;
                const int64_t stride = csize / ns;
                float* fv = reinterpret_cast<float*>(sh.coff);
                float mn = INFINITY, mx = -INFINITY;
                for (int i = tid; i < ns; i += NT) {
                    const float v = __double2float_rn(x[c0 + i * stride]);
                    fv[i] = v;
                    mn = fminf(mn, v);
                    mx = fmaxf(mx, v);
                }
                for (int b = tid; b < RM_NBK; b += NT) sh.bkt[b] = 0;
                if (tid == 0) sh.nf = 0;
                mn = block_reduce_min<float>(mn, reinterpret_cast<float*>(sh.tmp));
                mx = block_reduce_max<float>(mx, reinterpret_cast<float*>(sh.tmp));
                const float inv = (float)RM_NBK / (mx - mn);
                uint32_t same = 0;  // neighbours of one value: few values in all
                for (int i = tid; i < ns; i += NT) {
                    atomicAdd(&sh.bkt[min(max((int)((fv[i] - mn) * inv), 0), RM_NBK - 1)], 1u);
                    same += (i & 1) && fv[i] == fv[i - 1];
                }
                same = __reduce_add_sync(0xffffffffu, same);
                if (lane == 0) atomicAdd(&sh.nf, same);
                // a quarter of the proven rank range on each side of its
                // middle, and 2.5 sigma of the sample quantile
                const float f = (float)ns / (float)csize, mid = 0.5f * (float)(lo_need + hi_need) * f;
                const float d = 0.25f * (float)(hi_need - lo_need) * f + 1.25f * sqrtf((float)ns) + 1.0f;
                const int ilo = max((int)floorf(mid - d), 0), ihi = min((int)ceilf(mid + d), ns - 1);
                __syncthreads();
                block_find_rank(sh.bkt, RM_NBK, (uint32_t)ilo, sh.tmp, &sh.bin_a, &sh.below_a);
                block_find_rank(sh.bkt, RM_NBK, (uint32_t)ihi, sh.tmp, &sh.bin_b, &sh.below_b);
                levels = sh.nf >= (uint32_t)ns / 16;
                if (tid == 0)
                    set_bracket((double)(mn + (float)sh.bin_a / inv), (double)(mn + (float)(sh.bin_b + 1) / inv));
            } else {
                const uint32_t rho_lo = (uint32_t)lo_need, rho_hi = (uint32_t)hi_need;
                // pass 1: top 12 key bits over the core
                for (int b = tid; b < 4096; b += NT) {
                    sh.hist1[b] = 0;
                    sh.hist2a[b] = 0;
                    sh.hist2b[b] = 0;
                }
                __syncthreads();
                for (int64_t p = c0 + tid; p <= c1; p += NT) atomicAdd(&sh.hist1[dkey(x[p]) >> 52], 1u);
                __syncthreads();
                block_find_rank(sh.hist1, 4096, rho_lo, sh.tmp, &sh.bin_a, &sh.below_a);
                block_find_rank(sh.hist1, 4096, rho_hi, sh.tmp, &sh.bin_b, &sh.below_b);
                const uint32_t b1_lo = sh.bin_a, b1_hi = sh.bin_b;
                const uint32_t below1_lo = sh.below_a, below1_hi = sh.below_b;
                __syncthreads();
                // pass 2: next 12 bits inside the two selected top buckets
                for (int64_t p = c0 + tid; p <= c1; p += NT) {
                    uint64_t k = dkey(x[p]);
                    uint32_t top = (uint32_t)(k >> 52), sub = (uint32_t)(k >> 40) & 0xfff;
                    if (top == b1_lo) atomicAdd(&sh.hist2a[sub], 1u);
                    if (top == b1_hi && b1_hi != b1_lo) atomicAdd(&sh.hist2b[sub], 1u);
                }
                __syncthreads();
                block_find_rank(sh.hist2a, 4096, rho_lo - below1_lo, sh.tmp, &sh.bin_a, &sh.below_a);
                const uint32_t b2_lo = sh.bin_a;
                __syncthreads();
                block_find_rank(b1_hi == b1_lo ? sh.hist2a : sh.hist2b, 4096, rho_hi - below1_hi, sh.tmp, &sh.bin_b,
                                &sh.below_b);
                const uint32_t b2_hi = sh.bin_b;
                if (tid == 0) {
                    const uint64_t blo = (((uint64_t)b1_lo << 12) | b2_lo) << 40;
                    const uint64_t bhi = ((((uint64_t)b1_hi << 12) | b2_hi) << 40) | 0xffffffffffull;
                    set_bracket(dkey_inv(blo), dkey_inv(bhi));
                    sh.blo = blo;  // exactly, also where a key is no number's
                    sh.bhi = bhi;
                }
            }
            __syncthreads();  // blo, bhi; the sample and the histograms are done with
            const uint32_t klo = (uint32_t)(sh.blo >> 32), khi = (uint32_t)(sh.bhi >> 32), span = khi - klo;
            if (tid == 0) {
                sh.ccount = 0;
                sh.cbelow = 0;
            }
            __syncthreads();
            if (khi < klo) continue;
            if (levels) {
                done = rm_levels(x, n, h, a, no, sh.blo - 1, 4, resid, sh);
                known = done;
                if (done) {
                    learn();
                    continue;
                }
                levels = false;
                if (tid == 0) sh.cbelow = 0;
                __syncthreads();
            }
            // ---- gather the union's samples inside the bracket, count the
            // core's below it, flag the fringe's
            const unsigned long long* __restrict__ xb = reinterpret_cast<const unsigned long long*>(x);
            bool full = false;  // too many: the rest need not be looked at
            auto keep = [&](uint64_t bits, int64_t p) {
                const uint64_t k = (bits >> 63) ? ~bits : (bits | 0x8000000000000000ull);
                const uint32_t slot = atomicAdd(&sh.ccount, 1u);
                if (slot < RM_CAP) {
                    sh.ckey[slot] = k;
                    sh.coff[slot] = (uint32_t)(p - s_a);
                } else {
                    full = true;
                }
            };
            uint32_t below = 0;
            {
                const int64_t step = NT;
                int64_t p = c0 + tid;
                for (; !full && p + 7 * step <= c1; p += 8 * step) {
                    unsigned long long v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = xb[p + i * step];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t k = hi_key(v[i]);
                        below += k < klo;
                        if (k - klo <= span) keep(v[i], p + i * step);
                    }
                }
                for (; !full && p <= c1; p += step) {
                    const unsigned long long v = xb[p];
                    const uint32_t k = hi_key(v);
                    below += k < klo;
                    if (k - klo <= span) keep(v, p);
                }
            }
            for (int side = 0; side < 2; ++side) {
                const int64_t p0 = side ? e_a + 1 : s_a;
                const int sz = side ? rsz : lsz;
                for (int q0 = warp * 32; q0 < RM_MAXT; q0 += NT) {
                    const int q = q0 + lane;
                    bool lt = false;
                    if (q < sz) {
                        const unsigned long long v = xb[p0 + q];
                        const uint32_t k = hi_key(v);
                        lt = k < klo;
                        if (k - klo <= span) keep(v, p0 + q);
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, lt);
                    if (lane == 0) (side ? sh.rbits : sh.lbits)[q0 >> 5] = m;
                }
            }
            below = __reduce_add_sync(0xffffffffu, below);
            if (lane == 0) atomicAdd(&sh.cbelow, below);
            __syncthreads();
            const uint32_t cc = sh.ccount;
            over = cc > RM_CAP;
            if (over) {
                // many equal samples among those gathered: value by value
                uint32_t same = 0;
                for (int i = tid; i < RM_CAP / 2; i += NT) same += sh.ckey[2 * i] == sh.ckey[2 * i + 1];
                same = __reduce_add_sync(0xffffffffu, same);
                if (tid == 0) sh.cbelow = 0;
                __syncthreads();
                if (lane == 0) atomicAdd(&sh.cbelow, same);
                __syncthreads();
                const bool tied = sh.cbelow >= RM_CAP / 16;
                __syncthreads();
                if (tied) done = rm_levels(x, n, h, a, no, sh.blo - 1, 16, resid, sh);
                if (!done && attempt == 3) {
                    // exactly from the lowest value that can be a median on
                    const uint64_t lowest = cta_select_key(x, c0, c1, (uint32_t)lo_need, sh);
                    done = rm_levels(x, n, h, a, no, lowest - 1, RM_CAP, resid, sh);
                }
                known = done;
                if (done) learn();
                continue;
            }
            for (int b = tid; b < RM_CAP / 32; b += NT) sh.fbits[b] = 0;
            rm_sort(sh, cc);
            for (uint32_t j = tid; j < cc; j += NT) {
                const uint32_t off = sh.coff[sh.ord[j]];
                if (off < (uint32_t)lsz || off > (uint32_t)(e_a - s_a)) atomicOr(&sh.fbits[j >> 5], 1u << (j & 31));
            }
            __syncthreads();
            if (warp == 0) {
                rm_word_prefix(sh.lbits, sh.lpre);
                rm_word_prefix(sh.rbits, sh.rpre);
                sh.l2bits[lane] = 0;
                sh.r2bits[lane] = 0;
                // the gathered fringe samples, in key order
                const uint32_t cl = (uint32_t)lsz, cr = (uint32_t)(e_a - s_a);
                uint32_t fb[RM_CAP / 1024], cnt = 0;
#pragma unroll
                for (int i = 0; i < RM_CAP / 1024; ++i) {
                    fb[i] = sh.fbits[lane * (RM_CAP / 1024) + i];
                    cnt += __popc(fb[i]);
                }
                uint32_t at = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(0xffffffffu, at, o);
                    if (lane >= o) at += u;
                }
                if (lane == 31) sh.nf = at;
                at -= cnt;
#pragma unroll
                for (int i = 0; i < RM_CAP / 1024; ++i) {
                    while (fb[i]) {
                        const uint32_t j = (uint32_t)(lane * (RM_CAP / 1024) + i) * 32 + __ffs(fb[i]) - 1;
                        fb[i] &= fb[i] - 1;
                        const uint32_t off = sh.coff[sh.ord[j]];
                        sh.fringe[at++] = j | (off < cl ? off << 12 : ((off - cr - 1) << 12) | (1u << 23));
                    }
                }
                if (lane == 0) {
                    sh.mmin = 0xffffffffu;
                    sh.mmax = 0u;
                    sh.tmin = 0xffffffffu;
                }
            }
            __syncthreads();
            // ---- every output's order statistics
            const uint32_t nf = sh.nf, cb = sh.cbelow;
            // output o's windows: left fringe from q on, right fringe up to m;
            // the first wanted rank among the gathered samples (< 0: below
            // the bracket)
            auto place = [&](int o, uint32_t& q, uint32_t& m, int64_t& t2) -> int64_t {
                const int64_t s_i = win_s(a + o), e_i = win_e(a + o), n_i = e_i - s_i + 1;
                q = (uint32_t)(s_i - s_a);
                m = (uint32_t)(e_i - e_a);
                const int64_t below_i = (int64_t)cb + sh.lpre[32] - rm_bits_before(sh.lbits, sh.lpre, q) +
                                        rm_bits_before(sh.rbits, sh.rpre, m);
                t2 = n_i / 2 - below_i;
                return (n_i - 1) / 2 - below_i;
            };
            // Fringe samples sorted below every output's rank only count: how
            // many are in the output's window comes from bit counts again, and
            // the walk starts behind them.
            {
                uint32_t tm = 0xffffffffu;
                for (int o = tid; o < no; o += NT) {
                    uint32_t q, m;
                    int64_t t2;
                    const int64_t t1 = place(o, q, m, t2);
                    tm = min(tm, (uint32_t)(t1 < 0 ? 0 : (t1 > RM_CAP ? RM_CAP : t1)));
                }
                tm = __reduce_min_sync(0xffffffffu, tm);
                if (lane == 0) atomicMin(&sh.tmin, tm);
            }
            __syncthreads();
            {
                const uint32_t tmin = sh.tmin;
                for (uint32_t j = tid; j < nf; j += NT) {
                    const uint32_t e = sh.fringe[j], idx = (e >> 12) & 0x7ffu;
                    if ((e & 0xfffu) < tmin) atomicOr((e >> 23) ? &sh.r2bits[idx >> 5] : &sh.l2bits[idx >> 5], 1u << (idx & 31));
                }
            }
            __syncthreads();
            if (warp == 0) {
                rm_word_prefix(sh.l2bits, sh.l2pre);
                rm_word_prefix(sh.r2bits, sh.r2pre);
            }
            __syncthreads();
            const uint32_t nskip = sh.l2pre[32] + sh.r2pre[32];
            uint32_t lo32 = 0xffffffffu, hi32 = 0u;
            bool bad = false;
            for (int o = tid; o < no; o += NT) {
                uint32_t q, m;
                int64_t t2;
                const int64_t t1 = place(o, q, m, t2);
                if (t1 < 0 || t2 >= (int64_t)cc) {
                    bad = true;
                    continue;
                }
                uint32_t t = (uint32_t)t1, j = nskip, at = 0;
                uint32_t f = sh.l2pre[32] - rm_bits_before(sh.l2bits, sh.l2pre, q) + rm_bits_before(sh.r2bits, sh.r2pre, m);
                uint64_t k1 = 0;
                for (int want = 0; want < 2; ++want) {
                    bool hit = false;
                    for (; j < nf; ++j) {
                        const uint32_t e = sh.fringe[j], sp = e & 0xfffu, idx = (e >> 12) & 0x7ffu;
                        if (sp - j + f > t) break;  // a core sample comes first
                        if ((e >> 23) ? idx < m : idx >= q) {
                            if (sp - j + f == t) {
                                hit = true;
                                at = sp;
                                break;
                            }
                            ++f;
                        }
                    }
                    if (!hit) at = t - f + j;
                    if (at >= cc) {
                        bad = true;
                        break;
                    }
                    if (want == 0) k1 = sh.ckey[sh.ord[at]];
                    if (t2 == t1) break;
                    if (want == 0) {
                        ++t;
                        if (hit) {
                            ++f;
                            ++j;
                        }
                    }
                }
                if (bad) continue;
                const uint64_t k2 = sh.ckey[sh.ord[at]];
                const double v1 = dkey_inv(k1), v2 = dkey_inv(k2);
                const double med = (t1 == t2) ? v1 : (v1 + v2) / 2;
                resid[a + o] = x[a + o] - med;
                lo32 = min(lo32, (uint32_t)(k1 >> 32));
                hi32 = max(hi32, (uint32_t)(k2 >> 32));
            }
            lo32 = __reduce_min_sync(0xffffffffu, lo32);
            hi32 = __reduce_max_sync(0xffffffffu, hi32);
            if (lane == 0) {
                atomicMin(&sh.mmin, lo32);
                atomicMax(&sh.mmax, hi32);
            }
            done = !__syncthreads_or(bad);
            known = done;
            if (done) learn();
        }
        if (!done) {
            known = false;
            if (!bracket_ok) dev_fail(d_status, FFA_ERR_DEVICE);
            // slow exact path: per output, radix select over its own window
            for (int64_t q = a; q <= l; ++q) {
                int64_t s = win_s(q), e = win_e(q);
                int64_t cnt = e - s + 1;
                uint64_t k1 = cta_select_key(x, s, e, (uint32_t)((cnt - 1) / 2), sh);
                uint64_t k2 = (cnt % 2 == 1) ? k1 : cta_select_key(x, s, e, (uint32_t)(cnt / 2), sh);
                if (tid == 0) {
                    double v1 = dkey_inv(k1), v2 = dkey_inv(k2);
                    double med = (cnt % 2 == 1) ? v1 : (v1 + v2) / 2;
                    resid[q] = x[q] - med;
                }
                __syncthreads();
            }
        }
        __syncthreads();
        ++tile;
        if (++in_run == run) {
            in_run = 0;
            known = false;
            tile += (int64_t)(gridDim.x - 1) * run;
        }
    }
}

ffa_status launch_detrend(const double* d_raw, int64_t n, int32_t window, double* d_resid,
                          int32_t* d_status, cudaStream_t st) {
    if (n <= 0) return FFA_OK;
    int64_t w = window | 1;
    if (w <= 127) {
        k_runmed_small<<<grid_for(n, 256), 256, 0, st>>>(d_raw, n, w, d_resid);
        FFA_LAUNCH_CHECK("k_runmed_small");
        count_launch();
        return FFA_OK;
    }
    int T = 32;
    while (T * 2 <= RM_MAXT && T * 2 <= (w + 1) / 4) T *= 2;
    // a series inside one window: shorter tiles while few SMs have one (2^14
    // samples, W = 62501: 20.0 -> 18.4 us)
    while (n <= w && T > 256 && 4 * ((n + T - 1) / T) < (int64_t)sm_count()) T /= 2;
    size_t smem = sizeof(RmShared);
    ffa_status es = ensure_smem((const void*)k_runmed_tile, smem);
    if (es != FFA_OK) return es;
    const int64_t tiles = (n + T - 1) / T;
    // Shared memory fits three CTAs an SM whatever their threads: 512, or 256
    // for short tiles when every CTA takes many of them (barriers then count
    // for more than the samples).  Windows of 129 / 257 / 1025 samples: 2^22
    // samples 2.9 / 1.6 / 0.56 ms (6.1 / 3.5 / 0.67 with half a thread an
    // output, 3.2 / 1.7 / 0.60 with 512), 2^14 samples 43 / 22 / 20 us (129 / 70
    // / 27, and 50 / 26 / 20 with 256).
    // Persistent: consecutive tiles in one CTA predict each other's bracket.
    auto fn = (const void*)k_runmed_tile;
    int threads = RM_NT;
    int64_t grid = 0;
    es = resident_ctas(fn, threads, smem, &grid);
    if (es == FFA_OK && T <= 256 && tiles > 8 * grid) {
        threads = 256;
        es = resident_ctas(fn, threads, smem, &grid);
    }
    if (es != FFA_OK) return es;
    if (grid > tiles) grid = tiles;
    // runs of at most 16 tiles, as many for every CTA: 456 CTAs' runs of 1024
    // outputs cover 60 MB of the series, which L2 holds
    const int64_t rounds = (tiles + grid * 16 - 1) / (grid * 16);
    const int64_t run = (tiles + grid * rounds - 1) / (grid * rounds);
    k_runmed_tile<<<(unsigned)grid, threads, smem, st>>>(d_raw, n, w, T, tiles, run, d_resid, d_status);
    FFA_LAUNCH_CHECK("k_runmed_tile");
    count_launch();
    return FFA_OK;
}

// ---------------------------------------------------------------------------
// normalisation: FP64 mean and population std (fixed reduction tree)
// ---------------------------------------------------------------------------
constexpr int NRM_BLOCKS = 1024;
constexpr int NRM_THREADS = 256;

__device__ double block_sum_d(double v, double* s) {
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] = s[threadIdx.x] + s[threadIdx.x + o];
        __syncthreads();
    }
    double r = s[0];
    __syncthreads();
    return r;
}

// mode 0: partial sums of r; mode 1: partial sums of (r - mean)^2
__global__ void __launch_bounds__(NRM_THREADS) k_stats_partial(const double* __restrict__ r,
                                                               int64_t n, const double* stats,
                                                               int mode, double* partial) {
    __shared__ double s[NRM_THREADS];
    int64_t chunk = (n + NRM_BLOCKS - 1) / NRM_BLOCKS;
    int64_t b0 = (int64_t)blockIdx.x * chunk;
    int64_t b1 = b0 + chunk < n ? b0 + chunk : n;
    double mean = mode ? stats[0] : 0.0;
    double acc = 0.0;
    for (int64_t p = b0 + threadIdx.x; p < b1; p += NRM_THREADS) {
        double v = r[p];
        if (mode) {
            double d = v - mean;
            acc = acc + __dmul_rn(d, d);
        } else {
            acc = acc + v;
        }
    }
    double t = block_sum_d(acc, s);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void __launch_bounds__(NRM_BLOCKS) k_stats_final(int64_t n, int mode, double* stats,
                                                            const double* partial) {
    __shared__ double s[NRM_BLOCKS];
    double t = block_sum_d(partial[threadIdx.x], s);
    if (threadIdx.x == 0) {
        if (mode == 0) stats[0] = n > 0 ? t / (double)n : 0.0;
        else stats[1] = n > 0 ? sqrt(t / (double)n) : 0.0;
    }
}

// z = (r - mean) / sd in FP64 (0 for a constant series); bits[i] = z > cutoff
// (uncapped) when bits is given; then the cap z = min(max(z, -clip), clip)
// (clip = +inf when off) before the FP32 rounding or the int8 code.
__global__ void k_normalise_f32(const double* __restrict__ r, int64_t n, const double* stats,
                                double clip, double cutoff, int8_t* __restrict__ bits,
                                float* __restrict__ z) {
    double mean = stats[0], sd = stats[1];
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double v = sd > 0.0 ? __ddiv_rn(r[i] - mean, sd) : 0.0;
        if (bits) bits[i] = v > cutoff ? 1 : 0;
        v = fmin(fmax(v, -clip), clip);
        z[i] = __double2float_rn(v);
    }
}

__global__ void k_normalise_i8(const double* __restrict__ r, int64_t n, const double* stats,
                               double clip, double cutoff, int8_t* __restrict__ bits,
                               int8_t* __restrict__ q) {
    double mean = stats[0], sd = stats[1];
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        double v = sd > 0.0 ? __ddiv_rn(r[i] - mean, sd) : 0.0;
        if (bits) bits[i] = v > cutoff ? 1 : 0;
        v = fmin(fmax(v, -clip), clip);
        double c = rint(16.0 * v);
        c = c > 127.0 ? 127.0 : (c < -127.0 ? -127.0 : c);
        q[i] = (int8_t)(int)c;
    }
}

ffa_status launch_normalise(const double* d_resid, int64_t n, int32_t precision, void* d_out,
                            double* d_stats, cudaStream_t st, float clip, float cutoff,
                            int8_t* d_bits) {
    if (n <= 0) return FFA_OK;
    const double cl = clip > 0.0f ? (double)clip : INFINITY;
    double* partial = d_stats + 2;
    k_stats_partial<<<NRM_BLOCKS, NRM_THREADS, 0, st>>>(d_resid, n, d_stats, 0, partial);
    k_stats_final<<<1, NRM_BLOCKS, 0, st>>>(n, 0, d_stats, partial);
    k_stats_partial<<<NRM_BLOCKS, NRM_THREADS, 0, st>>>(d_resid, n, d_stats, 1, partial);
    k_stats_final<<<1, NRM_BLOCKS, 0, st>>>(n, 1, d_stats, partial);
    if (precision == FFA_FOLD_F32)
        k_normalise_f32<<<grid_for(n, 256), 256, 0, st>>>(d_resid, n, d_stats, cl, (double)cutoff,
                                                          d_bits, (float*)d_out);
    else
        k_normalise_i8<<<grid_for(n, 256), 256, 0, st>>>(d_resid, n, d_stats, cl, (double)cutoff,
                                                         d_bits, (int8_t*)d_out);
    FFA_LAUNCH_CHECK("k_normalise");
    count_launch(5);
    return FFA_OK;
}

}  // namespace ffa
