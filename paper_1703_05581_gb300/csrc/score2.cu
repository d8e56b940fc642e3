// Algorithm 2 (Section 2.2.2, Eq. 5) on the GPU, one CTA per folded profile
// at a time (persistent over trials), with the last FFA stage (Section 2.1)
// fused into the load; and the host parts both scorers share.
//
// The profile x (p0 bins) is extended cyclically to p0 + wmax bins and cut
// into blocks of R consecutive bins; thread t owns block t in registers.
// With the in-block exclusive prefix c_t[o] (FP32) and the block offsets
// Cb[t] = sum of earlier blocks (float-float), the cyclic box sum of width w
// starting at bin j is the difference of two prefixes.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "score.cuh"

namespace ffa {

namespace {

// CTA shapes.  A profile of p0 bins is cut into blocks of R bins, one per
// thread; T * R >= p0.  Long profiles take 1024-thread CTAs, one per SM;
// short ones smaller CTAs, several per SM, each on its own profile.  The
// shape is the first of 256 x 8, 512 x 16, 1024 x 16, 1024 x 32 that fits.
template <int TH>
struct Cfg;
template <>
struct Cfg<1024> {
    static constexpr int T = 1024, R = 32, MAXB = 2048, NBK = 2048, CAPM = 1024, MINB = 1;
};
template <>
struct Cfg<512> {
    static constexpr int T = 512, R = 16, MAXB = 1024, NBK = 1024, CAPM = 512, MINB = 2;
};
template <>
struct Cfg<256> {
    static constexpr int T = 256, R = 8, MAXB = 512, NBK = 512, CAPM = 512, MINB = 4;
};
// 1024 threads of 16 bins: profiles of 8193..16384 bins, which would leave
// half or more of a 1024 x 32 CTA idle
struct CMid {
    static constexpr int T = 1024, R = 16, MAXB = 2048, NBK = 2048, CAPM = 1024, MINB = 1;
};
using CBig = Cfg<1024>;

#define FFA_CFG_ALIASES                                   \
    constexpr int T2 = C::T, R2 = C::R, MAXB = C::MAXB;   \
    constexpr int NBK = C::NBK, CAPM = C::CAPM;           \
    constexpr int NW = T2 / 32;                           \
    (void)T2; (void)R2; (void)MAXB; (void)NBK; (void)CAPM; (void)NW;

// Shared-memory index of bin t: 4 pad words per 32-bin block keep every block
// 16-byte aligned (vector loads) and spread blocked accesses over the banks.
__device__ __forceinline__ int sidx(int t) { return t + 4 * (t >> 5); }

template <class C>
struct Sh2 {
    uint32_t hist[C::NBK];
    unsigned long long cand[C::CAPM];  // order-preserving keys of the candidates
    float candf[C::CAPM];    // gathered values; FP64 is applied per candidate afterwards
    double bw_max[16];       // per-width block maxima
    float cbh[C::MAXB + 1];  // block offsets (hi) / int offsets reinterpreted
    float cbl[C::MAXB + 1];  // block offsets (lo)
    float wred[16][32];   // per-width warp maxima (float profiles)
    int wredi[16][32];    // per-width warp maxima (int profiles)
    float fred[32];
    double dred[64];
    int ired[32];
    int ired2[C::CAPM];      // gathered int values
    unsigned long long ukey[2];
    uint32_t cnt, below;
    float mthr[4];  // MAD bracket: |x - med| <= D1 <=> mthr[0] <= x <= mthr[1]; D2: mthr[2], mthr[3]
    long long mthri[4];  // the same bounds for int profiles
    int mok;
    // Per-profile FP64 scalars, computed by one thread and broadcast: FP64
    // issues at a small fraction of the FP32 rate on this part, so a value
    // every thread needs is never recomputed by every thread.
    double smed, skmad;        // median, K * MAD
    float snr_mh, snr_ml, snr_kf;  // float S/N: median as a float pair, fl(K * MAD)
    int madpos;                // MAD > 0
    float bw_maxf[16];         // per-width block maxima (float profiles)
    int bin_a, bin_b;
    uint32_t below_a, below_b;
    uint32_t wkey[16];  // per-width maxima as order-preserving keys (item-distributed widths)
    int phase;
};

// ---- block helpers (T2 threads) --------------------------------------------
__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// block sums of a and b and the max of c (one barrier pair)
template <class C>
__device__ void blk_stats(float& a, float& b, float& c, Sh2<C>& sh) {
    FFA_CFG_ALIASES
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_max(c);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        sh.fred[w] = a;
        sh.wred[0][w] = b;
        sh.wred[1][w] = c;
    }
    __syncthreads();
    a = warp_sum(l < NW ? sh.fred[l] : 0.0f);
    b = warp_sum(l < NW ? sh.wred[0][l] : 0.0f);
    c = warp_max(l < NW ? sh.wred[1][l] : 0.0f);
    __syncthreads();
}
// exclusive scan of one uint32 per thread
template <class C>
__device__ uint32_t blk_exscan_u(uint32_t v, Sh2<C>& sh, uint32_t* total) {
    FFA_CFG_ALIASES
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    uint32_t* s = reinterpret_cast<uint32_t*>(sh.ired);
    if (lane == 31) s[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t y = lane < NW ? s[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
        s[lane] = y;
    }
    __syncthreads();
    uint32_t r = (warp ? s[warp - 1] : 0u) + x - v;
    if (total) *total = s[NW - 1];
    __syncthreads();
    return r;
}

// exclusive scan of float-float values (hi, lo) in block order
__device__ __forceinline__ void ff_add(float ah, float al, float bh, float bl, float& sh_, float& sl_) {
    float s, e;
    two_sum(ah, bh, s, e);
    e = __fadd_rn(e, __fadd_rn(al, bl));
    float s2 = __fadd_rn(s, e);
    sl_ = __fsub_rn(e, __fsub_rn(s2, s));
    sh_ = s2;
}

template <class C>
__device__ void blk_exscan_ff(float vh, Sh2<C>& sh, float& oh, float& ol, float& th, float& tl) {
    FFA_CFG_ALIASES
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float xh = vh, xl = 0.0f;
    for (int o = 1; o < 32; o <<= 1) {
        float uh = __shfl_up_sync(0xffffffffu, xh, o);
        float ul = __shfl_up_sync(0xffffffffu, xl, o);
        if (lane >= o) ff_add(xh, xl, uh, ul, xh, xl);
    }
    // inclusive warp result in (xh, xl)
    if (lane == 31) {
        sh.fred[warp] = xh;
        sh.wred[0][warp] = xl;
    }
    __syncthreads();
    if (warp == 0) {
        float yh = lane < NW ? sh.fred[lane] : 0.0f, yl = lane < NW ? sh.wred[0][lane] : 0.0f;
        for (int o = 1; o < 32; o <<= 1) {
            float uh = __shfl_up_sync(0xffffffffu, yh, o);
            float ul = __shfl_up_sync(0xffffffffu, yl, o);
            if (lane >= o) ff_add(yh, yl, uh, ul, yh, yl);
        }
        sh.fred[lane] = yh;
        sh.wred[0][lane] = yl;
    }
    __syncthreads();
    float bh = warp ? sh.fred[warp - 1] : 0.0f, bl = warp ? sh.wred[0][warp - 1] : 0.0f;
    // exclusive = base + inclusive - own  ->  compute base + (inclusive warp prefix excluding own)
    float eh, el;
    {
        float ph = __shfl_up_sync(0xffffffffu, xh, 1), pl = __shfl_up_sync(0xffffffffu, xl, 1);
        if (lane == 0) {
            ph = 0.0f;
            pl = 0.0f;
        }
        ff_add(bh, bl, ph, pl, eh, el);
    }
    oh = eh;
    ol = el;
    th = sh.fred[NW - 1];
    tl = sh.wred[0][NW - 1];
    __syncthreads();
}

template <class T>
struct Traits;
template <>
struct Traits<float> {
    static constexpr bool is_int = false;
};
template <>
struct Traits<int32_t> {
    static constexpr bool is_int = true;
};

}  // namespace

// Box-sum helpers.  C(32t + o) = Cb[t] + c_t[o]; a box of width w at bin
// 32t + r is C(32t + r + w) - C(32t + r).
template <class T>
struct BoxOps;
template <>
struct BoxOps<float> {
    template <class C>
    static __device__ __forceinline__ float blockdiff(const Sh2<C>& sh, int b2, int b1) {
        return __fadd_rn(__fsub_rn(sh.cbh[b2], sh.cbh[b1]), __fsub_rn(sh.cbl[b2], sh.cbl[b1]));
    }
    static __device__ __forceinline__ float box(float D, float c2, float c1) {
        return __fadd_rn(D, __fsub_rn(c2, c1));
    }
    static __device__ __forceinline__ float diff(float c2, float c1) { return __fsub_rn(c2, c1); }
    static __device__ __forceinline__ float lowest() { return -INFINITY; }
};
template <>
struct BoxOps<int32_t> {
    template <class C>
    static __device__ __forceinline__ int32_t blockdiff(const Sh2<C>& sh, int b2, int b1) {
        const int* cbi = reinterpret_cast<const int*>(sh.cbh);
        return (int32_t)((uint32_t)cbi[b2] - (uint32_t)cbi[b1]);
    }
    static __device__ __forceinline__ int32_t box(int32_t D, int32_t c2, int32_t c1) {
        return (int32_t)((uint32_t)D + ((uint32_t)c2 - (uint32_t)c1));
    }
    static __device__ __forceinline__ int32_t diff(int32_t c2, int32_t c1) {
        return (int32_t)((uint32_t)c2 - (uint32_t)c1);
    }
    static __device__ __forceinline__ int32_t lowest() { return INT32_MIN; }
};

// ---------------------------------------------------------------------------
// Algorithm 2 (Section 2.2.2, Eq. 5): boxcar first, then for each width the
// maximum I_max (first position j*), an exclusion window of the 2h+1 profile
// bins within cyclic distance h of the box's centre (j* + w/2) mod p0, and
// A_w = (I_max - w I_av) / (sigma sqrt(w)) with I_av and sigma the mean and
// population standard deviation of the other, unfiltered, profile bins;
// score = max over widths.  The profile's sum of squares about its mean is
// taken once; per width only the window's share is summed (its raw bins
// recovered as differences of the in-block prefix) and subtracted.  FP64
// per width, by one thread.
// ---------------------------------------------------------------------------
template <class T, class C>
__device__ __forceinline__ T box_at(const T (&c)[C::R], const Sh2<C>& sh, const T* buf, int tid, int w, int r) {
    FFA_CFG_ALIASES
    using B = BoxOps<T>;
    // cyclic box of width w starting at bin 32 tid + r, from the blocked prefix
    const int j2 = tid * R2 + r + w;
    const int b2 = j2 / R2, o2 = j2 % R2;
    return B::box(B::blockdiff(sh, b2, tid), buf[sidx(b2 * R2 + o2)], c[r]);
}

template <class C, class T, bool FUSED>
__global__ void __launch_bounds__(C::T, C::MINB) k_score_alg2(const T* __restrict__ prof_all, const ScoreGroup sg,
                                                              int64_t m_rows, int64_t trial0, int64_t count,
                                                              ScoreWidths wd, float excl_frac) {
    FFA_CFG_ALIASES
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Sh2<C>& sh = *reinterpret_cast<Sh2<C>*>(smem_raw);
    T* buf = reinterpret_cast<T*>(smem_raw + ((sizeof(Sh2<C>) + 15) & ~(size_t)15));
    using B = BoxOps<T>;
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int wmax = wd.w[wd.n - 1];
    for (int64_t it = blockIdx.x; it < count; it += gridDim.x) {
        const int ei = score_entry(sg, it);
        const int64_t p0_ = sg.p0[ei];
        const int p0 = (int)p0_;
        const T* __restrict__ prof = prof_all + sg.off[ei];
        const int nbe = (p0 + wmax + R2) / R2 + 1;
        const int h = (int)floorf(excl_frac * (float)p0 / 2.0f);
        const int n_off = p0 - min(p0, 2 * h + 1);
        const int64_t k = trial0 + (it - sg.t0[ei]);
        const T* hrow;
        const T* trow = nullptr;
        int sft = 0;
        const int64_t ld_ = sg.ld[ei];
        if (FUSED && m_rows > 1) {
            hrow = prof + (k >> 1) * ld_;
            trow = prof + ((m_rows >> 1) + (k >> 1)) * ld_;
            sft = (int)(((k + 1) >> 1) % p0_);
        } else if (FUSED) {
            hrow = prof;
        } else {
            hrow = prof + k * ld_;
        }
        if (trow) {
            const int n1 = p0 - sft;
            for (int j = tid; j < p0; j += T2) buf[sidx(j)] = hrow[j] + (j < n1 ? trow[j + sft] : trow[j - n1]);
        } else {
            for (int j = tid; j < p0; j += T2) buf[sidx(j)] = hrow[j];
        }
        __syncthreads();
        T x[R2];
        const int base_pos = tid * R2;
        int nvalid = p0 - base_pos;
        nvalid = nvalid < 0 ? 0 : (nvalid > R2 ? R2 : nvalid);
        float fs = 0.0f, fq = 0.0f, fm = 0.0f;
#pragma unroll
        for (int r = 0; r < R2; ++r) {
            x[r] = (r < nvalid) ? buf[sidx(base_pos + r)] : (T)0;
            if (r < nvalid) fs += (float)x[r];
        }
        blk_stats(fs, fq, fm, sh);
        const float mean = fs / (float)p0;
        // the whole profile's sums of (x - mean) and (x - mean)^2
        float ps = 0.0f, pq = 0.0f, pm = 0.0f;
#pragma unroll
        for (int r = 0; r < R2; ++r)
            if (r < nvalid) {
                const float d = (float)x[r] - mean;
                ps += d;
                pq = fmaf(d, d, pq);
            }
        blk_stats(ps, pq, pm, sh);
        // blocked cyclic prefix (as in k_score2)
        const bool one_wrap = nbe * R2 <= 2 * p0;
        const int eb2 = tid + T2;
        T tot = 0, tot2 = 0;
        if (eb2 < nbe) {
            for (int r = 0; r < R2; ++r) {
                const int j = eb2 * R2 + r;
                const T v = buf[sidx(one_wrap ? j - p0 : j % p0)];
                buf[sidx(j)] = tot2;
                tot2 = tot2 + v;
            }
        }
#pragma unroll
        for (int r = 0; r < R2; ++r) {
            const int j = base_pos + r;
            T v = x[r];
            if (j >= p0) v = (tid < nbe) ? buf[sidx(one_wrap ? j - p0 : j % p0)] : (T)0;
            x[r] = tot;
            tot = tot + v;
        }
        __syncthreads();
        {
            T* blk = buf + sidx(base_pos);
#pragma unroll
            for (int r = 0; r < R2; r += 4) *reinterpret_cast<int4*>(blk + r) = *reinterpret_cast<const int4*>(&x[r]);
        }
        if constexpr (Traits<T>::is_int) {
            uint32_t t0, t1;
            const uint32_t ex0 = blk_exscan_u((uint32_t)tot, sh, &t0);
            int* cbi = reinterpret_cast<int*>(sh.cbh);
            cbi[tid] = (int)ex0;
            if (nbe > T2) {
                const uint32_t ex1 = blk_exscan_u(eb2 < nbe ? (uint32_t)tot2 : 0u, sh, &t1);
                if (eb2 <= MAXB) cbi[eb2] = (int)(t0 + ex1);
            } else if (tid == 0) {
                cbi[T2] = (int)t0;
            }
        } else {
            float oh, ol, th, tl, oh2, ol2, th2, tl2;
            blk_exscan_ff((float)tot, sh, oh, ol, th, tl);
            sh.cbh[tid] = oh;
            sh.cbl[tid] = ol;
            if (nbe > T2) {
                blk_exscan_ff(eb2 < nbe ? (float)tot2 : 0.0f, sh, oh2, ol2, th2, tl2);
                if (eb2 <= MAXB) {
                    float hh, ll;
                    ff_add(th, tl, oh2, ol2, hh, ll);
                    sh.cbh[eb2] = hh;
                    sh.cbl[eb2] = ll;
                }
            } else if (tid == 0) {
                sh.cbh[T2] = th;
                sh.cbl[T2] = tl;
            }
        }
        __syncthreads();
        double best = -INFINITY;
        int best_w = 0, best_j = 0;
        for (int wi = 0; wi < wd.n; ++wi) {
            const int w = wd.w[wi];
            T m = B::lowest();
            int mpos = 0x7fffffff;
            if (nvalid > 0) {
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    if (r < nvalid) {
                        const T bx = box_at(x, sh, buf, tid, w, r);
                        if (bx > m) {
                            m = bx;
                            mpos = base_pos + r;
                        }
                    }
                }
            }
            // block: max with its first position
            float mf = (float)m;
            for (int o = 16; o > 0; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, mf, o);
                const int op = __shfl_xor_sync(0xffffffffu, mpos, o);
                if (om > mf || (om == mf && op < mpos)) {
                    mf = om;
                    mpos = op;
                }
            }
            __syncthreads();
            if (lane == 0) {
                sh.wred[0][warp] = mf;
                sh.wredi[0][warp] = mpos;
            }
            __syncthreads();
            mf = lane < NW ? sh.wred[0][lane] : -INFINITY;
            mpos = lane < NW ? sh.wredi[0][lane] : 0x7fffffff;
            for (int o = 16; o > 0; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, mf, o);
                const int op = __shfl_xor_sync(0xffffffffu, mpos, o);
                if (om > mf || (om == mf && op < mpos)) {
                    mf = om;
                    mpos = op;
                }
            }
            const int jstar = mpos;
            const int centre = (int)(((int64_t)jstar + w / 2) % p0);
            // sums of (x - mean) and its square over the window's profile bins;
            // bin r's value is the difference of the in-block prefix (the last
            // bin's: the block total minus the last prefix)
            float w1 = 0.0f, w2 = 0.0f;
            if (nvalid > 0) {
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const int j = base_pos + r;
                    int d = j - centre;
                    if (d < 0) d = -d;
                    d = min(d, p0 - d);
                    if (r < nvalid && d <= h) {
                        const T v = B::diff(r + 1 < R2 ? x[r + 1] : tot, x[r]);
                        const float dd = (float)v - mean;
                        w1 += dd;
                        w2 = fmaf(dd, dd, w2);
                    }
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                w1 += __shfl_xor_sync(0xffffffffu, w1, o);
                w2 += __shfl_xor_sync(0xffffffffu, w2, o);
            }
            __syncthreads();
            if (lane == 0) {
                sh.wred[3][warp] = w1;
                sh.wred[4][warp] = w2;
            }
            __syncthreads();
            w1 = lane < NW ? sh.wred[3][lane] : 0.0f;
            w2 = lane < NW ? sh.wred[4][lane] : 0.0f;
            for (int o = 16; o > 0; o >>= 1) {
                w1 += __shfl_xor_sync(0xffffffffu, w1, o);
                w2 += __shfl_xor_sync(0xffffffffu, w2, o);
            }
            if (tid == 0 && n_off >= 2) {  // only thread 0 keeps the score: FP64 once per width
                const double a1 = ((double)ps - (double)w1) / n_off;  // off-pulse mean - mean
                const double var = ((double)pq - (double)w2) / n_off - a1 * a1;
                const double sd = var > 0.0 ? sqrt(var) : 0.0;
                const double av = (double)mean + a1;
                if (sd > 0.0) {
                    const double a = ((double)mf - (double)w * av) / (sd * sqrt((double)w));
                    if (a > best) {
                        best = a;
                        best_w = wi;
                        best_j = jstar;
                    }
                }
            }
        }
        if (tid == 0) {
            ffa_record out;
            if (best == -INFINITY) {
                out.snr = 0.0f;
                out.width = wd.w[0];
                out.phase = 0;
                out.flags = 1;
            } else {
                out.snr = (float)best;
                out.width = wd.w[best_w];
                out.phase = best_j;
                out.flags = 0;
            }
            sg.rec[ei][it - sg.t0[ei]] = out;
        }
        __syncthreads();
    }
}

// Resident CTAs of a kernel for a dynamic shared-memory size, times the SM
// count, per device: queried once (launches come per base period).
ffa_status resident_ctas(const void* fn, int threads, size_t smem, int64_t* out) {
    static std::mutex mu;
    static std::map<std::tuple<const void*, size_t, int>, int64_t> cache;
    int dev = 0;
    FFA_CUDA_TRY(cudaGetDevice(&dev));
    const auto key = std::make_tuple(fn, smem, dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) {
            *out = it->second;
            return FFA_OK;
        }
    }
    int nsm = 0, per_sm = 0;
    FFA_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    FFA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem));
    const int64_t r = (int64_t)nsm * (per_sm < 1 ? 1 : per_sm);
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = r;
    *out = r;
    return FFA_OK;
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

namespace {

template <class C>
size_t score2_smem_bytes(int64_t p0, int wmax, size_t elem) {
    const int64_t nbe = (p0 + wmax + C::R) / C::R + 1;
    const int64_t nbins = (nbe > C::T ? nbe : C::T) * C::R + C::R;
    return ((sizeof(Sh2<C>) + 15) & ~(size_t)15) + (size_t)(nbins + 4 * (nbins / 32) + 64) * elem;
}

// does a profile of p0 bins with widths up to wmax fit configuration C?
template <class C>
bool fits(int64_t p0, int wmax) {
    return p0 >= 1 && (p0 + C::R - 1) / C::R <= C::T && (p0 + wmax + C::R) / C::R + 1 <= C::MAXB;
}

}  // namespace

// The scorer's CTA shape for a profile of p0 bins (0: 256 x 8, 1: 512 x 16,
// 2: 1024 x 16, 3: 1024 x 32); grouped launches hold one shape only, so a
// profile's record does not depend on what it is grouped with.
int score_shape(int64_t p0, int wmax) {
    if (fits<Cfg<256>>(p0, wmax)) return 0;
    if (fits<Cfg<512>>(p0, wmax)) return 1;
    if (fits<CMid>(p0, wmax)) return 2;
    return fits<CBig>(p0, wmax) ? 3 : -1;
}

namespace {

template <class C, class TT, bool FF>
ffa_status launch_alg2_cfg(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t p0,
                           int64_t m_rows, const ScoreWidths& wd, float excl_frac, ffa_record* d_rec,
                           cudaStream_t st) {
    const int wmax = wd.w[wd.n - 1];
    const size_t smem = score2_smem_bytes<C>(p0, wmax, 4);
    if (smem > 227 * 1024) return fail(FFA_ERR_UNSUPPORTED, "score: profile too long for shared memory");
    const void* fn = (const void*)k_score_alg2<C, TT, FF>;
    ffa_status es = ensure_smem(fn, smem);
    if (es != FFA_OK) return es;
    int64_t resident = 0;
    es = resident_ctas(fn, C::T, smem, &resident);
    if (es != FFA_OK) return es;
    const unsigned grid = (unsigned)(count < resident ? count : resident);
    (void)d_rec;  // the records go where sg.rec points
    k_score_alg2<C, TT, FF><<<grid, C::T, smem, st>>>((const TT*)d_prof, sg, m_rows, trial0, count, wd,
                                                      excl_frac);
    FFA_LAUNCH_CHECK("k_score_alg2");
    count_launch();
    return FFA_OK;
}

template <class TT, bool FF>
ffa_status launch_alg2_t(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t p0,
                         int64_t m_rows, const ScoreWidths& wd, float excl_frac, ffa_record* d_rec,
                         cudaStream_t st) {
    const int wmax = wd.w[wd.n - 1];
    if (fits<Cfg<256>>(p0, wmax))
        return launch_alg2_cfg<Cfg<256>, TT, FF>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, d_rec, st);
    if (fits<Cfg<512>>(p0, wmax))
        return launch_alg2_cfg<Cfg<512>, TT, FF>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, d_rec, st);
    if (fits<CMid>(p0, wmax))
        return launch_alg2_cfg<CMid, TT, FF>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, d_rec, st);
    return launch_alg2_cfg<CBig, TT, FF>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, d_rec, st);
}

ffa_status alg2_dispatch(const void* d_prof, const ScoreGroup& sg, int32_t precision, bool fused, int64_t count,
                         int64_t trial0, int64_t p0max, int64_t m_rows, const ScoreWidths& wd, float excl_frac,
                         ffa_record* d_rec, cudaStream_t st) {
    if (count <= 0) return FFA_OK;
    const int wmax = wd.w[wd.n - 1];
    if (!fits<CBig>(p0max, wmax)) return fail(FFA_ERR_UNSUPPORTED, "score: profile longer than 32768 bins");
    if (precision == FFA_FOLD_F32)
        return fused ? launch_alg2_t<float, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, d_rec, st)
                     : launch_alg2_t<float, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, d_rec, st);
    return fused ? launch_alg2_t<int32_t, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, d_rec, st)
                 : launch_alg2_t<int32_t, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, d_rec, st);
}

}  // namespace

ffa_status launch_score_alg2(const void* d_prof, int32_t precision, bool fused, int64_t count,
                             int64_t trial0, int64_t p0, int64_t ld, int64_t m_rows, const ScoreWidths& wd,
                             float excl_frac, ffa_record* d_rec, cudaStream_t st) {
    return alg2_dispatch(d_prof, score_single(p0, ld, count, d_rec), precision, fused, count, trial0, p0, m_rows, wd, excl_frac,
                         d_rec, st);
}

ffa_status launch_score_alg2_group(const void* d_plane, int32_t precision, int n, const int64_t* p0,
                                   const int64_t* off, int64_t m_rows, const ScoreWidths& wd, float excl_frac,
                                   ffa_record* const* recs, cudaStream_t st) {
    if (n < 1 || n > FOLD_GROUP_MAX) return fail(FFA_ERR_ARG, "score group: 1..FOLD_GROUP_MAX base periods");
    int64_t p0max = 0;
    const ScoreGroup sg = score_group(n, p0, off, m_rows, recs, &p0max);
    return alg2_dispatch(d_plane, sg, precision, true, (int64_t)n * m_rows, 0, p0max, m_rows, wd, excl_frac,
                         recs[0], st);
}

}  // namespace ffa
