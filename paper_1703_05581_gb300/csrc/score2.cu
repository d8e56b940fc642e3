// Algorithm 2 (Section 2.2.2, Eq. 5) on the GPU, one CTA per folded profile
// at a time (persistent over a run of consecutive trials), with the last FFA
// stage (Section 2.1) fused into the load.
//
// Boxcar first, then for each width the maximum I_max (first position j*), an
// exclusion window of the 2h+1 profile bins within cyclic distance h of the
// box's centre (j* + w/2) mod p0, and A_w = (I_max - w I_av) / (sigma sqrt(w))
// with I_av and sigma the mean and population standard deviation of the
// other, unfiltered, profile bins; score = max over widths.  The profile's
// sum of squares about its mean is taken once; per width only the window's
// share is summed (its raw bins recovered as differences of the in-block
// prefix) and subtracted.
//
// The layout, the blocked prefix and the box maxima are the Algorithm 1
// scorer's (score.cuh, score1.cu).  Every step takes all widths together --
// maxima, first positions, window sums, and the FP64 score with one lane per
// width -- so a profile costs about ten barriers and one FP64 chain, whatever
// the number of widths: 200 us for 4096 profiles of 4201 bins and 11 widths,
// 812 us with six barriers and a chain on one thread per width.  Sums over the profile keep one
// order: a lane sums a block, a warp 32 consecutive blocks (a "chunk"), and
// the chunks' sums are added as one more warp sum.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "score.cuh"

namespace ffa {

namespace {

struct S2Sh {
    float part[3][32];        // per chunk: sum, sum and sum of squares about the mean
    float2 win[16][32];       // per width and chunk: the window's sums
    float2 wtot[16];
    float2 seg[SCORE_MAXSEG]; // segment totals of the offset scan
    uint32_t wkey[16];        // largest box of width 2^n, as an order-preserving key of its float
    uint32_t pos[16];         // its first bin
};

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// tots: where the block totals start in dynamic shared memory; offs: the offsets
template <class V, int R, bool FUSED, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    k_score_alg2(const V* __restrict__ prof_all, const ScoreGroup sg, int64_t m_rows, int64_t trial0, int64_t count,
                 const ScoreWidths wd, uint32_t wmask, float excl_frac, uint32_t lay_offs, uint32_t lay_tots,
                 int group) {
    constexpr int PARTS = R < 16 ? 1 : R / 16;
    constexpr int NS = R == 8 ? 12 : 16;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ S2Sh sh;
    using Off = typename Offset<V>::type;
    Off* offs = reinterpret_cast<Off*>(smem + lay_offs);
    V* tots = reinterpret_cast<V*>(smem + lay_tots);
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = T >> 5;
    const int wmax = wd.w[wd.n - 1];
    const int64_t it_end = count * (int64_t)(blockIdx.x + 1) / gridDim.x;
    int64_t it = count * (int64_t)blockIdx.x / gridDim.x;
    int ei = it < it_end ? score_entry(sg, it) : 0;
    for (; it < it_end; ++it) {
        if (it >= sg.t0[ei + 1]) ++ei;
        const int p0 = sg.p0[ei];
        const int64_t ld = sg.ld[ei];
        const V* __restrict__ prof = prof_all + sg.off[ei];
        const int64_t k = trial0 + (it - sg.t0[ei]);
        const int nblk = (p0 + R - 1) / R, nfull = p0 / R, rem = p0 - nfull * R;
        const int nbx = nblk + (wmax > R ? wmax / R : 1);
        const int nchunk = (nblk + 31) >> 5;  // at most 32
        const int h = (int)floorf(excl_frac * (float)p0 / 2.0f);
        const int n_off = p0 - min(p0, 2 * h + 1);

        // ---- load (fused last FFA stage), cyclic extension, mean
        {
            const bool two = FUSED && m_rows > 1;
            const V* hrow = prof + (FUSED ? (k >> 1) * ld : k * ld);
            const V* trow = prof + ((m_rows >> 1) + (k >> 1)) * ld;  // two only
            const int sft = two ? (int)((uint32_t)((k + 1) >> 1) % (uint32_t)p0) : 0;
            load_profile<V, R>(smem, hrow, trow, sft, two, p0, tid, T, [](V) {});
        }
        if (tid < 16) {
            sh.wkey[tid] = 0u;
            sh.pos[tid] = 0x7fffffffu;
        }
        __syncthreads();
        extend_profile<V, R>(smem, p0, nbx, tid, T);
        for (int c = warp; c < nchunk; c += NW) {
            const int b = c * 32 + lane;
            const int nvalid = min(max(p0 - b * R, 0), R);
            const uint32_t a = blk_addr<R>((uint32_t)b);
            float fs = 0.0f;
            if (nvalid > 0) {
#pragma unroll
                for (int s = 0; s < R / 4; ++s) {
                    V v[4];
                    load_quad(smem, a ^ (s << 4), v);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (4 * s + i < nvalid) fs += (float)v[i];
                }
            }
            fs = warp_sum(fs);
            if (lane == 0) sh.part[0][c] = fs;
        }
        __syncthreads();
        const float mean = warp_sum(lane < nchunk ? sh.part[0][lane] : 0.0f) / (float)p0;
        // ---- sums of (x - mean) and (x - mean)^2; blocked cyclic prefix, in
        // place, with the block totals
        for (int c = warp; c * 32 < nbx; c += NW) {
            const int b = c * 32 + lane;
            const int nvalid = min(max(p0 - b * R, 0), R);
            const uint32_t a = blk_addr<R>((uint32_t)b);
            float ps = 0.0f, pq = 0.0f;
            if (b < nbx) {
                V t = 0;
#pragma unroll
                for (int s = 0; s < R / 4; ++s) {
                    V v[4], x[4];
                    load_quad(smem, a ^ (s << 4), v);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (4 * s + i < nvalid) {
                            const float d = (float)v[i] - mean;
                            ps += d;
                            pq = fmaf(d, d, pq);
                        }
                        x[i] = t;
                        t = t + v[i];
                    }
                    *reinterpret_cast<int4*>(smem + (a ^ (s << 4))) = *reinterpret_cast<const int4*>(x);
                }
                if constexpr (std::is_same<V, float>::value) offs[b].x = t;
                else offs[b] = t;
                if (b < nblk) tots[b] = t;
            }
            if (c < nchunk) {
                ps = warp_sum(ps);
                pq = warp_sum(pq);
                if (lane == 0) {
                    sh.part[1][c] = ps;
                    sh.part[2][c] = pq;
                }
            }
        }
        __syncthreads();
        scan_offsets<V, false>(offs, sh.seg, nbx, group);

        // ---- every width's largest box that starts in the profile (the
        // whole blocks' by items, the last block's bins one by one)
        V M[NS];
        const int nitem = nfull * PARTS;
        width_maxima<V, R, NS>(smem, offs, wmask, tid, T, nitem, M);
        {
            uint32_t wk = 0;
#pragma unroll
            for (int n = 0; n < NS; ++n) {
                const float m = (float)warp_max(M[n]);
                wk = lane == n ? fkey(m) : wk;
            }
            if (lane < 16 && (wmask >> lane & 1u)) atomicMax(&sh.wkey[lane], wk);
            for (int i = tid; i < rem * wd.n; i += T) {
                const int w = wd.w[i / rem];
                atomicMax(&sh.wkey[__ffs(w) - 1], fkey((float)box_at<V, R>(smem, offs, nfull * R + i % rem, w)));
            }
        }
        __syncthreads();
        // ---- its first position: the blocks of the threads that hold it, a
        // warp's lanes on the bins of 32 / R blocks at a time (a block's
        // maximum counts if it equals the width's as a float, at its first bin)
        for (int kw = 0; kw < wd.n; ++kw) {
            const int w = wd.w[kw], n = __ffs(w) - 1;
            const float top = fkey_inv(sh.wkey[n]);
            V own = box_lowest((V)0);
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (i == n) own = M[i];
            auto look = [&](int b, int nvalid) {  // lanes of one block: b and nvalid uniform in each R lanes
                const int r = lane % R, j = b * R + r;
                V bx = box_lowest((V)0);
                if (r < nvalid) bx = box_at<V, R>(smem, offs, j, w);
                V m = bx;
#pragma unroll
                for (int o = R / 2; o > 0; o >>= 1) {
                    const V u = __shfl_xor_sync(0xffffffffu, m, o);
                    m = u > m ? u : m;
                }
                uint32_t f = r < nvalid && bx == m && (float)m == top ? (uint32_t)j : 0x7fffffffu;
                f = __reduce_min_sync(0xffffffffu, f);
                if (lane == 0 && f != 0x7fffffffu) atomicMin(&sh.pos[n], f);
            };
            unsigned who = __ballot_sync(0xffffffffu, tid < nitem && (float)own == top);
            while (who) {
                const int src = warp * 32 + __ffs(who) - 1;
                who &= who - 1;
                const int nk = (nitem - src + T - 1) / T;
                for (int i0 = 0; i0 < nk; i0 += 32 / R) {
                    const int im = src + (i0 + lane / R) * T;
                    const bool on = im < nitem;
                    look(on ? im / PARTS : 0, on ? R : 0);
                }
            }
            if (rem && warp == kw % NW) look(nfull, lane < R ? rem : 0);
        }
        __syncthreads();
        // ---- sums of (x - mean) and its square over each width's window: bin
        // r's value is the difference of the in-block prefix (the last bin's:
        // the block total minus the last prefix)
        for (int p = warp; p < wd.n * nchunk; p += NW) {
            const int kw = p / nchunk, c = p - kw * nchunk;
            const int w = wd.w[kw];
            const int centre = (int)((sh.pos[__ffs(w) - 1] + (uint32_t)(w / 2)) % (uint32_t)p0);
            const int b = c * 32 + lane, j0 = b * R;
            const int nvalid = min(max(p0 - j0, 0), R);
            // cyclic distance to the centre: the block meets the window only
            // if one of its ends does or it holds the centre
            auto dist = [&](int j) {
                int d = j - centre;
                if (d < 0) d = -d;
                return min(d, p0 - d);
            };
            float w1 = 0.0f, w2 = 0.0f;
            const bool meets = nvalid > 0 && (dist(j0) <= h || dist(j0 + nvalid - 1) <= h ||
                                              (centre >= j0 && centre < j0 + nvalid));
            if (__ballot_sync(0xffffffffu, meets)) {
                if (meets) {
                    const uint32_t a = blk_addr<R>((uint32_t)b);
                    V x[4];
                    load_quad(smem, a, x);
                    const V tot = tots[b];
#pragma unroll
                    for (int s = 0; s < R / 4; ++s) {
                        V nx[4];
                        if (s + 1 < R / 4) load_quad(smem, a ^ ((s + 1) << 4), nx);
                        else nx[0] = tot;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int r = 4 * s + i;
                            if (r < nvalid && dist(j0 + r) <= h) {
                                const V v = box_sub(i < 3 ? x[i + 1] : nx[0], x[i]);
                                const float dd = (float)v - mean;
                                w1 += dd;
                                w2 = fmaf(dd, dd, w2);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) x[i] = nx[i];
                    }
                }
                w1 = warp_sum(w1);
                w2 = warp_sum(w2);
            }
            if (lane == 0) sh.win[kw][c] = make_float2(w1, w2);
        }
        __syncthreads();
        for (int kw = warp; kw < wd.n; kw += NW) {
            const float2 v = lane < nchunk ? sh.win[kw][lane] : make_float2(0.0f, 0.0f);
            const float w1 = warp_sum(v.x), w2 = warp_sum(v.y);
            if (lane == 0) sh.wtot[kw] = make_float2(w1, w2);
        }
        __syncthreads();
        // ---- the scores in FP64, one width per lane; the best, ties to the
        // smaller width
        if (warp == 0) {
            const float ps = warp_sum(lane < nchunk ? sh.part[1][lane] : 0.0f);
            const float pq = warp_sum(lane < nchunk ? sh.part[2][lane] : 0.0f);
            double a = -INFINITY;
            if (lane < wd.n && n_off >= 2) {
                const int w = wd.w[lane];
                const float w1 = sh.wtot[lane].x, w2 = sh.wtot[lane].y, mf = fkey_inv(sh.wkey[__ffs(w) - 1]);
                const double a1 = ((double)ps - (double)w1) / n_off;  // off-pulse mean - mean
                const double var = ((double)pq - (double)w2) / n_off - a1 * a1;
                const double sd = var > 0.0 ? sqrt(var) : 0.0;
                const double av = (double)mean + a1;
                if (sd > 0.0) a = ((double)mf - (double)w * av) / (sd * sqrt((double)w));
            }
            // as integer keys; a NaN never wins
            const uint64_t none = dkey(-INFINITY);
            uint64_t key = a == a ? dkey(a) : none;
            int best = lane;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t ok = __shfl_xor_sync(0xffffffffu, key, o);
                const int ob = __shfl_xor_sync(0xffffffffu, best, o);
                if (ok > key || (ok == key && ob < best)) {
                    key = ok;
                    best = ob;
                }
            }
            if (lane == 0) {
                ffa_record out;
                if (key == none) {
                    out.snr = 0.0f;
                    out.width = wd.w[0];
                    out.phase = 0;
                    out.flags = 1;
                } else {
                    out.snr = (float)dkey_inv(key);
                    out.width = wd.w[best];
                    out.phase = (int32_t)sh.pos[__ffs(wd.w[best]) - 1];
                    out.flags = 0;
                }
                sg.rec[ei][it - sg.t0[ei]] = out;
            }
        }
        __syncthreads();
    }
}

template <class V, int R, bool FF, int MAXT, int MINB>
ffa_status alg2_launch(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t p0,
                       int64_t m_rows, const ScoreWidths& wd, float excl_frac, cudaStream_t st) {
    uint32_t wmask = 0;
    for (int i = 0; i < wd.n; ++i) wmask |= (uint32_t)wd.w[i];
    const int wmax = wd.w[wd.n - 1];
    const int64_t nblk = (p0 + R - 1) / R, nbx = nblk + (wmax > R ? wmax / R : 1);
    const size_t offs = (size_t)nbx * R * 4;
    const size_t tots = offs + (((size_t)nbx * sizeof(typename Offset<V>::type) + 15) & ~(size_t)15);
    const size_t smem = tots + (size_t)nblk * 4;
    if (smem + sizeof(S2Sh) > 227 * 1024) return fail(FFA_ERR_UNSUPPORTED, "score: profile too long for shared memory");
    // three chunks of 32 blocks a warp (two at 32 bins a block): several
    // profiles per SM hide one another's barriers
    const int nchunk = (int)((nblk + 31) / 32), per = R == 32 ? 2 : 3;
    int threads = 32 * ((nchunk + per - 1) / per);
    threads = threads < 64 ? 64 : (threads > MAXT ? MAXT : threads);
    const void* fn = (const void*)k_score_alg2<V, R, FF, MAXT, MINB>;
    ffa_status es = ensure_smem(fn, smem);
    if (es != FFA_OK) return es;
    int64_t resident = 0;  // persistent: every CTA resident
    es = resident_ctas(fn, threads, smem, &resident);
    if (es != FFA_OK) return es;
    const unsigned grid = (unsigned)(count < resident ? count : resident);
    k_score_alg2<V, R, FF, MAXT, MINB><<<grid, threads, smem, st>>>((const V*)d_prof, sg, m_rows, trial0, count, wd, wmask,
                                                                    excl_frac, (uint32_t)offs, (uint32_t)tots,
                                                                    score_scan_group(score_shape(p0, wmax)));
    FFA_LAUNCH_CHECK("k_score_alg2");
    count_launch();
    return FFA_OK;
}

template <class V, bool FF>
ffa_status alg2_t(const void* d_prof, const ScoreGroup& sg, int64_t count, int64_t trial0, int64_t p0, int64_t m_rows,
                  const ScoreWidths& wd, float excl_frac, cudaStream_t st) {
    switch (score_shape(p0, wd.w[wd.n - 1])) {
        case 0: return alg2_launch<V, 8, FF, 128, 8>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, st);
        case 1:
        case 2: return alg2_launch<V, 16, FF, 384, 2>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, st);
        case 3: return alg2_launch<V, 32, FF, 512, 1>(d_prof, sg, count, trial0, p0, m_rows, wd, excl_frac, st);
        default: return fail(FFA_ERR_UNSUPPORTED, "score: profile longer than 32768 bins");
    }
}

ffa_status alg2_dispatch(const void* d_prof, const ScoreGroup& sg, int32_t precision, bool fused, int64_t count,
                         int64_t trial0, int64_t p0max, int64_t m_rows, const ScoreWidths& wd, float excl_frac,
                         cudaStream_t st) {
    if (count <= 0) return FFA_OK;
    if (precision == FFA_FOLD_F32)
        return fused ? alg2_t<float, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, st)
                     : alg2_t<float, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, st);
    return fused ? alg2_t<int32_t, true>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, st)
                 : alg2_t<int32_t, false>(d_prof, sg, count, trial0, p0max, m_rows, wd, excl_frac, st);
}

}  // namespace

ffa_status launch_score_alg2(const void* d_prof, int32_t precision, bool fused, int64_t count, int64_t trial0,
                             int64_t p0, int64_t ld, int64_t m_rows, const ScoreWidths& wd, float excl_frac,
                             ffa_record* d_rec, cudaStream_t st) {
    return alg2_dispatch(d_prof, score_single(p0, ld, count, d_rec), precision, fused, count, trial0, p0, m_rows, wd,
                         excl_frac, st);
}

ffa_status launch_score_alg2_group(const void* d_plane, int32_t precision, int n, const int64_t* p0,
                                   const int64_t* off, int64_t m_rows, const ScoreWidths& wd, float excl_frac,
                                   ffa_record* const* recs, cudaStream_t st) {
    if (n < 1 || n > FOLD_GROUP_MAX) return fail(FFA_ERR_ARG, "score group: 1..FOLD_GROUP_MAX base periods");
    int64_t p0max = 0;
    const ScoreGroup sg = score_group(n, p0, off, m_rows, recs, &p0max);
    return alg2_dispatch(d_plane, sg, precision, true, (int64_t)n * m_rows, 0, p0max, m_rows, wd, excl_frac, st);
}

}  // namespace ffa
