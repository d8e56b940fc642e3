// The FFA fold on the GPU (Section 2.1).
//
// Recursion: output trial k of a block of 2^s rows is head[k>>1] plus
// tail[k>>1] read ceil(k/2) bins further on (cyclic).  Unrolled, row r of a
// 2^m-row block enters trial k with the cyclic shift
//     shift(r, k) = sum_l bit_(m-1-l)(r) * ceil((k >> l) / 2).
//
// Multi-stage passes.  After s stages the plane holds, for every group g of
// 2^s consecutive input rows, its 2^s partial trials at row g*2^s + kappa.
// A pass of q further stages combines blocks of 2^q groups.  For a fixed
// input trial kappa, output trial kappa*2^q + v of a block takes group u's
// partial trial kappa at the shift  kappa*u + shift_q(u, v)  where shift_q
// is the shift table of a 2^q-row block (because ceil((kappa*2^(q-l) +
// (v>>l))/2) = kappa*2^(q-l-1) + ceil((v>>l)/2) for l < q).  So each pass is
// a plain 2^q-row FFA whose input row u starts at column kappa*u: the same
// adds in the same tree as the recursion, hence bit-identical results.
//
// A CTA owns (block, kappa, column tile): it stages 2^q rows of B + 2^q - 1
// columns (the halo covers the local shifts) in shared memory, runs the q
// local stages in registers (two register-blocked sub-passes) and writes 2^q
// rows of B columns.  Planes inside a search have a row pitch padded to a
// multiple of 4 elements, so rows are 16-byte aligned for the staging copies
// and the 128-bit output stores.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "internal.h"

namespace ffa {


// Base periods folded by one launch: an entry has p0 bins, m_data data rows
// (all share m_rows), its plane at element offset `off` of the plane buffers
// with row pitch ld (>= p0; a multiple of 4 makes every row 16-byte aligned),
// its rows cut into n_ct column tiles, and owns the launch's CTAs from unit0 to
// the next entry's.  A single base period is a group of one.  The first pass
// reads the series itself: row g of an entry is src[g * p0 ...], densely
// packed (entries of a batch read their own series).  An entry's fields lie
// together: a CTA starts with one or two lines of kernel parameters.
struct FoldEntry {
    const void* src;
    int64_t p0, m_data, off, ld;
    uint32_t unit0;
    int32_t n_ct;
};
struct alignas(64) FoldGroup {
    FoldEntry e[FOLD_GROUP_MAX];
    int32_t n;
};

// this CTA's entry
__device__ __forceinline__ int group_entry(const FoldGroup& g, int n, uint32_t unit) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.e[mid].unit0 <= unit) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <class T>
struct FoldIn;
template <>
struct FoldIn<float> { using type = float; };
template <>
struct FoldIn<int32_t> { using type = int8_t; };

// Asynchronous global -> shared copies (cp.async): a lane issues all of its
// copies for a tile without waiting, then waits once (cp_async_wait).  The
// 16-byte form bypasses L1 (each element is read by one tile only, apart from
// the halo, which the next tile finds in L2).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Stage `wt` cyclic columns of a row starting at column `base` (< p0) into
// shared memory at rowp[off ...] (one warp per row), element by element: the
// rows that wrap past p0, that do not start at alignment `off`, or that are
// shorter than the segment.
template <class T, class S>
__device__ __forceinline__ void stage_elements(T* __restrict__ rowp, const S* __restrict__ row, int64_t base,
                                               int64_t p0, int wt, int lane) {
    int64_t col = base + lane;
    while (col >= p0) col -= p0;
    for (int x = lane; x < wt; x += 32) {
        if constexpr (sizeof(T) == sizeof(S)) cp_async4(rowp + x, row + col);
        else rowp[x] = (T)row[col];
        col += 32;
        while (col >= p0) col -= p0;
    }
}

// ---------------------------------------------------------------------------
// The FFA of R = 2^QQ rows on W = 4 + R - 1 consecutive columns held in
// registers (compile-time shifts): out[v][0..3] is trial v at the first four
// columns.  load() reads a row's W values starting at the compile-time
// element offset OFF of a 16-byte aligned pointer, in 128-bit loads.
// ---------------------------------------------------------------------------
template <class T, int QQ>
struct RegFFA {
    static constexpr int R = 1 << QQ;
    static constexpr int W = 4 + R - 1;
    template <int OFF>
    static __device__ __forceinline__ void load(const T* p, T (&a)[W]) {
        constexpr int NV = (OFF + W + 3) / 4;
        T r[4 * NV];
#pragma unroll
        for (int k = 0; k < NV; ++k)
            *reinterpret_cast<int4*>(&r[4 * k]) = *reinterpret_cast<const int4*>(p + 4 * k);
#pragma unroll
        for (int k = 0; k < W; ++k) a[k] = r[k + OFF];
    }
    // rows u = 0 .. R-1, row u at p + u * pitch + (k * u & ~3), its values at
    // offset (TT * u) & 3 (TT = k & 3)
    template <int TT, size_t... U>
    static __device__ __forceinline__ void load_rows(const T* p, int pitch, int k, T (&a)[R][W],
                                                     std::index_sequence<U...>) {
        (load<(TT * (int)U) & 3>(p + (int)U * pitch + ((k * (int)U) & ~3), a[U]), ...);
    }
    static __device__ __forceinline__ void run(T (&a)[R][W], T (&out)[R][4]) {
#pragma unroll
        for (int t = 1; t <= QQ; ++t) {
            const int g = 1 << t, half = g >> 1;
            T b[R][W];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int gb = r & ~(g - 1), v = r - gb;
                const int hr = gb + (v >> 1), tr = gb + half + (v >> 1), sf = (v + 1) >> 1;
#pragma unroll
                for (int x = 0; x < W; ++x)
                    if (x + g - 1 < W) b[r][x] = a[hr][x] + a[tr][x + sf];
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int x = 0; x < W; ++x) a[r][x] = b[r][x];
        }
#pragma unroll
        for (int v = 0; v < R; ++v)
#pragma unroll
            for (int x = 0; x < 4; ++x) out[v][x] = a[v][x];
    }
};

template <class T>
__device__ __forceinline__ int as_bits(T v) {
    if constexpr (sizeof(T) == 4 && !std::is_integral<T>::value) return __float_as_int(v);
    else return (int)v;
}

// Four consecutive outputs to global memory: one 128-bit store when the row
// is 16-byte aligned (vec; what lies behind its end is padding), else element
// stores of columns [skip, left).
template <class T>
__device__ __forceinline__ void store4(T* d, const T (&v)[4], int left, bool vec, int skip = 0) {
    if (vec) {
        *reinterpret_cast<int4*>(d) = make_int4(as_bits(v[0]), as_bits(v[1]), as_bits(v[2]), as_bits(v[3]));
    } else {
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (x >= skip && x < left) d[x] = v[x];
    }
}

// A warp's 128 consecutive outputs (four per lane) to a row that is not
// 16-byte aligned, off elements past such a boundary: every lane but the first
// stores the aligned quad that ends in its own values, with the lane before's
// last `off` in front, so that a sector is written once and not in four parts
// (dense, against
// element stores: int8 8192 x 1489 81 us, 88; 4096 x 19977 380 us, 442).
template <class T>
__device__ __forceinline__ void store_row(T* d, const T (&v)[4], int off) {
    const int lane = threadIdx.x & 31;
    const T u1 = __shfl_up_sync(0xffffffffu, v[1], 1);
    const T u2 = __shfl_up_sync(0xffffffffu, v[2], 1);
    const T u3 = __shfl_up_sync(0xffffffffu, v[3], 1);
    const int a = as_bits(off == 1 ? u3 : off == 2 ? u2 : u1), b = as_bits(off == 1 ? v[0] : off == 2 ? u3 : u2);
    const int c = as_bits(off == 1 ? v[1] : off == 2 ? v[0] : u3), e = as_bits(off == 1 ? v[2] : off == 2 ? v[1] : v[0]);
    if (lane > 0) {
        *reinterpret_cast<int4*>(d - off) = make_int4(a, b, c, e);
    } else {
#pragma unroll
        for (int x = 0; x < 3; ++x)
            if (x < 4 - off) d[x] = v[x];
    }
    if (lane == 31) {
#pragma unroll
        for (int x = 1; x < 4; ++x)
            if (x >= 4 - off) d[x] = v[x];
    }
}

// ---------------------------------------------------------------------------
// One pass of q = Q1 + Q2 <= 6 stages.  A CTA owns (block, kappa, column
// tile of B columns): it stages 2^q input rows of B + 2^q - 1 columns, row u
// starting at column c + kappa*u (cyclically), in shared memory.  Sub-pass 1:
// each thread takes 4 consecutive columns of a group of 2^Q1 rows, applies
// Q1 stages in registers and stores the group's 2^Q1 partial trials,
// unshifted, with 128-bit stores.  Sub-pass 2: for trial k1 of sub-pass 1,
// input row u2 of the last Q2 stages is read at column offset k1*u2 (the
// shift that the unrolled recursion assigns it), Q2 stages in registers, and
// the tile's output rows go to global memory (128-bit stores on a padded
// pitch).  Tiles are B = 256 columns up to 5 stages and 128 for 6 (64 rows).
//
// Alignment.  The staging copies are 16 bytes wide, so a row's columns keep
// the misalignment 0..3 of their address.  It is (t0 + t * u) & 3 in row u for
// one t0 and t per CTA -- the rows of the first pass are p0 elements apart (t =
// p0 & 3), row u of a later pass is (ld << s) elements on and starts kappa * u
// columns on (t = (kappa + (ld << s)) & 3) -- and so is the offset k1*u2 of
// sub-pass 2 (t = k1 & 3, one per warp).  The tile starts t0 columns early, so
// that t0 is 0, and both sub-passes are compiled for each t, with every row's
// offset known, and need no select on it.  Rows off that pattern (they wrapped
// past p0) are staged element by element onto it.  t0 is 0 on padded planes;
// on dense ones it is kappa * p0: without the early start three in four tiles
// of the later passes were staged by elements (256 x 2001: 8.3 us, 7.2; 4096 x
// 19977: 424 us, 380).  ALIGNED kernels, of planes where t0 is 0 and every row
// starts on such a boundary, leave all of it out.
//
// What bounds it.  4096 rows of 19977 bins: the six-stage first pass takes
// 150 us at 39 thread-instructions an element, its shared memory 73 % busy
// (234 us and 62 with two selects per value on each row's offset and 64-bit
// divisions for each row); the five-stage second pass 129 us, 4.7 TB/s of DRAM
// traffic (142 us before).
// ---------------------------------------------------------------------------
constexpr int FK_THREADS = 256;
// quads: rows off a boundary of four elements are stored as whole quads
// (store_row).  That code and the variants of sub-pass 2 do not fit the
// instruction cache of a short launch: it pays from about a CTA an SM on
// (32 x 2001: 5.7 us with it, 5.2 without).
// Six stages (3 + 3): sub-pass 1 works in place, a warp on each of the eight
// groups, so one buffer of 64 rows (50 KB) serves both sub-passes and four
// CTAs fit an SM, where two buffers left room for two: 4096 x 19977, first
// pass, 163 us with two CTAs that staged the next tile under sub-pass 2, 153
// in place with three, 149 with four; int8 4096 x 29 500: 230, 200, 181.
__host__ __device__ constexpr bool fk_inplace(int q1, int q2) { return q1 == 3 && q2 == 3; }
__host__ __device__ constexpr int fk_r4(int x) { return (x + 3) & ~3; }
__host__ __device__ constexpr int fk_max(int a, int b) { return a > b ? a : b; }
__host__ __device__ constexpr int fk_wt(int q, int b) { return b + (1 << q) - 1; }                  // staged columns
__host__ __device__ constexpr int fk_w1(int q, int q1, int b) { return b + (1 << q) - (1 << q1); }  // valid after sub-pass 1
// Row widths (elements) of the two shared buffers: room for the staging
// copies and for every 128-bit load of the two sub-passes.
__host__ __device__ constexpr int fk_wa(int q, int q1, int b) {
    return fk_max(fk_r4(fk_wt(q, b) + 3), 4 * ((fk_w1(q, q1, b) + 3) / 4 - 1) + 4 * ((4 + (1 << q1) - 1 + 6) / 4));
}
__host__ __device__ constexpr int fk_wb(int q, int q1, int b) {
    return fk_max(fk_r4(fk_w1(q, q1, b)), (b - 4) + 4 * ((((1 << q1) - 1) * ((1 << (q - q1)) - 1)) / 4) +
                                              4 * ((4 + (1 << (q - q1)) - 1 + 6) / 4));
}

template <class T, bool FIRST, int Q1, int Q2, int B, bool ALIGNED>
__global__ void __launch_bounds__(FK_THREADS, fk_inplace(Q1, Q2) ? 4 : ALIGNED ? 2 : 3) k_fold(const void* __restrict__ src_v, T* __restrict__ dst_all, int s, int n,
                                                       bool quads, const FoldGroup fg) {
    constexpr int q = Q1 + Q2;
    constexpr bool INPLACE = fk_inplace(Q1, Q2);
    constexpr int rows = 1 << q;
    constexpr int R1 = 1 << Q1, R2 = 1 << Q2;
    constexpr int WT = fk_wt(q, B), W1 = fk_w1(q, Q1, B);
    constexpr int WB = fk_wb(q, Q1, B), WA = INPLACE ? fk_max(fk_wa(q, Q1, B), WB) : fk_wa(q, Q1, B);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* bufA = reinterpret_cast<T*>(smem_raw);
    T* bufB = bufA + rows * WA;

    using S = typename std::conditional<FIRST, typename FoldIn<T>::type, T>::type;
    constexpr bool WIDEN = sizeof(S) == 1;  // int8 series
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NW = FK_THREADS / 32;
    constexpr int RPW = (rows + NW - 1) / NW;            // rows staged by a warp
    constexpr int KPL = ((WT + 6) / 4 + 31) / 32;        // aligned words per lane and row (WIDEN)

    struct Tile {
        int64_t p0, ld, blk, c;  // c: first column, -3 .. -1 in an early first tile
        uint32_t kappa;
        int ei, t;
    };
    auto source = [&](int ei) { return FIRST ? (const S*)fg.e[ei].src : (const S*)src_v + fg.e[ei].off; };
    auto locate = [&](uint32_t u) {
        Tile w;
        w.ei = group_entry(fg, n, u);
        w.p0 = fg.e[w.ei].p0;
        w.ld = fg.e[w.ei].ld;
        const uint32_t unit = u - fg.e[w.ei].unit0;
        const uint32_t n_ct = (uint32_t)fg.e[w.ei].n_ct;
        const uint32_t rest = unit / n_ct;
        w.kappa = rest & ((1u << s) - 1);
        w.blk = rest >> s;
        w.c = (int64_t)(unit - rest * n_ct) * B;
        w.t = (int)((FIRST ? (uint32_t)w.p0 : w.kappa) & 3);
        if constexpr (!ALIGNED) {
            // row 0's first element and the distance of rows, mod 4
            const uint32_t row0 = FIRST ? (rows % 4 ? (uint32_t)w.blk * rows * (uint32_t)w.p0 : 0u)
                                        : ((((uint32_t)w.blk * rows) << s) + w.kappa) * (uint32_t)w.ld;
            w.c -= ((uint32_t)(reinterpret_cast<uintptr_t>(source(w.ei)) / sizeof(S)) + row0) & 3;
            if (!FIRST) w.t = (int)((w.kappa + ((uint32_t)w.ld << s)) & 3);
        }
        return w;
    };
    uint32_t wv[WIDEN ? RPW : 1][KPL];  // WIDEN: the tile's words between issue and store
    int64_t my_row = 0, my_base = 0;
    int my_how = 0;
    auto row_how = [&](int j) { return __shfl_sync(0xffffffffu, my_how, j); };
    auto row_base = [&](int j) { return __shfl_sync(0xffffffffu, my_base, j); };
    // Start staging a tile.  cp.async copies straight into bufA; the words of
    // an int8 series (cp.async cannot widen) are loaded into registers, every
    // row's before any is needed.
    auto stage_issue = [&](const Tile& w) {
        // lane j: where row warp + j * NW starts, and how it is staged (0:
        // beyond the data, zeros; 1: 16-byte copies; 2: element by element)
        const S* __restrict__ src = source(w.ei);
        my_how = 0;
        {
            const int u = warp + lane * NW;
            if (lane < RPW && u < rows) {
                const int64_t g = w.blk * rows + u;
                const int64_t c = !ALIGNED && w.c < 0 ? w.c + 4 * w.p0 : w.c;
                if (w.p0 < (1 << 25))
                    my_base = ((uint32_t)c + (w.kappa % (uint32_t)w.p0) * (uint32_t)u) % (uint32_t)w.p0;
                else
                    my_base = (c + (int64_t)w.kappa * u) % w.p0;
                my_row = FIRST ? g * w.p0 : ((g << s) + w.kappa) * w.ld;
                const uintptr_t a = reinterpret_cast<uintptr_t>(src + my_row + my_base) / sizeof(S);
                if (!FIRST || g < fg.e[w.ei].m_data) my_how = my_base + WT <= w.p0 && (a & 3) == ((w.t * u) & 3) ? 1 : 2;
            }
        }
#pragma unroll
        for (int j = 0; j < RPW; ++j) {
            const int u = warp + j * NW, off = (w.t * u) & 3;
            if (u >= rows) break;
            T* rowp = bufA + u * WA;
            const int how = row_how(j);
            const S* rp = src + __shfl_sync(0xffffffffu, my_row, j);
            const int64_t base = row_base(j);
            if (how == 1) {
                // from the aligned-down start; the chunk (word) holding the
                // segment's last element ends within that element's 16-byte
                // (4-byte) block
                const S* g0 = rp + base - off;
                const int nc = (WT + off + 3) >> 2;
                if constexpr (WIDEN) {
#pragma unroll
                    for (int i = 0; i < KPL; ++i) {
                        const int k = lane + 32 * i;
                        wv[j][i] = k < nc ? __ldg(reinterpret_cast<const uint32_t*>(g0) + k) : 0u;
                    }
                } else {
                    for (int k = lane; k < nc; k += 32) cp_async16(rowp + 4 * k, g0 + 4 * k);
                }
            } else if (how == 2) {
                stage_elements(rowp + off, rp, base, w.p0, WT, lane);
            } else {
                for (int x = 4 * lane; x < WT + 3; x += 128) *reinterpret_cast<int4*>(rowp + x) = make_int4(0, 0, 0, 0);
            }
        }
    };
    // Finish it: bufA holds the tile after the next barrier.
    auto stage_finish = [&](int t) {
        if constexpr (WIDEN) {
#pragma unroll
            for (int j = 0; j < RPW; ++j) {
                const int u = warp + j * NW, off = (t * u) & 3;
                if (u >= rows) break;
                if (row_how(j) != 1) continue;
                const int nc = (WT + off + 3) >> 2;
#pragma unroll
                for (int i = 0; i < KPL; ++i) {
                    const int k = lane + 32 * i;
                    const uint32_t v = wv[j][i];
                    if (k < nc)
                        *reinterpret_cast<int4*>(bufA + u * WA + 4 * k) = make_int4(
                            (int)(v << 24) >> 24, (int)(v << 16) >> 24, (int)(v << 8) >> 24, (int)v >> 24);
                }
            }
        } else {
            cp_async_wait();
        }
    };

    const Tile w = locate(blockIdx.x);
    if (!ALIGNED && w.c >= w.p0) return;  // (an early start may leave the last tile nothing)
    stage_issue(w);
    stage_finish(w.t);
    {
        __syncthreads();
        T* __restrict__ dst = dst_all + fg.e[w.ei].off;
        const int64_t ld = w.ld;
        const int ncols = (w.c + B <= w.p0) ? B : (int)(w.p0 - w.c);
        T* __restrict__ drow = dst + ((w.blk << (s + q)) + ((int64_t)w.kappa << q)) * ld + w.c;

        // (ALIGNED: always true, but not known to the compiler, which then
        // schedules the stores worse: 1024 x 2004 12.6 us, 13.3; the 8-bit
        // beam's search 13.77 ms, 13.98)
        const bool vec = ALIGNED ? !quads : (ld & 3) == 0 && (w.c & 3) == 0 && ((uintptr_t)dst & 15) == 0;
        const int early = !ALIGNED && w.c < 0 ? (int)-w.c : 0;  // columns before the row's start

        // sub-pass 1: groups of R1 consecutive rows
        auto sub1 = [&](auto tt) {
            using F = RegFFA<T, Q1>;
            constexpr int nstrips = (W1 + 3) / 4;
            if constexpr (INPLACE) {
                // 32 strips at a time from the left: a strip's halo lies in
                // its own wave, read before the wave's stores, or to the right
                T* grp = bufA + warp * R1 * WA;
                for (int s0 = 0; s0 < nstrips; s0 += 32) {
                    const int x0 = 4 * (s0 + lane);
                    const bool on = s0 + lane < nstrips;
                    T a[R1][F::W], out[R1][4];
                    if (on) {
                        F::template load_rows<decltype(tt)::value>(grp + x0, WA, 0, a, std::make_index_sequence<R1>{});
                        F::run(a, out);
                    }
                    __syncwarp();
                    if (on) {
#pragma unroll
                        for (int v = 0; v < R1; ++v)
                            *reinterpret_cast<int4*>(grp + v * WA + x0) =
                                make_int4(as_bits(out[v][0]), as_bits(out[v][1]), as_bits(out[v][2]), as_bits(out[v][3]));
                    }
                    __syncwarp();
                }
            } else {
                constexpr int items = (rows / R1) * nstrips;
                for (int it = threadIdx.x; it < items; it += FK_THREADS) {
                    const int strip = it % nstrips, g = it / nstrips;
                    const int x0 = 4 * strip;
                    T a[R1][F::W];
                    // rows g * R1 + u: (t * (g * R1 + u)) & 3 = (t * u) & 3 when R1 is a multiple of 4
                    F::template load_rows<decltype(tt)::value>(bufA + g * R1 * WA + x0, WA, 0, a,
                                                               std::make_index_sequence<R1>{});
                    T out[R1][4];
                    F::run(a, out);
                    if (Q2 == 0) {
                        if (x0 < ncols) {
#pragma unroll
                            for (int v = 0; v < R1; ++v) store4(drow + v * ld + x0, out[v], ncols - x0, vec, early - x0);
                        }
                    } else {
                        // group g is input row u2 = g of sub-pass 2
#pragma unroll
                        for (int v = 0; v < R1; ++v)
                            *reinterpret_cast<int4*>(bufB + (v * R2 + g) * WB + x0) =
                                make_int4(as_bits(out[v][0]), as_bits(out[v][1]), as_bits(out[v][2]), as_bits(out[v][3]));
                    }
                }
            }
        };
        static_assert(Q2 == 0 || R1 % 4 == 0, "a group's rows start on the pattern");
        switch (w.t) {
            case 0: sub1(std::integral_constant<int, 0>{}); break;
            case 1: sub1(std::integral_constant<int, 1>{}); break;
            case 2: sub1(std::integral_constant<int, 2>{}); break;
            default: sub1(std::integral_constant<int, 3>{}); break;
        }
        __syncthreads();
        if constexpr (Q2 > 0) {
            constexpr int nstrips = B / 4;
            constexpr int items = R1 * nstrips;
            static_assert(nstrips % 32 == 0, "one trial of sub-pass 1 per warp");
            for (int it = threadIdx.x; it < items; it += FK_THREADS) {
                const int strip = it % nstrips, k1 = it / nstrips;
                const int x0 = 4 * strip;
                const int whole = ncols - (x0 - 4 * lane);  // columns from the warp's first on
                if (x0 >= ncols) continue;
                auto sub2 = [&](auto tt) {
                    using F = RegFFA<T, Q2>;
                    T a[R2][F::W];
                    // trial k1 of group u2
                    if constexpr (INPLACE)
                        F::template load_rows<decltype(tt)::value>(bufA + k1 * WA + x0, R1 * WA, k1, a,
                                                                   std::make_index_sequence<R2>{});
                    else
                        F::template load_rows<decltype(tt)::value>(bufB + k1 * R2 * WB + x0, WB, k1, a,
                                                                   std::make_index_sequence<R2>{});
                    T out[R2][4];
                    F::run(a, out);
                    T* d = drow + (int64_t)(k1 * R2) * ld + x0;
                    // (64-row tiles: bound by instructions, not by sectors)
                    if (q == 6 || vec || !quads || whole < 128 || x0 - 4 * lane < early) {
#pragma unroll
                        for (int v = 0; v < R2; ++v) store4(d + v * ld, out[v], ncols - x0, vec, early - x0);
                    } else {
#pragma unroll
                        for (int v = 0; v < R2; ++v) {
                            const int off = (int)((uintptr_t)(d + v * ld) >> 2) & 3;  // the same in every lane
                            if (off == 0) store4(d + v * ld, out[v], 4, true);
                            else store_row(d + v * ld, out[v], off);
                        }
                    }
                };
                switch (k1 & 3) {
                    case 0: sub2(std::integral_constant<int, 0>{}); break;
                    case 1: sub2(std::integral_constant<int, 1>{}); break;
                    case 2: sub2(std::integral_constant<int, 2>{}); break;
                    default: sub2(std::integral_constant<int, 3>{}); break;
                }
            }
        }
    }
}

// Split m stages into passes of at most `qmax`, as evenly as possible.
static int split_passes(int m, int qmax, int* qs) {
    if (m == 0) return 0;
    int np = (m + qmax - 1) / qmax;
    for (int i = 0; i < np; ++i) qs[i] = m / np + (i < m % np ? 1 : 0);
    return np;
}

// Fill the group's CTA ranges for a pass whose CTAs cover `rows` output rows
// and `tile` columns; returns the launch's CTA count.  The pass reads rows of
// `plane` (null: of the series) and writes rows of `dst`; *aligned: every row's
// tiles start on four-element boundaries in both.  Otherwise a tile may begin
// up to three columns early.
static int64_t group_units(FoldGroup& fg, int64_t m_rows, int rows, int tile, const void* plane, const void* dst,
                           size_t esz, bool* aligned) {
    int64_t u = 0;
    uint64_t all = reinterpret_cast<uintptr_t>(dst) / 4;
    for (int i = 0; i < fg.n; ++i) {
        const uint64_t base = reinterpret_cast<uintptr_t>(plane ? plane : fg.e[i].src) / esz;
        const uint64_t pitch = plane ? (uint64_t)fg.e[i].ld : rows % 4 == 0 ? 0 : (uint64_t)fg.e[i].p0;
        all |= base | pitch | (uint64_t)fg.e[i].ld | (uint64_t)fg.e[i].off;
        const int64_t tiles = (fg.e[i].p0 + ((base | pitch) & 3 ? 3 : 0) + tile - 1) / tile;
        fg.e[i].n_ct = (int32_t)std::min<int64_t>(tiles, INT32_MAX);
        fg.e[i].unit0 = (uint32_t)u;
        u += (m_rows / rows) * tiles;
    }
    *aligned = (all & 3) == 0;
    return u;
}

template <class T, bool FIRST, int Q1, int Q2, int B>
static ffa_status launch_k(const void* src, T* dst, FoldGroup& fg, int64_t m_rows, int s, cudaStream_t st) {
    constexpr int q = Q1 + Q2;
    constexpr int rows = 1 << q;
    constexpr int wa = fk_wa(q, Q1, B), wb = fk_wb(q, Q1, B);
    const size_t smem = sizeof(T) * (size_t)rows * (fk_inplace(Q1, Q2) ? fk_max(wa, wb) : wa + (Q2 > 0 ? wb : 0));
    using S = typename std::conditional<FIRST, typename FoldIn<T>::type, T>::type;
    bool aligned = false;
    const int64_t units = group_units(fg, m_rows, rows, B, FIRST ? nullptr : src, dst, sizeof(S), &aligned);
    if (units <= 0) return FFA_OK;
    if (units > INT32_MAX) return fail(FFA_ERR_UNSUPPORTED, "fold: plane too large for one launch");
    const ffa_status es = ensure_smem(aligned ? (const void*)k_fold<T, FIRST, Q1, Q2, B, true>
                                              : (const void*)k_fold<T, FIRST, Q1, Q2, B, false>, smem);
    if (es != FFA_OK) return es;
    if (aligned) k_fold<T, FIRST, Q1, Q2, B, true><<<(unsigned)units, FK_THREADS, smem, st>>>(src, dst, s, fg.n, false, fg);
    else k_fold<T, FIRST, Q1, Q2, B, false><<<(unsigned)units, FK_THREADS, smem, st>>>(src, dst, s, fg.n, units >= sm_count(), fg);
    FFA_LAUNCH_CHECK("k_fold");
    count_launch();
    return FFA_OK;
}

// Tile width of a pass: `wide` != 0 takes 256 columns, else 128.
template <class T, bool FIRST, int Q1, int Q2>
static ffa_status launch_kb(bool wide, const void* src, T* dst, FoldGroup& fg, int64_t m_rows, int s,
                            cudaStream_t st) {
    return wide ? launch_k<T, FIRST, Q1, Q2, 256>(src, dst, fg, m_rows, s, st)
                : launch_k<T, FIRST, Q1, Q2, 128>(src, dst, fg, m_rows, s, st);
}

template <class T, bool FIRST>
static ffa_status pass_q(int q, bool wide, const void* src, T* dst, FoldGroup& fg, int64_t m_rows, int s,
                         cudaStream_t st) {
    switch (q) {
        case 0: return launch_kb<T, FIRST, 0, 0>(wide, src, dst, fg, m_rows, s, st);
        case 1: return launch_kb<T, FIRST, 1, 0>(wide, src, dst, fg, m_rows, s, st);
        case 2: return launch_kb<T, FIRST, 2, 0>(wide, src, dst, fg, m_rows, s, st);
        case 3: return launch_kb<T, FIRST, 3, 0>(wide, src, dst, fg, m_rows, s, st);
        case 4: return launch_kb<T, FIRST, 2, 2>(wide, src, dst, fg, m_rows, s, st);
        case 5: return launch_kb<T, FIRST, 3, 2>(wide, src, dst, fg, m_rows, s, st);
        case 6: return launch_kb<T, FIRST, 3, 3>(wide, src, dst, fg, m_rows, s, st);
        default: break;
    }
    return fail(FFA_ERR_ARG, "fold: at most 6 stages per pass");
}

// The fold's launch shape: at most `qmax` stages per pass, tiles of `tile`
// columns (0: 256 below six stages, 128 at six, so that four CTAs fit an SM).
struct FoldShape {
    int qmax;
    int tile;
};

template <class T>
static ffa_status fold_impl(const void* d_z, FoldGroup& fg, int64_t m_rows, int stages, T* d_plane, T* d_tmp,
                            cudaStream_t st, FoldShape fs) {
    int qs[64];
    int np = split_passes(stages, fs.qmax, qs);
    if (np == 0) {
        // no stage to run: copy the (zero-padded) rows
        np = 1;
        qs[0] = 0;
    }
    // ping-pong so that the last pass lands in d_plane
    T* bufs[2] = {d_plane, d_tmp};
    int s = 0;
    for (int pi = 0; pi < np; ++pi) {
        T* dst = bufs[(np - 1 - pi) & 1];
        const void* src = pi == 0 ? d_z : (const void*)bufs[(np - pi) & 1];
        const bool wide = fs.tile == 256 || (fs.tile == 0 && qs[pi] < 6);
        ffa_status e = pi == 0 ? pass_q<T, true>(qs[pi], wide, src, dst, fg, m_rows, s, st)
                               : pass_q<T, false>(qs[pi], wide, src, dst, fg, m_rows, s, st);
        if (e != FFA_OK) return e;
        s += qs[pi];
    }
    return FFA_OK;
}

// ---------------------------------------------------------------------------
// Stages per pass and tile width, tuned.  Any split of the stages into passes,
// and any tile width, gives the same add tree (bit-identical planes); only the
// time differs.  The cache maps (device, precision, stages, floor(log2 p0),
// rows on 16-byte boundaries) to the fastest shape measured by tune_fold;
// untuned shapes use six stages per pass with the default widths.
// ---------------------------------------------------------------------------
namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int, bool>, FoldShape> g_tune;
constexpr FoldShape SHAPE_DEFAULT = {6, 0};

int log2i(int64_t v) {
    int r = 0;
    while ((int64_t)2 << r <= v) ++r;
    return r;
}

FoldShape tuned_shape(int precision, int stages, int64_t p0, int64_t ld) {
    // Untuned, twelve stages on dense rows that are not 16-byte aligned: three
    // passes of four instead of two of six (4096 x 366 / 1489 / 4001 / 7001 /
    // 19977: 19 / 38 / 86 / 142 / 373 us, 17 / 37 / 85 / 138 / 376; int8 20 / 38
    // / 84 / 140 / 367, 23 / 39 / 82 / 128 / 346).  Eleven stages stay two
    // passes (2048 x 19977: 167 us, 229 as four, four and three).
    const FoldShape none = (ld & 3) != 0 && stages == 12 ? FoldShape{5, 0} : SHAPE_DEFAULT;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return none;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune.find(std::make_tuple(dev, precision, stages, log2i(p0), (ld & 3) == 0));
    return it == g_tune.end() ? none : it->second;
}
}  // namespace

static ffa_status fold_group(const void* d_z, int32_t precision, FoldGroup& fg, int64_t m_rows, int stages,
                             void* d_plane, void* d_tmp, cudaStream_t st, FoldShape fs) {
    if (precision == FFA_FOLD_F32)
        return fold_impl<float>(d_z, fg, m_rows, stages, (float*)d_plane, (float*)d_tmp, st, fs);
    return fold_impl<int32_t>(d_z, fg, m_rows, stages, (int32_t*)d_plane, (int32_t*)d_tmp, st, fs);
}

static ffa_status fold_with(const void* d_z, int32_t precision, int64_t p0, int64_t m_data, int64_t m_rows,
                            int stages, int64_t ld, void* d_plane, void* d_tmp, cudaStream_t st, FoldShape fs) {
    FoldGroup fg;
    fg.n = 1;
    fg.e[0].p0 = p0;
    fg.e[0].m_data = m_data;
    fg.e[0].off = 0;
    fg.e[0].ld = ld;
    fg.e[0].src = d_z;
    return fold_group(d_z, precision, fg, m_rows, stages, d_plane, d_tmp, st, fs);
}

// A group of n base periods on padded planes.
static FoldGroup padded_group(const void* d_z, int n, const int64_t* p0, const int64_t* m_data, const int64_t* off,
                              const void* const* z) {
    FoldGroup fg;
    fg.n = n;
    for (int i = 0; i < n; ++i) {
        fg.e[i].p0 = p0[i];
        fg.e[i].m_data = m_data[i];
        fg.e[i].off = off[i];
        fg.e[i].ld = plane_pitch(p0[i]);
        fg.e[i].src = z ? z[i] : d_z;
    }
    return fg;
}

// Time each maximum pass depth 3..6 with each tile width (128 and 256
// columns) on one group (CUDA events, best of 2 after a warm-up) and cache
// the fastest.  The planes are scratch.
ffa_status tune_fold(const void* d_z, int32_t precision, int n, const int64_t* p0, const int64_t* m_data,
                     const int64_t* off, int64_t m_rows, int stages, void* d_plane, void* d_tmp, cudaStream_t st) {
    if (n < 1 || n > FOLD_GROUP_MAX) return fail(FFA_ERR_ARG, "fold group: 1..FOLD_GROUP_MAX base periods");
    FoldGroup fg = padded_group(d_z, n, p0, m_data, off, nullptr);
    auto fold = [&](FoldShape fs) { return fold_group(d_z, precision, fg, m_rows, stages, d_plane, d_tmp, st, fs); };
    cudaEvent_t e0, e1;
    FFA_CUDA_TRY(cudaEventCreate(&e0));
    FFA_CUDA_TRY(cudaEventCreate(&e1));
    float best = 1e30f;
    FoldShape bs = SHAPE_DEFAULT;
    ffa_status s = FFA_OK;
    for (int q = 3; q <= 6 && s == FFA_OK; ++q) {
        for (int tile : {128, 256}) {
            const FoldShape fs = {q, tile};
            s = fold(fs);  // warm-up
            float t_q = 1e30f;
            for (int rep = 0; rep < 2 && s == FFA_OK; ++rep) {
                cudaEventRecord(e0, st);
                s = fold(fs);
                cudaEventRecord(e1, st);
                if (cudaEventSynchronize(e1) != cudaSuccess) s = cuda_fail(cudaGetLastError(), "tune_fold");
                float ms = 0.0f;
                cudaEventElapsedTime(&ms, e0, e1);
                t_q = ms < t_q ? ms : t_q;
            }
            if (s != FFA_OK) break;
            if (t_q < best) {
                best = t_q;
                bs = fs;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (s != FFA_OK) return s;
    int dev = 0;
    FFA_CUDA_TRY(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tune[std::make_tuple(dev, precision, stages, log2i(p0[n - 1]), true)] = bs;
    }
    return FFA_OK;
}

ffa_status launch_fold_group(const void* d_z, int32_t precision, int n, const int64_t* p0, const int64_t* m_data,
                             const int64_t* off, int64_t m_rows, int stages, void* d_plane, void* d_tmp,
                             cudaStream_t st, const void* const* z) {
    if (n < 1 || n > FOLD_GROUP_MAX) return fail(FFA_ERR_ARG, "fold group: 1..FOLD_GROUP_MAX base periods");
    FoldGroup fg = padded_group(d_z, n, p0, m_data, off, z);
    return fold_group(d_z, precision, fg, m_rows, stages, d_plane, d_tmp, st,
                      tuned_shape(precision, stages, p0[n - 1], plane_pitch(p0[n - 1])));
}

// Run the first `stages` FFA stages (all of them when stages < 0).  With
// fewer stages the plane holds, per group of 2^stages rows, its partial
// trials (row g * 2^stages + kappa); zero stages copy the (zero-padded) rows.
ffa_status launch_fold(const void* d_z, int32_t precision, int64_t p0, int64_t m_data,
                       int64_t m_rows, int stages, int64_t ld, void* d_plane, void* d_tmp, cudaStream_t st) {
    int m = 0;
    while ((1ll << m) < m_rows) ++m;
    if (stages < 0 || stages > m) stages = m;
    return fold_with(d_z, precision, p0, m_data, m_rows, stages, ld, d_plane, d_tmp, st,
                     tuned_shape(precision, stages, p0, ld));
}

}  // namespace ffa

// ---------------------------------------------------------------------------
// Fold without any allocation (see ffa_fold_noalloc in include/ffa.h).
// ---------------------------------------------------------------------------
namespace {
// Scratch plane shared by every ffa_fold_noalloc call on a device; it lives
// in the module image, so every GPU that loads the library holds it.
static __device__ __align__(256) float g_fold_scratch[FFA_NOALLOC_FOLD_MAX_ELEMS];

// The array's device address is looked up once per device and context: a
// cudaDeviceReset (or any re-creation of the primary context) reloads the
// module, so the address is looked up again when the current context's
// unique id changes.  The driver calls come through the runtime's entry
// point query, so the library still links only against the runtime.
typedef CUresult (*ctx_get_current_t)(CUcontext*);
typedef CUresult (*ctx_get_id_t)(CUcontext, unsigned long long*);

std::mutex g_scratch_mu;
struct ScratchSlot {
    void* ptr = nullptr;
    unsigned long long ctx_id = 0;
    bool has_id = false;
};
ScratchSlot g_scratch[64];

// Unique id of the calling thread's current context; false if none is
// current yet or the driver does not offer the query.
bool current_ctx_id(unsigned long long* id) {
    static ctx_get_current_t get_cur = nullptr;
    static ctx_get_id_t get_id = nullptr;
    static bool looked = false;
    if (!looked) {
        looked = true;
        cudaDriverEntryPointQueryResult q1, q2;
        void* f1 = nullptr;
        void* f2 = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
            q1 == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
            q2 == cudaDriverEntryPointSuccess) {
            get_cur = (ctx_get_current_t)f1;
            get_id = (ctx_get_id_t)f2;
        }
    }
    if (!get_cur || !get_id) return false;
    CUcontext ctx = nullptr;
    if (get_cur(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return get_id(ctx, id) == CUDA_SUCCESS;
}
}  // namespace

extern "C" ffa_status ffa_fold_noalloc(const void* d_z, int32_t precision, int64_t p0, int64_t m_data,
                                       int64_t m_rows, void* d_plane, void* stream) {
    using namespace ffa;
    if (p0 < 1 || m_data < 0 || m_rows < 1 || (m_rows & (m_rows - 1)) != 0 || m_data > m_rows)
        return fail(FFA_ERR_ARG, "fold_noalloc: need p0 >= 1, m_rows a power of two >= m_data");
    if (precision != FFA_FOLD_F32 && precision != FFA_FOLD_I8)
        return fail(FFA_ERR_ARG, "fold_noalloc: bad precision");
    if (!d_z || !d_plane) return fail(FFA_ERR_ARG, "fold_noalloc: null buffer");
    // m_rows >= 1 here; the division form cannot overflow
    if (p0 > (int64_t)FFA_NOALLOC_FOLD_MAX_ELEMS / m_rows)
        return fail(FFA_ERR_UNSUPPORTED,
                    "fold_noalloc: m_rows * p0 exceeds FFA_NOALLOC_FOLD_MAX_ELEMS (the fixed scratch)");
    int dev = 0;
    FFA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(FFA_ERR_UNSUPPORTED, "fold_noalloc: device index >= 64");
    void* scratch;
    {
        // set-up once per device and context, with that device current: the
        // device address of the array (its host-side name is only a stand-in,
        // not a device address)
        std::lock_guard<std::mutex> lk(g_scratch_mu);
        ScratchSlot& sl = g_scratch[dev];
        unsigned long long id = 0;
        const bool has_id = current_ctx_id(&id);
        if (!sl.ptr || !has_id || !sl.has_id || id != sl.ctx_id) {
            void* ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_fold_scratch);
            if (e != cudaSuccess || !ptr) return cuda_fail(e, "fold_noalloc: cudaGetSymbolAddress");
            sl.ptr = ptr;
            // the lookup makes the primary context current if none was
            sl.has_id = current_ctx_id(&sl.ctx_id);
        }
        scratch = sl.ptr;
    }
    return launch_fold(d_z, precision, p0, m_data, m_rows, -1, p0, d_plane, scratch, as_stream(stream));
}
