// hjlo_dense.cuh -- the axis pass by register tiles: the monotone search for
// windows of up to kDenseMaxWindow displacements.
//
// The screen.  Per tile, u and k are turned into 32-bit keys on one scale:
//     f[jj] = floor((u - min u) / 2^q) masked,   K[t] = floor((k + max|k|) / 2^q) masked,
// 2^q so that every sum of a value and a table entry stays below 2^31.  The
// low kBits bits are masked off, so those of a sum are free for a candidate's
// number: one instruction (add, unsigned minimum) both compares a candidate and
// remembers where it came from.  Two candidates' sums (without the number)
// are off their exact difference by less than 2 (2^kBits + 1) key units, and
// binary64 rounding of the exact sums adds at most one more (2^q >= 8 ulp):
// kThr.  When the kernel's second differences are at least 2^kCurv key units
// (checked per tile), K is strictly convex, so the screened candidate matrix
// is Monge by itself and its row minima are monotone.
//
// Flat search (windows of up to kFlatMaxWindow).  Every row is compared with
// its whole window, four rows a lane: 16 add-minimums per two 128-bit loads.
// That is more comparisons than monotonicity asks for (65 a row against 5.7)
// at 1.1 instructions each, with every lane busy and no row waiting for
// another; divide and conquer spent 208 instructions a row, at 55-70 % of the
// lanes.  256^3 grid, 65 displacements, binary64: 235 -> 157 us a pass.
//
// Banded search (wider windows).  A lane owns a segment of S rows: it scans
// the whole window for the first (the pivot), and after a barrier it knows
// sources jl and jr of its own and the next segment's pivot, between which every
// row of its segment finds its minimum.  Away from shocks jr - jl is about S,
// and the S - 1 rows are searched together, in registers: chunks of 4 sources
// by S - 1 rows, each chunk 4 loads of f, 4 of K (the table window slides) and
// 4 (S - 1) add-minimums.  Segments with more than 16 sources (shocks) are
// shared by the lanes of the warp, two rows a lane, several lanes a source
// range when few segments are left.  1024^2 grid, 129 displacements: 27 -> 19
// us a pass.  Above kScanWindow displacements (kWide) the lanes of a warp find
// the pivots together, halving the distance between known ones; four number
// bits leave room for the curvature of a window that wide (its square over 2^23
// of the table's range), up to kDenseMaxWindow.
//
// Making it exact.  A row's screened argmin is the binary64 one unless a rival
// lies within kThr of it.  In a wide segment the runner-up is kept.  Elsewhere
// each row keeps four minima, one per source number mod 4: a rival of another
// class shows in them, and one of the same class is 4 or more sources away;
// since it gains at least 2^kCurv - kFlag on the nearer sources with each row,
// the neighbouring row's source (the row before's for a rival to the left, the
// row after's for one to the right) has passed it, so it shows as a step of 4 or
// more between two rows' sources.  Every pair of neighbours is looked at: two
// rows of a lane, a lane's last row and the next lane's first, and round the
// end of the line: row N - 1 and row 0's image one period on (when the last
// segment is a wide one, the image row is searched with it, over the whole of
// its window), or for row blocks row NR - 1 and row NR, and row -1 (row N - 1
// of the block's periodic line) and row 0.  The flat search, which has none of
// a row block's outer rows, flags row 0 of every block instead; wide windows'
// pivots keep their runner-up.  Rows flagged by either are searched again
// between their neighbours' sources (a rival further out would have taken the
// neighbour), survivors of the screen compared in binary64, smallest source
// first (1-4 % of the rows on the solver's fields).
//
// What bounds it.  The pipe of the 32-bit minimum, logic and shift instructions
// (64 lanes a clock and SM, 62-68 % busy), shared-memory words (62 %) and issue
// slots (65 %) are within a factor of 1.1 of one another; staging and write-back
// alone take 68 of the 155 us on the 256^3 grid.
#pragma once

#include "hjlo_device.cuh"

namespace hjlo {

constexpr int kDenseMaxWindow = 3584;            // widest window (displacements; see kWide)
constexpr int kScanWindow = 512;                 // widest window a lane scans alone for its pivot
constexpr int kWide = 11;                        // the S of the banded search for wider ones
constexpr int kFlat = 4;                         // the S of the flat search
constexpr int kFlatMaxWindow = 96;               // widest window it takes (at most 128, its key numbers)
constexpr unsigned kDensePad = 0x80000000u;      // table entries outside the window
constexpr int kDenseLow = 16, kDenseHigh = 32;   // padding of the table K
constexpr int kDenseOver = 16;                   // halo entries past N + weff - 1 (row N's last, full bands)

// Low key bits (a source's number in its band; the displacement's in the flat
// search), the screen's error between two sums without and with them, and the
// curvature it needs (2^kCurv key units).
template <int S>
struct DenseKey {
    static constexpr int kBits = (S == kFlat) ? 7 : (S == kWide) ? 4 : 5;
    static constexpr unsigned kMask = (1u << kBits) - 1u, kThr = 2u * kMask + 6u, kFlag = kThr + kMask;
    static constexpr int kCurv = kBits + 3;
};

// Threads of a CTA at most, and CTAs an SM must hold (which caps registers).
__host__ __device__ constexpr int dense_threads(int S) { return S == kFlat ? 256 : 512; }
__host__ __device__ constexpr int dense_ctas(int S) { return S == kFlat ? 4 : S <= 9 ? 2 : 1; }

// Per-tile facts, in shared memory after the mbarrier.
struct DenseInfo {
    int kmin, kmax;             // extremes of the tile (float_key)
    unsigned fref, kref;        // keys' references: below min u and -max|k| at 2^q
    int q;                      // key unit 2^q (32 of them: 2^(q+5))
    int ok;                     // the screen holds: finite values, enough curvature
};

// Sources of a bracket that one lane searches.
template <int S>
struct DenseBand {
    static constexpr int kChunks = 4, kSources = 4 * kChunks;
};

// x / 2^q as an integer, modulo 2^32 (two's complement), for |x| < 2^(q + 50)
// and q >= -960, two ways: rounded, by adding 1.5 * 2^(q + 52), which leaves it
// in the low word (one binary64 add); and truncated, by shifting the
// significand (eleven integer instructions; no left shift and no subnormals
// under these bounds).  A tile's keys are made half by each, since the first
// alone waits for the binary64 pipe and the second for the logic pipe.
__device__ __forceinline__ double key_magic(int q) { return __hiloint2double(((q + 52 + 1023) << 20) | 0x80000, 0); }
__device__ __forceinline__ unsigned fixkey(double x, double magic)
{
    return (unsigned)__double2loint(__dadd_rn(x, magic));
}

__device__ __forceinline__ unsigned fixshift(double x, int q)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int s = 1075 + q - (int)((hi >> 20) & 0x7ffu);
    const unsigned a = __funnelshift_rc(lo, (hi & 0xfffffu) | 0x100000u, (unsigned)s);
    const unsigned v = __funnelshift_rc(a, 0u, (unsigned)max(s - 32, 0));
    const unsigned sg = (unsigned)((int)hi >> 31);
    return (v ^ sg) - sg;
}

// min / max of the values in 32 bits: a binary64 value's high word taken as a
// binary32 number (same order; NaN for NaN, infinity and magnitudes from
// 2^1017, kept by the NaN-propagating minimum), a binary32 value itself.
// float_key: the extremes as integers of the same order; key_hi: their high
// words as binary64 numbers.
__device__ __forceinline__ void hi_minmax(float h, float &mn, float &mx)
{
    asm("min.NaN.f32 %0, %0, %1;" : "+f"(mn) : "f"(h));
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(mx) : "f"(h));
}
__device__ __forceinline__ void hi_minmax(double x, float &mn, float &mx)
{
    hi_minmax(__int_as_float(__double2hiint(x)), mn, mx);
}
__device__ __forceinline__ int float_key(float x)
{
    const int b = __float_as_int(x);
    return b ^ ((b >> 31) & 0x7fffffff);
}
template <typename T>
__device__ __forceinline__ int key_hi(int key);
template <>
__device__ __forceinline__ int key_hi<double>(int key) { return key ^ ((key >> 31) & 0x7fffffff); }
template <>
__device__ __forceinline__ int key_hi<float>(int key)
{
    return __double2hiint(widen(__int_as_float(key ^ ((key >> 31) & 0x7fffffff))));
}
// +-significand(h) 2^(e(h) - 1043 - q), h the high word of a binary64 number of
// either sign, rounded down (the low word as large as it can be for a negative
// one), modulo 2^32: a reference below every key of values from that number on.
__device__ __forceinline__ unsigned key_below(int h, int q)
{
    const int e = (h >> 20) & 0x7ff, s = e - 1043 - q;
    const unsigned neg = (unsigned)(h >> 31);
    unsigned m = ((unsigned)h & 0xfffffu) | 0x100000u;
    if (e == 0) return neg;                          // far below one unit
    m += neg & 1u;
    if (s >= 0) m = s < 32 ? m << s : 0u;
    else m = -s < 32 ? (neg ? ~(~0u << -s) + m : m) >> -s : (neg & 1u);
    return (m ^ neg) - neg;
}

// Scale of a tile, and whether the screen holds there, from its extremes' high
// words (a lower and an upper bound) with 32-bit instructions only, by one thread: the binary64 pipe is
// busy with other CTAs' sums, and a chain of a dozen dependent operations on it
// took 2200 clocks of a tile's 25000.
__device__ __forceinline__ void dense_scale(int hmin, int hmax, double kmax, double curv, int cbits, DenseInfo *info)
{
    const int hk = __double2hiint(kmax), hc = __double2hiint(curv);
    const int E = max(max(max(hmin & 0x7fffffff, hmax & 0x7fffffff), hk) >> 20, 1);
    // the numbers scaled by 2^(1023 - E), to 20 bits
    auto scaled = [&](int h) -> float {
        const int e = ((h >> 20) & 0x7ff) - E + 127;
        return e <= 0 ? 0.0f : __int_as_float((h & (int)0x80000000) | (e << 23) | ((h & 0xfffff) << 3));
    };
    // the four discarded low words are worth less than 2^-18 together
    const float Rk = scaled(hmax) - scaled(hmin) + 2.0f * scaled(hk) + 0x1.4p-18f;
    const int q = max(max((__float_as_int(Rk) >> 23) - 127 + E - 1023 - 30, E - 1022 - 49), -960);
    // curvature of at least 2^cbits units; with 2^q >= 8 ulp that is far more
    // than binary64 ties need
    const bool ok = E < 0x7ff && q <= 900 && hc > 0 && (hc >> 20) - 1023 >= q + cbits;
    info->q = q;
    info->ok = ok ? 1 : 0;
    info->fref = key_below(hmin, q);
    info->kref = key_below(hk | (int)0x80000000, q);
}

// NCH chunks of 4 sources (as many as hold the first n; n uniform over the
// warp) against the S - 1 rows after a pivot row: fj = f at the band's first
// source, kq = K at that source seen from the pivot row; the sources are
// numbered from 0.  The next chunk's words are loaded before a chunk is used.
template <int S, int NCH>
__device__ __forceinline__ void dense_band(const unsigned *fj, const unsigned *kq, int n,
                                           unsigned (&a)[S - 1][4])
{
    unsigned w[S + 2];          // K at offsets 4c - (S - 1) .. 4c + 2
    unsigned f[4], fn[4], wn[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) f[e] = fj[e];
#pragma unroll
    for (int o = 0; o < S + 2; ++o) w[o] = kq[o - (S - 1)];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        if (c + 1 < NCH) {
#pragma unroll
            for (int e = 0; e < 4; ++e) fn[e] = fj[4 * c + 4 + e];
#pragma unroll
            for (int e = 0; e < 4; ++e) wn[e] = kq[4 * c + 3 + e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned fv = f[e] + (unsigned)(4 * c + e);
#pragma unroll
            for (int q = 1; q < S; ++q) a[q - 1][e] = __viaddmin_u32(fv, w[e - q + S - 1], a[q - 1][e]);
        }
        if (4 * c + 4 >= n) break;
#pragma unroll
        for (int e = 0; e < 4; ++e) f[e] = fn[e];
#pragma unroll
        for (int o = 0; o < S - 2; ++o) w[o] = w[o + 4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[S - 2 + e] = wn[e];
    }
}

// Best and second best of four class minima.
__device__ __forceinline__ void best_two(const unsigned (&a)[4], unsigned &m, unsigned &m2)
{
    const unsigned lo1 = min(a[0], a[1]), hi1 = max(a[0], a[1]);
    const unsigned lo2 = min(a[2], a[3]), hi2 = max(a[2], a[3]);
    m = min(lo1, lo2);
    m2 = min(max(lo1, lo2), min(hi1, hi2));
}

// One row's candidates by offset t: the screened sum, and among the offsets
// tlo, tlo + step, ... <= thi whose screened sum is at most thr the smallest
// binary64 sum (smallest offset on ties).
template <typename T, int LAYOUT>
struct DenseRow {
    const T *su;
    const double *kr64;
    const unsigned *f, *k;      // key halo at row r, table at offset 0
    int N, hoff, log2C;
    int l, r;

    __device__ __forceinline__ unsigned key(int t) const { return f[t] + k[t]; }
    __device__ __forceinline__ Key2 sum(int t) const
    {
        const int pos = wrapN(r + t + hoff, N);
        const int at = (LAYOUT == LAYOUT_CONTIG) ? l * N + pos : (pos << log2C) + l;
        return key2(__dadd_rn(widen(su[at]), kr64[t]));
    }
    __device__ __forceinline__ void exact(int tlo, int thi, int step, unsigned thr, Key2 &best, int &bt) const
    {
        for (int t = tlo; t <= thi; t += step)
            if (key(t) <= thr) {
                const Key2 c = sum(t);
                if (key2_less(c, best)) { best = c; bt = t; }
            }
    }
};

// A staged tile whose screen does not hold (a value that is not finite, one
// line far from the others, or too little curvature for the range): divide and
// conquer, with its own scale, survivors and margin for every line, and brute
// force for a line that fails the margin.  Kept out of line, where it leaves the
// searches' registers alone.
template <typename T, int LAYOUT, typename OFF>
__device__ __noinline__ void dense_leave(const PassParams &p, long long tile)
{
    clear_line_ranges(p, reinterpret_cast<LineInfo *>(pass_smem() + p.off_misc + 16));
    __syncthreads();
    search_tile<T, LAYOUT, KALGO_MONGE, OFF>(p, tile);
}

// `launch`: where p lies in memory (kernel parameters, shared memory), or null
// for a copy in registers.
template <typename T, int LAYOUT, typename OFF, int S>
__device__ __forceinline__ void dense_tile(const CUtensorMap *tmap, const PassParams &p, long long tile,
                                           const PassParams *launch)
{
    extern __shared__ __align__(128) unsigned char smem[];
    T *su = reinterpret_cast<T *>(smem + p.off_u);
    unsigned *fx = reinterpret_cast<unsigned *>(smem + p.off_fx);
    unsigned *kpad = reinterpret_cast<unsigned *>(smem + p.off_kfx);      // K, padded on both sides
    unsigned *kp = reinterpret_cast<unsigned *>(smem + p.off_kp);         // K with chunk numbers (pivots)
    OFF *tt = reinterpret_cast<OFF *>(smem + p.off_t);
    double *kr64 = reinterpret_cast<double *>(smem + p.off_k64);
    DenseInfo *info = reinterpret_cast<DenseInfo *>(smem + p.off_misc + 16);

    using Key = DenseKey<S>;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int N = (int)p.N, C = p.C, weff = p.weff, lpl = p.lpl;
    const Tile<LAYOUT> tl = tile_of<LAYOUT>(p, tile);
    // the threads that search a line: a group of lpl of them, or a warp where
    // that is more (several lines); groups run apart from one another between
    // the keys and the write-back, each with its own queue of flagged rows
    const int glog = max(p.log2lpl, 5), gsize = 1 << glog, grp = tid >> glog, gt = tid & (gsize - 1);
    unsigned *queue = reinterpret_cast<unsigned *>(smem + p.off_q) + grp * (p.qcap + 1);   // [0]: entries
    const bool member = tid < C * lpl;
    if (member && gt == 0) queue[0] = 0;
    if (tid == 0) {
        info->kmin = 0x7fffffff;
        info->kmax = (int)0x80000000;
    }
    if (!stage_tile<T, LAYOUT, true>(tmap, p, tile, su, kr64, reinterpret_cast<uint64_t *>(smem + p.off_misc))) return;

    const int cl = tid >> p.log2lpl, sub = tid & (lpl - 1);
    {
        // ---- range of the tile
        const int l = (LAYOUT == LAYOUT_CONTIG) ? cl : tid & (C - 1);
        const int first = (LAYOUT == LAYOUT_CONTIG) ? sub : tid >> p.log2C;
        const int step = (LAYOUT == LAYOUT_CONTIG) ? lpl : nthr >> p.log2C;
        const bool mine = l < tl.valid;
        float mn = __int_as_float(0x7f800000), mx = __int_as_float((int)0xff800000);
        {
            // every thread its share of the staged values (a full tile of
            // strided lines, and any of contiguous ones, is one array)
            const int n = (LAYOUT == LAYOUT_CONTIG) ? tl.valid * N : (mine ? C * N : 0);
            const T *x = su + tid;
            int i = tid;
            for (; i + 3 * nthr < n; i += 4 * nthr) {
                T v[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) v[b] = x[b * nthr];
                x += 4 * nthr;
#pragma unroll
                for (int b = 0; b < 4; ++b) hi_minmax(v[b], mn, mx);
            }
            for (; i < n; i += nthr, x += nthr) hi_minmax(*x, mn, mx);
        }
        const int a = __reduce_min_sync(0xffffffffu, float_key(mn));
        const int b = __reduce_max_sync(0xffffffffu, float_key(mx));
        if (lane == 0) {
            atomicMin(&info->kmin, a);
            atomicMax(&info->kmax, b);
        }
        __syncthreads();
        // ---- the tile's scale
        if (tid == 0) dense_scale(key_hi<T>(info->kmin), key_hi<T>(info->kmax), p.kmax, p.curv, Key::kCurv, info);
        __syncthreads();
        if (!info->ok) {
            __syncthreads();                         // everyone has looked
            if (launch) {
                dense_leave<T, LAYOUT, OFF>(*launch, tile);
            } else {
                const PassParams left = p;
                dense_leave<T, LAYOUT, OFF>(left, tile);
            }
            return;
        }
        const int q = info->q;
        // ---- keys: the halo (its first weff entries repeat one period later:
        // row N, row 0's image, is searched with the last segment when that is
        // a wide one, over its whole window; a few more entries are read by full
        // bands, beside no displacement of the window) and the table
        const double magic = key_magic(q);
        const unsigned fref = info->fref, kref = info->kref;
        const int dup = weff;
        if (mine) {
            const T *x = (LAYOUT == LAYOUT_CONTIG) ? su + l * N + first : su + tid;
            const int xs = (LAYOUT == LAYOUT_CONTIG) ? lpl : nthr;
            unsigned *lfx = fx + l * p.lp, *lfn = lfx + N;
            auto put = [&](T v, int pos, bool add) {
                const unsigned f = ((add ? fixkey(widen(v), magic) : fixshift(widen(v), q)) - fref) & ~Key::kMask;
                const int y = pos - p.hoff;                      // in (-N, N)
                const int jj = (int)min((unsigned)y, (unsigned)(y + N));
                lfx[jj] = f;
                if (jj < dup) lfn[jj] = f;
            };
            int pos = first;
            for (; pos + 3 * step < N; pos += 4 * step) {
                T v[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) v[b] = x[b * xs];
                x += 4 * xs;
#pragma unroll
                for (int b = 0; b < 4; ++b) put(v[b], pos + b * step, b & 1);
            }
            for (; pos < N; pos += step, x += xs) put(*x, pos, false);
            for (int i = first; i < kDenseOver - 1; i += step) lfn[dup + i] = 0u;
        }
        for (int i = tid; i < kDenseLow + weff + kDenseHigh; i += nthr) {
            const int t = i - kDenseLow;
            unsigned k = kDensePad;
            if (t >= 0 && t < weff) k = (fixkey(kr64[t], magic) - kref) & ~Key::kMask;
            kpad[i] = k;
            if (t >= 0 && t < ((weff + 3) & ~3)) kp[t] = k | ((unsigned)(S == kFlat ? t : t >> 2) & Key::kMask);
        }
        __syncthreads();
    }
    const unsigned *kd = kpad + kDenseLow;
    const int NR = p.rows;
    int rescans = 0;
    if (member) {
        auto gsync = [&] {
            if (gsize == 32) __syncwarp();
            else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gsize) : "memory");
        };
        auto flag = [&](int line, int row) {
            const unsigned at = atomicAdd(&queue[0], 1u);
            if (at < (unsigned)p.qcap) queue[1 + at] = ((unsigned)line << 16) | (unsigned)row;
        };
        if constexpr (S == kFlat) {
            // ---- four rows a lane at a time over the whole window: a chunk of
            // four displacements takes one 128-bit load of f (the other four
            // sources are the last chunk's), one of K for all lanes, and 16
            // add-minimums
            const unsigned *lf = fx + (cl < tl.valid ? cl : 0) * p.lp;
            OFF *lt = tt + (cl < tl.valid ? cl : 0) * p.tp;
            const uint4 *k4 = reinterpret_cast<const uint4 *>(kp);
            const int nch = (weff + 3) >> 2, end = cl < tl.valid ? NR : 0;
            for (int r = 4 * sub; r < end; r += 4 * lpl) {
                const uint4 *f4 = reinterpret_cast<const uint4 *>(lf + r);
                unsigned a[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) a[i][e] = 0xffffffffu;
                uint4 lo = f4[0];
#pragma unroll 4
                for (int c = 0; c < nch; ++c) {
                    const uint4 hi = f4[c + 1], k = k4[c];
                    const unsigned w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    const unsigned kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) a[i][e] = __viaddmin_u32(w[i + e], kk[e], a[i][e]);
                    lo = hi;
                }
                int tp = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (r + i >= end) break;
                    unsigned m, m2;
                    best_two(a[i], m, m2);
                    const int t = (int)(m & Key::kMask);
                    lt[r + i] = (OFF)t;
                    if (m2 - m <= Key::kFlag) flag(cl, r + i);
                    if (i && t - tp >= 3) { flag(cl, r + i - 1); flag(cl, r + i); }
                    tp = t;
                }
            }
            gsync();
            // steps of four sources between one lane's rows and the next's
            for (int r = 4 * sub; r < end; r += 4 * lpl) {
                const int rl = min(r + 3, NR - 1), rn = rl + 1;
                const int jn = rn < NR ? rn + lt[rn] : N + lt[0];
                if (jn - rl - lt[rl] >= 4) { flag(cl, rl); flag(cl, rn < NR ? rn : 0); }
                if (p.vN && r == 0) flag(cl, 0);         // a row block's first row has no left neighbour
            }
        } else {
        const int s0 = min(sub * S, NR), s1 = min(s0 + S, NR), nseg = (NR + S - 1) / S;
        const bool work = cl < tl.valid && s0 < s1;
        const unsigned *lfx = fx + (cl < tl.valid ? cl : 0) * p.lp;
        OFF *lt = tt + (cl < tl.valid ? cl : 0) * p.tp;
        // ---- pivots: the first row of every segment over the whole window.  A
        // row block is a periodic line of N points of which rows 0 .. NR - 1
        // are wanted; rows NR and N - 1 are searched too, as the neighbours of
        // the last one and the first.
        auto last = [&] { return p.vN ? NR + lt[NR] : N + lt[0]; };       // source of the row after the last
        unsigned fl = 0;            // flagged rows, bit i: row s0 + i
        int jl = 0;
        if constexpr (S == kWide) {
            // wide windows (a warp's lanes hold one line's segments): the warp
            // scans its first pivot's window together, then halves the
            // distance between known pivots, the lanes between two of them
            // sharing the sources between theirs
            const int g0 = (sub >> 5) << 5;
            const bool line = cl < tl.valid;
            auto search = [&](int r, int j0, int j1, int i, int width, bool act, bool own) {
                unsigned m = 0xffffffffu, m2 = 0xffffffffu;
                int js = j0;
                if (act) {
                    const unsigned *f = lfx, *k = kd - r;
                    const int jz = min(j1, r + weff - 1);
#pragma unroll 4
                    for (int j = max(j0, r) + i; j <= jz; j += width) {
                        const unsigned c = f[j] + k[j];
                        m2 = min(m2, max(m, c));
                        js = (c < m) ? j : js;
                        m = min(m, c);
                    }
                }
                for (int o = 1; o < width; o <<= 1) {
                    const unsigned om = __shfl_xor_sync(0xffffffffu, m, o), om2 = __shfl_xor_sync(0xffffffffu, m2, o);
                    const int oj = __shfl_xor_sync(0xffffffffu, js, o);
                    m2 = min(min(m2, om2), max(m, om));
                    js = (om < m || (om == m && oj < js)) ? oj : js;
                    m = min(m, om);
                }
                if (act && i == 0) {
                    lt[r] = (OFF)(js - r);
                    if (own && m2 - m <= Key::kThr) flag(cl, r);
                }
            };
            search(g0 * S, 0, 0x3fffffff, lane, 32, line && g0 * S < NR, true);
            if (p.vN) {                              // (see below)
                if (g0 == 0) search(N - 1, 0, 0x3fffffff, lane, 32, line, false);
                if (g0 == (nseg - 1) / 32 * 32) search(NR, 0, 0x3fffffff, lane, 32, line, false);
            }
            gsync();
            for (int d = 16; d; d >>= 1) {
                const int b = lane & ~(2 * d - 1), rl = (g0 + b) * S, r = rl + d * S, rr = rl + 2 * d * S;
                const bool act = line && r < NR;
                const int j0 = act ? rl + lt[rl] : 0, j1 = act ? (rr < NR ? rr + lt[rr] : last()) : 0;
                search(r, j0, j1, lane - b, 2 * d, act, true);
                __syncwarp();
            }
            if (work) jl = s0 + lt[s0];
        } else if (work || (p.vN && cl < tl.valid && sub <= nseg + 1)) {
            const int pr = work ? s0 : sub == nseg ? NR : N - 1;
            const unsigned *f = lfx + pr;
            const uint4 *k4 = reinterpret_cast<const uint4 *>(kp);
            const int nch = (weff + 3) >> 2;
            unsigned m = 0xffffffffu, m2 = 0xffffffffu;
            int t = 0;
            for (int c0 = 0; c0 < nch; c0 += (int)Key::kMask + 1) {
                unsigned a[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu};
                const int c1 = min(c0 + (int)Key::kMask + 1, nch);
#pragma unroll 4
                for (int c = c0; c < c1; ++c) {
                    const uint4 k = k4[c];
                    a[0] = __viaddmin_u32(f[4 * c], k.x, a[0]);
                    a[1] = __viaddmin_u32(f[4 * c + 1], k.y, a[1]);
                    a[2] = __viaddmin_u32(f[4 * c + 2], k.z, a[2]);
                    a[3] = __viaddmin_u32(f[4 * c + 3], k.w, a[3]);
                }
                unsigned b, b2;
                best_two(a, b, b2);
                const int e = (b == a[0]) ? 0 : (b == a[1]) ? 1 : (b == a[2]) ? 2 : 3;
                const int tb = 4 * (c0 + (int)(b & Key::kMask)) + e;
                m2 = min(min(m2, b2), max(m, b));
                t = (b < m) ? tb : t;
                m = min(m, b);
            }
            lt[pr] = (OFF)t;
            if (work) jl = s0 + t;
            if (work && m2 - m <= Key::kFlag) fl = 1u;
        }
        gsync();
        // a row block's first row and the one before it: on whole lines the last
        // segment sees this step
        if (S != kWide && p.vN && work && sub == 0 && lt[0] - (lt[N - 1] - 1) >= 4) fl |= 1u;
        // ---- the rows between two pivots (lanes without a segment search a
        // line's first rows again and keep nothing)
        constexpr int kB = DenseBand<S>::kSources;
        const int jr = (s1 < NR) ? s1 + lt[s1] : last();
        const int jc = min(jr, s1 + weff - 2);       // last source in any row's window
        const int span = work ? jc - jl + 1 : 1;
        {
            unsigned a[S - 1][4];
#pragma unroll
            for (int i = 0; i < S - 1; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[i][e] = 0xffffffffu;
            const int most = min(__reduce_max_sync(0xffffffffu, span), kB);
            dense_band<S, DenseBand<S>::kChunks>(lfx + jl, kd + (work ? jl - s0 : 0), most, a);
            if (work && span <= kB) {
                const int ta = jl - s0, cnt = s1 - s0;
                int tp = ta;                         // source of the row before, from s0
                OFF *lr = lt + s0;
#pragma unroll
                for (int i = 1; i <= S; ++i) {
                    int t = jr - s0;
                    if (i < S && i < cnt) {
                        unsigned m, m2;
                        best_two(a[i < S ? i - 1 : 0], m, m2);
                        t = ta + (int)(m & Key::kMask);
                        lr[i] = (OFF)(t - i);
                        if (m2 - m <= Key::kFlag) fl |= 1u << i;
                    }
                    // the next pivot counts once, as the first row past the segment
                    if (t - tp >= 4) fl |= 3u << (i - 1);
                    tp = t;
                }
            }
        }
        // ---- wide segments, shared by the warp: rows s0 .. s1 (with both
        // pivots, for their rivals), two a lane, over all sources jl .. jr, the
        // sources in H parts when lanes are left over
        unsigned wide = __ballot_sync(0xffffffffu, work && span > kB);
        while (wide) {
            constexpr int kPairs = (S + 1) / 2;
            const int k = __popc(wide);
            const int H = (4 * kPairs * k <= 32) ? 4 : (2 * kPairs * k <= 32) ? 2 : 1;
            const int slots = 32 / kPairs / H;
            const int unit = lane / kPairs, pair = lane - unit * kPairs;
            const int slot = unit / H, part = unit - slot * H;
            unsigned rest = wide;
            for (int i = 0; i < slot; ++i) rest &= rest - 1;
            const bool act = slot < slots && rest != 0;
            const int from = act ? __ffs(rest) - 1 : lane;
            for (int i = 0; i < slots && wide; ++i) wide &= wide - 1;
            const int b0 = __shfl_sync(0xffffffffu, s0, from);
            const int nrow = __shfl_sync(0xffffffffu, s1 - s0 + 1, from);  // rows to search
            const int j0 = __shfl_sync(0xffffffffu, jl, from);
            const int j1 = __shfl_sync(0xffffffffu, jr, from);
            const int ln = __shfl_sync(0xffffffffu, cl, from);
            const int i0 = 2 * pair;                                 // rows b0 + i0, b0 + i0 + 1
            const int len = (j1 - j0 + H) / H;
            const int ja = j0 + part * len, jz = min(ja + len, j1 + 1);
            unsigned m[2] = {0xffffffffu, 0xffffffffu}, m2[2] = {0xffffffffu, 0xffffffffu};
            int js[2] = {j0, j0};
            if (act && i0 < nrow) {
                const unsigned *f = fx + ln * p.lp;
                const unsigned *kr = kd - (b0 + i0);                 // kr[j]: K for row b0 + i0
                for (int jb = ja; jb < jz; jb += (int)Key::kMask + 1) {
                    unsigned x[2] = {0xffffffffu, 0xffffffffu}, x2[2] = {0xffffffffu, 0xffffffffu};
                    unsigned k1 = kr[jb - 1];
                    const int je = min(jb + (int)Key::kMask + 1, jz);
#pragma unroll 4
                    for (int j = jb; j < je; ++j) {
                        const unsigned fv = f[j] + (unsigned)(j - jb), k0 = kr[j];
                        x2[0] = min(x2[0], __viaddmax_u32(fv, k0, x[0]));
                        x[0] = __viaddmin_u32(fv, k0, x[0]);
                        x2[1] = min(x2[1], __viaddmax_u32(fv, k1, x[1]));
                        x[1] = __viaddmin_u32(fv, k1, x[1]);
                        k1 = k0;
                    }
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        m2[b] = min(min(m2[b], x2[b]), max(m[b], x[b]));
                        js[b] = (x[b] < m[b]) ? jb + (int)(x[b] & Key::kMask) : js[b];
                        m[b] = min(m[b], x[b]);
                    }
                }
            }
            for (int o = H >> 1; o; o >>= 1) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const unsigned om = __shfl_down_sync(0xffffffffu, m[b], o * kPairs);
                    const unsigned om2 = __shfl_down_sync(0xffffffffu, m2[b], o * kPairs);
                    const int oj = __shfl_down_sync(0xffffffffu, js[b], o * kPairs);
                    m2[b] = min(min(m2[b], om2), max(m[b], om));
                    js[b] = (om < m[b]) ? oj : js[b];
                    m[b] = min(m[b], om);
                }
            }
            if (act && part == 0) {
                OFF *wt = tt + ln * p.tp;
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int i = i0 + b, r = b0 + i;
                    if (i >= nrow) continue;
                    const bool own = i > 0 && i < S && r < NR;       // a row of the segment, no pivot
                    if (own) wt[r] = (OFF)(js[b] - r);
                    if (m2[b] - m[b] <= Key::kFlag && (r < NR || !p.vN)) flag(ln, r < NR ? r : 0);
                }
            }
        }
        // ---- queue the flagged rows (bit s1 - s0: the next pivot)
        while (fl) {
            const int b = __ffs(fl) - 1;
            fl &= fl - 1;
            const int r = s0 + b;
            if (r < NR || !p.vN) flag(cl, r < s1 ? r : (s1 < NR) ? s1 : 0);
        }
        }
        gsync();
        // ---- flagged rows (all rows of the group's lines when the queue ran over)
        {
            const unsigned nf = queue[0];
            const bool over = nf > (unsigned)p.qcap;
            const int l0 = (grp << glog) >> p.log2lpl;               // the group's first line
            const int lines = min(max(gsize >> p.log2lpl, 1), tl.valid - l0);
            const int total = over ? max(lines, 0) * NR : (int)nf;
            constexpr int kLong = 40;                                // more candidates: the warp's lanes share them
            for (int x0 = gt & ~31; x0 < total; x0 += gsize) {
                const int x = x0 + lane;
                const bool has = x < total;
                int l = 0, r = 0, tlo = 0, thi = -1, t1 = 0;
                unsigned thr = 0;
                DenseRow<T, LAYOUT> row{su, kr64, fx, kd, N, p.hoff, p.log2C, 0, 0};
                if (has) {
                    if (over) { l = x / NR; r = x - l * NR; l += l0; }
                    else { const unsigned e = queue[1 + x]; l = (int)(e >> 16); r = (int)(e & 0xffffu); }
                    const OFF *ql = tt + l * p.tp;
                    // row -1 is row N - 1 one period back; the flat search has none of a
                    // row block's outer rows
                    const int lo = (r > 0) ? r - 1 + ql[r - 1] : (S == kFlat && p.vN) ? 0 : ql[N - 1] - 1;
                    const int hi = (r + 1 < NR) ? r + 1 + ql[r + 1] : (S != kFlat && p.vN) ? NR + ql[NR] : N + ql[0];
                    row.f = fx + l * p.lp + r;
                    row.l = l;
                    row.r = r;
                    tlo = max(lo - r, 0);
                    thi = min(hi - r, weff - 1);
                    t1 = ql[r];
                    thr = row.key(t1) + Key::kThr;
                }
                if (has && (S == kFlat || thi - tlo < kLong)) {
                    unsigned mo = 0xffffffffu;                       // the best of the others
#pragma unroll 4
                    for (int t = tlo; t < t1; ++t) mo = __viaddmin_u32(row.f[t], row.k[t], mo);
#pragma unroll 4
                    for (int t = t1 + 1; t <= thi; ++t) mo = __viaddmin_u32(row.f[t], row.k[t], mo);
                    if (mo <= thr) {
                        ++rescans;
                        Key2 best = key2_max();
                        int bt = t1;
                        row.exact(tlo, thi, 1, thr, best, bt);
                        tt[l * p.tp + r] = (OFF)bt;
                    }
                }
                if constexpr (S != kFlat) {
                    unsigned lng = __ballot_sync(0xffffffffu, has && thi - tlo >= kLong);
                    while (lng) {
                        const int from = __ffs(lng) - 1;
                        lng &= lng - 1;
                        const int wl = __shfl_sync(0xffffffffu, l, from), wr = __shfl_sync(0xffffffffu, r, from);
                        const int w0 = __shfl_sync(0xffffffffu, tlo, from), w1 = __shfl_sync(0xffffffffu, thi, from);
                        const int wt = __shfl_sync(0xffffffffu, t1, from);
                        const unsigned wthr = __shfl_sync(0xffffffffu, thr, from);
                        const DenseRow<T, LAYOUT> wrow{su, kr64, fx + wl * p.lp + wr, kd, N, p.hoff, p.log2C, wl, wr};
                        Key2 best = key2_max();
                        int bt = wt, near = 0;
#pragma unroll 4
                        for (int t = w0 + lane; t <= w1; t += 32) near += (wrow.key(t) <= wthr) ? 1 : 0;
                        if (__reduce_add_sync(0xffffffffu, near) <= 1) continue;
                        wrow.exact(w0 + lane, w1, 32, wthr, best, bt);
                        for (int o = 1; o < 32; o <<= 1) {
                            const Key2 ob = key2_shfl_xor(best, o);
                            const int ot = __shfl_xor_sync(0xffffffffu, bt, o);
                            if (key2_less(ob, best) || (key2_eq(ob, best) && ot < bt)) { best = ob; bt = ot; }
                        }
                        if (lane == from) {
                            ++rescans;
                            tt[wl * p.tp + wr] = (OFF)bt;
                        }
                    }
                }
            }
        }
        gsync();
    }
    {
        const int wr = __reduce_add_sync(0xffffffffu, rescans);
        if (lane == 0 && wr) atomicAdd(&p.counters[CNT_RESCAN], (unsigned long long)wr);
    }
    // ---- exact values, potential term, stores
    pdl_next();
    int edges = 0;
    if constexpr (LAYOUT == LAYOUT_CONTIG) {
        if (cl < tl.valid) {
            long long xb = tl.base + cl * tl.lstride;
            int rows = N;
            if (p.vN) {
                const RowBlock rb = row_block(p, (tile << p.log2C) + cl);
                xb = rb.base;
                rows = rb.rows;
            }
            edges = write_rows_contig<T, OFF>(p, su + cl * N, tt + cl * p.tp, kr64, xb, sub, rows,
                                              lpl);
        }
    } else {
        __syncthreads();
        edges = write_rows_strided<T, OFF, 4>(p, tl, su, tt, kr64);
    }
    count_edges(p, edges);
}

template <typename T, int LAYOUT, int S>
__global__ void __launch_bounds__(dense_threads(S), dense_ctas(S)) pass_kernel_dense_batch(const BatchItem *__restrict__ items, PassParams p,
                                                               long long count)
{
    const unsigned inst = blockIdx.x / (unsigned)p.ntiles;
    const long long tile = blockIdx.x - inst * (unsigned)p.ntiles;
    if ((long long)inst >= count) return;
    const BatchItem *it = items + inst;
    PassParams q = p;
    batch_fields(q, it);
    if (q.use_tma && LAYOUT == LAYOUT_STRIDED && threadIdx.x == 0)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&it->tmap) : "memory");
    dense_tile<T, LAYOUT, unsigned short, S>(&it->tmap, q, tile, nullptr);
}

template <typename T, int LAYOUT, int S>
__global__ void __launch_bounds__(dense_threads(S), dense_ctas(S)) pass_kernel_dense(const __grid_constant__ CUtensorMap tmap,
                                                                                    const __grid_constant__ PassParams p)
{
    const long long tile = blockIdx.x;
    if (tile >= p.ntiles) return;
    dense_tile<T, LAYOUT, unsigned short, S>(&tmap, p, tile, &p);
}

}  // namespace hjlo
