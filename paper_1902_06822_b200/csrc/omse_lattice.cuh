// The error curve of the line search of Section 3.4 from one look at every value.
//
// For a scale alpha and a range with codes 0..L of one sign, rounding x/alpha to the nearest code is counting the
// thresholds (j - 1/2)*alpha, j = 1..L, below |x|, and the squared error is
//     (|x| - alpha*q)^2 = x^2 - 2*alpha * sum_j ( |x| - (j - 1/2)*alpha )_+ .
// On the grid alpha_c = (c+1)*step every threshold is an odd multiple of h = step/2: (2j-1)*(c+1)*h.  With
//     P(m) = sum_i ( |x_i|/h - m )_+ ,   m = 1, 2, ...
// the whole curve is  SSE(c)/h^2 = sum_i (x_i/h)^2 - 4*(c+1) * sum_{j <= L} P((2j-1)*(c+1)),
// and P is the second-order suffix sum of a histogram of |x|/h with unit bins that keeps, per bin, the number of values
// and the sum of their fractional parts.  So the C candidates cost K insertions, a scan of 2C bins and at most L
// look-ups per candidate instead of C*K evaluations of the error.  A value has to be in its own bin: one at m + d that is put into
// bin m - 1 is missing from P(m) with all of d, 4*(c+1)*d in the error of the candidate c whose threshold m is, and rows whose
// values repeat add that up.  So bins are exact (lattice_bin).
//
// The counts and the fractional sums are integers in shared memory (32-bit shared atomics run at 12 values per clock
// and SM, 64-bit and floating ones are compare-and-swap loops at a fifth of that or less), so the curve does not depend
// on the order of the insertions.  What the fixed point and the rounding of the scales can change is bounded by
// lattice_band(); the candidates within the bound of the smallest value are re-scored exactly by the caller.
//
// Measured on one B200 against a sweep of all candidates over all values that they do not code as 0, 1024 candidates: 4096 x
// 25,088 values in two tensors 7.25 -> 1.41 ms, 2674 x 25,088 on 8 bits 2.43 -> 0.43 ms, 14,563 x 4608 2.38 -> 0.49 ms.
// Short rows are cheaper to search by evaluating some 25 candidates (omse_rows_short.cuh): the 2C bins cost a block as much as a few
// thousand values.  (A warp with a smaller form of the histogram comes out ahead from some 450 values on: hist_search there.)
//
// A signed range has one more code on the negative side: that level's thresholds are the multiples of D*h,
// D = 2*|lo| - 1, and only negative values count; they go to a second, D times coarser histogram.
#pragma once
#include "omse_device.cuh"

namespace omse {

// The threads of the block that works on a row.
struct BlockTeam {
    int t, n;             // this thread's index, their number
    __device__ __forceinline__ int size() const { return n; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// Shared-memory words that the searches of a block team exchange partial results through; every use within a row has
// words of its own, so one barrier between the write and the reads is enough.
constexpr int kTeamWarps = 24;
struct TeamScratch {
    unsigned int amax[kTeamWarps];
    float esum[kTeamWarps];
    union {
        struct { unsigned int scan_n[kTeamWarps], scan_s[kTeamWarps], scan_f[kTeamWarps]; };
        double energy[kTeamWarps];          // direct_begin
    };
    union {
        struct {
            float dmin[2][kTeamWarps];
            int didx[2][kTeamWarps];
            int lo[kTeamWarps], hi[kTeamWarps];
        };
        struct {              // lattice_search_wide, before it looks for the minimum
            double wide_n[kTeamWarps], wide_s[kTeamWarps], wide_e[kTeamWarps];
        };
    };
};

__device__ __forceinline__ unsigned int warp_umax(unsigned int v) { return __reduce_max_sync(0xffffffffu, v); }
template <class V>
__device__ __forceinline__ V warp_allsum(V v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned int team_umax(const BlockTeam& tm, unsigned int v, TeamScratch* ts) {
    v = warp_umax(v);
    if ((tm.t & 31) == 0) ts->amax[tm.t >> 5] = v;
    __syncthreads();
    unsigned int r = 0;
    for (int w = 0; w < (tm.n >> 5); ++w) r = max(r, ts->amax[w]);
    return r;
}
// leaves the team's sum to team_esum_read() after the team's next barrier
__device__ __forceinline__ void team_esum_write(const BlockTeam& tm, float& v, TeamScratch* ts) {
    v = warp_allsum(v);
    if ((tm.t & 31) == 0) ts->esum[tm.t >> 5] = v;
}
__device__ __forceinline__ float team_esum_read(const BlockTeam& tm, float, TeamScratch* ts) {
    float r = 0.f;
    for (int w = 0; w < (tm.n >> 5); ++w) r += ts->esum[w];
    return r;
}
// smallest value and the lowest index that has it (slot: one of two sets of exchange words)
__device__ __forceinline__ void team_argmin(const BlockTeam& tm, float& v, int& idx, TeamScratch* ts, int slot) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
        if (ov < v || (ov == v && oi < idx)) {
            v = ov;
            idx = oi;
        }
    }
    if ((tm.t & 31) == 0) {
        ts->dmin[slot][tm.t >> 5] = v;
        ts->didx[slot][tm.t >> 5] = idx;
    }
    __syncthreads();
    v = ts->dmin[slot][0];
    idx = ts->didx[slot][0];
    for (int w = 1; w < (tm.n >> 5); ++w) {
        const float ov = ts->dmin[slot][w];
        const int oi = ts->didx[slot][w];
        if (ov < v || (ov == v && oi < idx)) {
            v = ov;
            idx = oi;
        }
    }
}

__device__ __forceinline__ void team_range(const BlockTeam& tm, int& lo, int& hi, TeamScratch* ts) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((tm.t & 31) == 0) {
        ts->lo[tm.t >> 5] = lo;
        ts->hi[tm.t >> 5] = hi;
    }
    __syncthreads();
    for (int w = 0; w < (tm.n >> 5); ++w) {
        lo = min(lo, ts->lo[w]);
        hi = max(hi, ts->hi[w]);
    }
}

// The grid of Section 3.4 on a row with max|x| = m, in binary32: alpha_c = fl(fl(c+1)*step), step = fl(fl(hi_frac*m)/fl(C)).
struct Grid {
    float step;
    bool usable;          // some candidate is a normal positive scale
};
__device__ __forceinline__ Grid grid_of(float m, float hi_frac, int n_cand) {
    Grid g;
    g.step = __fdiv_rn(__fmul_rn(hi_frac, m), (float)n_cand);
    g.usable = m > 0.f && __fmul_rn((float)n_cand, g.step) >= FLT_MIN && g.step <= FLT_MAX;
    return g;
}
__device__ __forceinline__ bool usable_scale(float a) { return a >= FLT_MIN && a <= FLT_MAX; }

// What the search of one row needs to know about the launch.
struct LatticeShape {
    int n_cand;
    int n_bins;           // bins m = 1 .. n_bins hold every |x|/h of a row; bin m is word m-1
    float hi_frac;
    int flo, fhi;         // range of the codes
    int window;           // lattice_search_wide: bins per window
    int direct;           // lattice_coarse: lanes per candidate (log2)
};

// Shared memory of the search of one row.
struct LatticeSmem {
    unsigned int* n;      // [max(bins (bins/2 when packed), n_cand)] counts, then the curve (float) of the n_cand candidates
    unsigned int* f;      // [bins] fractional sums, then P
    unsigned int* n2;     // [coarse bins], f2 alike: the same for the extra negative level
    unsigned int* f2;
    float* curve;         // the curve: aliases n, or an array of its own for lattice_search_wide
};
// The counts, a word each or (PACKED; a row has at most 28,672 values) two to a word.  Adding a constant 1 (shared_add1) is what
// shared memory does fastest when many values of a warp meet in one bin (rows of 23,000 values 551 us, packed 585), so packed counts
// are for the rows whose bins would not leave room for a second block on the SM otherwise (of 25,088 values 539 us, 443).
template <bool PACKED>
struct Counts {
    static __host__ __device__ __forceinline__ int words(int bins) { return PACKED ? bins >> 1 : bins; }
    static __device__ __forceinline__ uint4 four(const unsigned int* n, int w) {
        if (!PACKED) return *reinterpret_cast<const uint4*>(n + w);
        const uint2 a = *reinterpret_cast<const uint2*>(n + (w >> 1));
        return make_uint4(a.x & 0xffffu, a.x >> 16, a.y & 0xffffu, a.y >> 16);
    }
};

// Words of the arrays: every thread scans a run of 2^lb >= 16 bins, padded so that all runs are whole.
__host__ __device__ __forceinline__ int lattice_log_run(int bins, int team) {
    int lb = 4;
    while ((team << lb) < bins) ++lb;
    return lb;
}
// (32 words at least: the address swizzle below moves words within aligned groups of 32)
__host__ __device__ __forceinline__ int lattice_padded(int bins, int team) {
    const int lb = lattice_log_run(bins, team), lp = lb < 5 ? 5 : lb;
    return (bins + (1 << lp) - 1) >> lp << lp;
}
// A thread reads its run four words at a time; XOR-ing the run's index into the word address spreads the eight threads
// of a 128-bit access phase over all banks (runs of 16 or more words all start at the same few banks otherwise).
__device__ __forceinline__ int lattice_word(int i, int lb) { return i ^ ((i >> (lb - 2)) & 0x1c); }

struct LatticeResult {
    bool degenerate;      // no usable scale, or a value that is not finite
    bool bad;             // a value is not finite
    float step;
    int best;             // candidate with the smallest value on the curve (lowest index)
    float dmin, band;     // that value; candidates with curve[c] <= band may be the exact minimum
    int lo, hi;           // curve[] holds the coarse candidates (lattice_coarse) and all of [lo, hi]
    int evaluated;        // looks at the row
};

// The candidates that are looked at first: c + 1 = 1 .. 16, then eight per octave, and the last one.
__device__ __forceinline__ int coarse_a1(int i, int n_cand) {
    const int o = (i >> 3) - 2;                                     // octave above 16
    const int a1 = i < 16 ? i + 1 : (16 << o) + (((i & 7) + 1) << (o + 1));
    return min(a1, n_cand);
}
__device__ __forceinline__ int coarse_count(int n_cand) {           // smallest n with coarse_a1(n - 1) = n_cand
    if (n_cand <= 16) return n_cand;
    const int o = 31 - __clz((n_cand - 1) >> 4);                    // 16 << o < n_cand <= 32 << o
    return 16 + 8 * o + ((n_cand - (16 << o) + (2 << o) - 1) >> (o + 1));
}
__device__ __forceinline__ bool lattice_evaluated(const LatticeResult& r, int c, int n_cand) {
    const int a1 = c + 1;
    if ((c >= r.lo && c <= r.hi) || a1 <= 16 || a1 == n_cand) return c < n_cand;
    return (a1 & ((2 << (31 - __clz((a1 - 1) >> 4))) - 1)) == 0 && c < n_cand;
}

// Lower bound of the error between two scales.  With W(alpha) = sum_i sum_j (|x_i| - (j - 1/2)*alpha)_+ the error is
// E - 2*alpha*W, and W is convex and decreasing, so between two scales it lies below the chord of its values there.
// a = c + 1 stands for the scale; w0, w1: 2*step*W at a0 and a1, that is (E - error)/a.
__device__ __forceinline__ float chord_bound_w(float e, float a0, float w0, float a1, float w1) {
    const float slope = __fdividef(w0 - w1, a1 - a0);
    float at = slope > 0.f ? 0.5f * (__fdividef(w0, slope) + a0) : a1;     // where a*(w0 - slope*(a - a0)) is largest
    at = fminf(fmaxf(at, a0), a1);
    return e - at * (w0 - slope * (at - a0));
}
__device__ __forceinline__ float chord_bound(float e, int a0, float v0, int a1, float v1) {
    return chord_bound_w(e, (float)a0, __fdividef(e - v0, (float)a0), (float)a1, __fdividef(e - v1, (float)a1));
}

// Calls f(c) for this thread's share of the candidates that curve[] holds.
template <class F>
__device__ __forceinline__ void lattice_each(const BlockTeam& tm, const LatticeResult& r, int n_cand, F f) {
    for (int c = r.lo + tm.t; c <= r.hi; c += tm.size()) f(c);
    const int n = coarse_count(n_cand);
    for (int i = tm.t; i < n; i += tm.size()) {
        const int c = coarse_a1(i, n_cand) - 1;
        if (c < r.lo || c > r.hi) f(c);
    }
}

// additions to a word of shared memory by its 32-bit address
__device__ __forceinline__ void shared_add(unsigned int at, unsigned int v) { asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory"); }
__device__ __forceinline__ void shared_add1(unsigned int at) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(at) : "memory"); }

// The bin m of a >= h and the remainder r = a - m*h, 0 <= r < h.  inv_up exceeds 1/h by 2.3e-7 to 4.8e-7 of it, so floor(a*inv_up)
// is m or, where it is the bin above, the remainder is negative (a/h < 2^21).  No rounding: r is a multiple of the last place of h.
__device__ __forceinline__ float lattice_inv_up(float inv) { return inv * (1.0f + 3.0e-7f); }
__device__ __forceinline__ float lattice_bin(float a, float h, float inv_up, int& m) {
    const float u = __fmaf_rd(a, inv_up, kMagic), r = fmaf(-(u - kMagic), h, a);    // M + floor
    const bool above = r < 0.f;
    m = magic_int(u) - (above ? 1 : 0);
    return above ? r + h : r;
}

// Most the curve (in units of h^2) can be off by at a candidate that could be the minimum.  T = |x|/h, E = sum T^2.
// A value's fractional part is off by at most 2^-(F+1) (rounding to the fixed point) + 2e-7 (binary32 evaluation), which
// enters sum_j P_j once per level below it, times 4(c+1) <= 4T per level: 4*err*sum T <= 4*err*sqrt(K*E).  The extra
// level's fixed point has D times fewer levels at D times larger T.  P itself is truncated to 2^-s: 4(c+1)*2^-s for at
// most n_bins/(2(c+1)) + 2 levels.  The scale alpha_c differs from (c+1)*step by 2^-24, which moves the error by at most
// 2*2^-24*sqrt(E*SSE) to first order.  The IEEE quotient x/alpha rounds a value within 2^-24*|x| of a threshold to either side; its
// error, half a step squared, moves by 2*alpha*2^-24*|x|, and over the row again by at most 4*2^-24*sqrt(E*SSE).
// st = sqrt(K*E), inv_f = 2^-F, inv_d_f2 = the coarse histogram's 2^-F divided by D.
__device__ __forceinline__ float lattice_band(float dmin, float e, float st, float inv_f, float inv_d_f2, float truncation) {
    const float d = fmaxf(dmin, 0.f) + 1e-6f * e;            // e is a binary32 sum: the curve's zero is known to this
    const float noise = (2.0f * inv_f + 8e-7f + 4.0f * inv_d_f2) * st + truncation +
                        3.6e-7f * sqrtf(d * e) + 1e-9f * e;
    return dmin + (float)kRescoreBand * d + 2.0f * noise;    // both the minimum's and the candidate's value may be off
}

// Suffix scan of the bins [0, padded) of (n, f): afterwards f[word(i)] = P(i+1) in units of 2^-shift.
//   N(i) = sum_{b>=i} n_b,  S(i) = sum_{b>=i} (b-i)*n_b,  F(i) = sum_{b>=i} f_b;  P(i+1) = S(i) + F(i)*2^-fbits.
// The shift is taken as large as the row's total allows (at most fbits).
struct ScanPart {
    unsigned int n, s, f;
};
template <bool PACKED>
__device__ __forceinline__ ScanPart scan_run(const unsigned int* nb, const unsigned int* fb, int first, int run, int lb) {
    ScanPart p = {0u, 0u, 0u};
    for (int q = run - 4; q >= 0; q -= 4) {
        const int w = lattice_word(first + q, lb);
        const uint4 a = Counts<PACKED>::four(nb, w);
        const uint4 b = *reinterpret_cast<const uint4*>(fb + w);
        p.s += p.n;
        p.n += a.w;
        p.s += p.n;
        p.n += a.z;
        p.s += p.n;
        p.n += a.y;
        p.s += p.n;
        p.n += a.x;
        p.f += (b.x + b.y) + (b.z + b.w);
    }
    return p;
}
template <bool PACKED>
__device__ __forceinline__ void scan_write(const unsigned int* nb, unsigned int* fb, int first, int run, int lb, ScanPart p,
                                           int shift, int drop, int mul) {
    // value = ((S*mul) << shift) + (F >> drop)   (drop < 0 shifts left)
    auto put = [&](unsigned int n, unsigned int f) -> unsigned int {
        p.s += p.n;
        p.n += n;
        p.f += f;
        return ((p.s * (unsigned)mul) << shift) + (drop >= 0 ? p.f >> drop : p.f << -drop);
    };
    for (int q = run - 4; q >= 0; q -= 4) {
        const int w = lattice_word(first + q, lb);
        const uint4 a = Counts<PACKED>::four(nb, w);
        uint4 b = *reinterpret_cast<const uint4*>(fb + w);
        b.w = put(a.w, b.w);
        b.z = put(a.z, b.z);
        b.y = put(a.y, b.y);
        b.x = put(a.x, b.x);
        *reinterpret_cast<uint4*>(fb + w) = b;
    }
}
// inclusive suffix over the lanes of a warp; lane l's run starts (run) bins after lane l-1's
__device__ __forceinline__ void scan_warp(ScanPart& p, int lb) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int n = __shfl_down_sync(0xffffffffu, p.n, o);
        const unsigned int s = __shfl_down_sync(0xffffffffu, p.s, o);
        const unsigned int f = __shfl_down_sync(0xffffffffu, p.f, o);
        if (lane + o < 32) {
            p.s += s + ((unsigned)o << lb) * n;
            p.n += n;
            p.f += f;
        }
    }
}
__device__ __forceinline__ ScanPart scan_exclusive(const ScanPart& p) {
    const int lane = threadIdx.x & 31;
    ScanPart x;
    x.n = __shfl_down_sync(0xffffffffu, p.n, 1);
    x.s = __shfl_down_sync(0xffffffffu, p.s, 1);
    x.f = __shfl_down_sync(0xffffffffu, p.f, 1);
    if (lane == 31) x = ScanPart{0u, 0u, 0u};
    return x;
}
// largest shift <= fbits with (P(1) << shift) < 2^32
__device__ __forceinline__ int scan_shift(unsigned int n_tot, unsigned int s_tot, int fbits) {
    return min(fbits, __clz((int)(s_tot + 2u * n_tot + 1u)));
}

template <bool PACKED>
__device__ __forceinline__ int lattice_scan(const BlockTeam& tm, const unsigned int* nb, unsigned int* fb, int padded, int lb,
                                            int fbits, TeamScratch* ts) {
    const int lane = tm.t & 31, warp = tm.t >> 5, nwarp = tm.n >> 5, first = tm.t << lb, run = first < padded ? 1 << lb : 0;
    ScanPart p = scan_run<PACKED>(nb, fb, first, run, lb);
    scan_warp(p, lb);
    if (lane == 0) {
        ts->scan_n[warp] = p.n;
        ts->scan_s[warp] = p.s;
        ts->scan_f[warp] = p.f;
    }
    ScanPart x = scan_exclusive(p);
    __syncthreads();
    ScanPart acc = {0u, 0u, 0u}, mine = {0u, 0u, 0u};
    for (int w = nwarp - 1; w >= 0; --w) {
        if (w == warp) mine = acc;                       // what lies behind this warp's runs
        acc.s = ts->scan_s[w] + acc.s + (32u << lb) * acc.n;
        acc.n += ts->scan_n[w];
        acc.f += ts->scan_f[w];
    }
    const int shift = scan_shift(acc.n, acc.s, fbits);
    x.s += mine.s + ((unsigned)(31 - lane) << lb) * mine.n;
    x.n += mine.n;
    x.f += mine.f;
    scan_write<PACKED>(nb, fb, first, run, lb, x, shift, fbits - shift, 1);
    return shift;
}

// fixed-point bits of a row's fractional sums: k values of less than 1.01 each stay below 2^31
__device__ __forceinline__ int lattice_fbits(long long terms) {
    return max(0, min(20, 30 - (64 - __clzll(terms - 1))));
}

// Puts the row's values into the histograms; returns this thread's share of sum T^2.
// Bound: the two atomics (eight clocks each for a warp's random words) and instruction issue.  Per value: the bin (M - 1 + m by one
// rounded-down multiply-add, so that its low bits are the word's index and no integer is formed), the remainder, two atomics at
// addresses that come out of the float's bits by a shift and an addition that wraps; one test in four values for those that the
// reciprocal put into the bin above.  With the codes of the passes four at a time: 2674 rows of 25,088 values on 8 bits 427 -> 416 us,
// two tensors of 4 bits 1411 -> 1377.
template <bool PACKED, bool TINY>
__device__ __forceinline__ float lattice_insert(const BlockTeam& tm, const LatticeSmem& sm, const float4* xs4, int k4, float step,
                                                bool sgn, int n_bins, int lb, int fbits, int d, int n_bins2, int lb2, int f2bits) {
    const float pre = TINY ? 18446744073709551616.0f : 1.0f;       // 2^64: keeps 1/h finite for the smallest steps
    const float h = __fmul_rn(__fmul_rn(step, pre), 0.5f);
    const float inv = __fdiv_rn(1.0f, h);
    const float inv_up = lattice_inv_up(inv);
    const float inv_fix = inv * (float)(1 << fbits);
    const unsigned int rd = d > 0 ? (unsigned)((0x100000000ull + d - 1) / d) : 0u;   // m/d = (m*rd) >> 32 for m < 2^24
    const int d_from = d > 0 ? d : 0x7fffffff;
    constexpr float kBase = kMagic - 1.0f;
    constexpr unsigned int kBits = 0x4B400000u;                     // of M: bin 1, word 0
    const unsigned int n_at = (unsigned)__cvta_generic_to_shared(sm.n), f_at = (unsigned)__cvta_generic_to_shared(sm.f) - 4u * kBits;
    const u64 inv2 = pack2(inv, inv), zero2 = pack2(-0.f, -0.f), pre2 = pack2(pre, pre);
    u64 e2 = 0ull;
    for (int i4 = tm.t; i4 < k4; i4 += tm.size()) {
        float4 v = xs4[i4];
        u64 ya = pack2(v.x, v.y), yb = pack2(v.z, v.w);
        if (TINY) {
            ya = fma2(ya, pre2, zero2);
            yb = fma2(yb, pre2, zero2);
            unpack2(ya, v.x, v.y);
            unpack2(yb, v.z, v.w);
        }
        const u64 ta = fma2(ya, inv2, zero2), tb = fma2(yb, inv2, zero2);
        e2 = fma2(tb, tb, fma2(ta, ta, e2));
        const float y[4] = {v.x, v.y, v.z, v.w};
        float u[4], r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = sgn ? fabsf(y[j]) : y[j];               // an unsigned range codes negative values as 0
            u[j] = __fmaf_rd(a, inv_up, kBase);
            r[j] = fmaf(-(u[j] - kBase), h, a);
        }
        if (fminf(fminf(fminf(r[0], r[1]), r[2]), r[3]) < 0.f) {    // below an edge by a few 1e-7
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (r[j] < 0.f) {
                    r[j] += h;
                    u[j] -= 1.0f;
                }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (TINY) u[j] = fminf(u[j], kBase + (float)n_bins);    // (a subnormal step is off by more than the last bin allows for)
            if (!(u[j] >= kMagic)) continue;                        // below the first bin
            const unsigned int bits = __float_as_uint(u[j]), w = bits ^ ((bits >> (lb - 2)) & 0x1cu);      // lattice_word of the index
            const unsigned int fi = __float_as_uint(fmaf(r[j], inv_fix, kMagic)) - kBits;
            if (PACKED) shared_add(n_at + ((w >> 1) << 2) - 2u * kBits, 1u << ((w & 1u) << 4));
            else shared_add1(n_at + (w << 2) - 4u * kBits);
            shared_add(f_at + (w << 2), fi);
            const int m = (int)(bits - kBits) + 1;
            if (y[j] < 0.f && m >= d_from) {
                const unsigned int m2 = __umulhi((unsigned)m, rd);
                const unsigned int rem = (unsigned)m - m2 * (unsigned)d;
                const int w2 = lattice_word(min((int)m2, n_bins2) - 1, lb2);
                atomicAdd(sm.n2 + w2, 1u);
                atomicAdd(sm.f2 + w2, (rem << f2bits) + (fi >> (fbits - f2bits)));
            }
        }
    }
    float ea, eb;
    unpack2(e2, ea, eb);
    return ea + eb;
}

// sum over the levels first, first + stride, ... of P at candidate c (a1 = c+1), in units of 2^-shift
__device__ __forceinline__ unsigned long long lattice_levels(const LatticeSmem& sm, int a1, int levels, int n_bins, int lb,
                                                             int n_bins2, int lb2, int first, int stride) {
    unsigned long long acc = 0ull;
    const int last = min(n_bins, (2 * levels - 1) * a1);
    for (int m = (2 * first + 1) * a1; m <= last; m += 2 * stride * a1) acc += sm.f[lattice_word(m - 1, lb)];
    if (first == 0 && a1 <= n_bins2) acc += sm.f2[lattice_word(a1 - 1, lb2)];
    return acc;
}
__device__ __forceinline__ double u52_double(unsigned long long v) {       // exact for v < 2^52
    return __hiloint2double(0x43300000 + (int)(v >> 32), (int)(unsigned)v) - 4503599627370496.0;
}

// The error curve of the row in xs (k values, zero padded to k4 float4s), its minimum and the band of candidates that the
// caller has to re-score.  amax_bits: this thread's maximum of the bit patterns of |x| over its share of the row.
// Callers must have passed a team barrier since the bins were last used; on return curve[] may be read after the barrier
// that the function ends with.
template <bool PACKED>
__device__ __forceinline__ LatticeResult lattice_search(const BlockTeam& tm, const LatticeShape& g, const LatticeSmem& sm,
                                                        const float4* xs4, int k, int k4, unsigned int amax_bits, TeamScratch* ts) {
    LatticeResult res;
    res.degenerate = true;
    res.bad = false;
    res.best = -1;
    res.step = 0.f;
    res.dmin = res.band = 0.f;
    res.lo = 0;
    res.hi = -1;
    res.evaluated = 1;
    const bool sgn = g.flo < 0;
    const int levels = g.fhi, d = sgn ? 2 * (-g.flo) - 1 : 0;       // common levels, spacing of the extra negative level
    const int n_bins = g.n_bins, lb = lattice_log_run(n_bins, tm.size()), padded = lattice_padded(n_bins, tm.size());
    const int n_bins2 = sgn ? n_bins / d : 0;
    const int lb2 = lattice_log_run(n_bins2, 32), padded2 = n_bins2 > 0 ? lattice_padded(n_bins2, 32) : 0;   // scanned by one warp
    // ---- clear the bins while the maximum is reduced
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tm.t; i < (padded >> 2); i += tm.size()) {
        if (PACKED) reinterpret_cast<uint2*>(sm.n)[i] = make_uint2(0u, 0u);
        else reinterpret_cast<uint4*>(sm.n)[i] = z;
        reinterpret_cast<uint4*>(sm.f)[i] = z;
    }
    for (int i = tm.t; i < (padded2 >> 2); i += tm.size()) {
        reinterpret_cast<uint4*>(sm.n2)[i] = z;
        reinterpret_cast<uint4*>(sm.f2)[i] = z;
    }
    const unsigned int mb = team_umax(tm, amax_bits, ts);
    const float m = __uint_as_float(mb);
    const Grid gr = grid_of(m, g.hi_frac, g.n_cand);
    res.bad = mb >= 0x7f800000u;
    if (res.bad || !gr.usable) return res;                          // not finite, or no usable scale
    res.step = gr.step;
    // ---- histogram
    const int fbits = lattice_fbits(k), f2bits = min(fbits, lattice_fbits((long long)k * max(d, 1)));
    const bool tiny = !(gr.step > 1e-30f);
    float e = tiny ? lattice_insert<PACKED, true>(tm, sm, xs4, k4, gr.step, sgn, n_bins, lb, fbits, n_bins2 > 0 ? d : 0, n_bins2, lb2, f2bits)
                   : lattice_insert<PACKED, false>(tm, sm, xs4, k4, gr.step, sgn, n_bins, lb, fbits, n_bins2 > 0 ? d : 0, n_bins2, lb2, f2bits);
    team_esum_write(tm, e, ts);
    tm.sync();
    e = team_esum_read(tm, e, ts);
    // ---- P
    const int shift = lattice_scan<PACKED>(tm, sm.n, sm.f, padded, lb, fbits, ts);
    if (n_bins2 > 0 && (tm.t >> 5) == (tm.size() >> 5) - 1) {       // the coarse histogram: one warp
        const int lane = tm.t & 31, first = lane << lb2, run = first < padded2 ? 1 << lb2 : 0;
        ScanPart p = scan_run<false>(sm.n2, sm.f2, first, run, lb2);
        scan_warp(p, lb2);
        scan_write<false>(sm.n2, sm.f2, first, run, lb2, scan_exclusive(p), shift, f2bits - shift, d);
    }
    tm.sync();
    // ---- the curve.  W = sum_j P((2j-1)*(c+1)) is convex and decreasing in c, so between two candidates it lies below
    //      the chord, which bounds the curve from below; only the stretch of the grid where that bound does not exclude
    //      the minimum is evaluated candidate by candidate (a tenth of the grid, say).
    const double ed = (double)e, scale = -4.0 * __longlong_as_double((long long)(1023 - shift) << 52);
    float bv = INFINITY;
    int bi = 0x7fffffff;
    auto value = [&](int c, unsigned long long p) {
        float v = (float)fma(scale * int_double(c + 1), u52_double(p), ed);
        if (!usable_scale(__fmul_rn((float)(c + 1), gr.step))) v = INFINITY;
        sm.curve[c] = v;
        if (v < bv || (v == bv && c < bi)) {
            bv = v;
            bi = c;
        }
    };
    auto evaluate = [&](int c) { value(c, lattice_levels(sm, c + 1, levels, n_bins, lb, n_bins2, lb2, 0, 1)); };
    const int n_coarse = coarse_count(g.n_cand);
    // (a few candidates per thread are evaluated sooner than they are bounded: two barriers of the team)
    const bool all = g.n_cand <= 8 * tm.size();
    int done = 0;
    if (levels > 8) {           // the smallest scales have the most levels below max|x|: eight threads share each of them
        done = min(16, g.n_cand);
        for (int i0 = 0; i0 < 8 * done; i0 += tm.size()) {
            const int i = i0 + tm.t, a1 = (i >> 3) + 1;
            unsigned long long p = 0ull;
            if (a1 <= done) p = lattice_levels(sm, a1, levels, n_bins, lb, n_bins2, lb2, i & 7, 8);
            p += __shfl_xor_sync(0xffffffffu, p, 1);
            p += __shfl_xor_sync(0xffffffffu, p, 2);
            p += __shfl_xor_sync(0xffffffffu, p, 4);
            if (a1 <= done && (i & 7) == 0) value(a1 - 1, p);
        }
    }
    if (all) {
        for (int c = done + tm.t; c < g.n_cand; c += tm.size()) evaluate(c);
    } else {
        for (int i = done + tm.t; i < n_coarse; i += tm.size()) evaluate(coarse_a1(i, g.n_cand) - 1);
    }
    float cv = bv;
    int ci = bi;
    team_argmin(tm, cv, ci, ts, 0);
    if (ci == 0x7fffffff) return res;
    const float q = __int_as_float((127 - shift) << 23), qn = (2.0f * (float)n_bins + 8.0f * (float)g.n_cand) * q;
    const float st = sqrtf((float)k * e), inv_f = __int_as_float((127 - fbits) << 23);
    const float inv_d = n_bins2 > 0 ? __int_as_float((127 - f2bits) << 23) / (float)d : 0.f;
    int lo = 0, hi = g.n_cand - 1;
    if (!all) {
        const float keep = lattice_band(cv, e, st, inv_f, inv_d, qn) + 2.0f * qn + 1e-6f * e;   // 1e-6: binary32 in the bound below
        lo = g.n_cand;
        hi = -1;
        for (int i = tm.t; i + 1 < n_coarse; i += tm.size()) {
            const int a0 = coarse_a1(i, g.n_cand), a1 = coarse_a1(i + 1, g.n_cand);
            if (a1 - a0 < 2) continue;
            if (!(chord_bound(e, a0, sm.curve[a0 - 1], a1, sm.curve[a1 - 1]) > keep)) {       // (an unusable end keeps the interval)
                lo = min(lo, a0);
                hi = max(hi, a1 - 2);
            }
        }
        team_range(tm, lo, hi, ts);
        for (int c = lo + tm.t; c <= hi; c += tm.size()) evaluate(c);
        team_argmin(tm, bv, bi, ts, 1);
        cv = bv;
        ci = bi;
    }
    res.degenerate = false;
    res.best = ci;
    res.dmin = cv;
    res.lo = lo;
    res.hi = hi;
    res.band = lattice_band(cv, e, st, inv_f, inv_d, qn);
    return res;
}

// The same for grids whose bins do not fit in shared memory at once (many candidates with a grid that ends far below
// max|x|): the bins are taken in windows from the top down, positive and negative values in turn, each window with an
// insertion pass of its own; values above the last threshold are summed in registers.  P is kept in binary32 and the
// curve is added up in binary32, so the band is wider than above.  For long rows and a few windows (see launch_rows).
__device__ __forceinline__ LatticeResult lattice_search_wide(const BlockTeam& tm, const LatticeShape& g, const LatticeSmem& sm,
                                                             const float4* xs4, int k, int k4, unsigned int amax_bits, TeamScratch* ts) {
    LatticeResult res;
    res.degenerate = true;
    res.bad = false;
    res.best = -1;
    res.step = 0.f;
    res.dmin = res.band = 0.f;
    res.lo = 0;
    res.hi = -1;
    res.evaluated = 1;
    const int lane = tm.t & 31, warp = tm.t >> 5, nwarp = tm.n >> 5;
    const unsigned int mb = team_umax(tm, amax_bits, ts);
    const float m_abs = __uint_as_float(mb);
    const Grid gr = grid_of(m_abs, g.hi_frac, g.n_cand);
    res.bad = mb >= 0x7f800000u;
    if (res.bad || !gr.usable) return res;
    res.step = gr.step;
    const bool tiny = !(gr.step > 1e-30f);
    const float pre = tiny ? 18446744073709551616.0f : 1.0f;
    const float h = __fmul_rn(__fmul_rn(gr.step, pre), 0.5f), inv = __fdiv_rn(1.0f, h), inv_up = lattice_inv_up(inv);
    const int fbits = lattice_fbits(k);
    const float inv_fix = inv * (float)(1 << fbits);
    const int win = g.window, lb = lattice_log_run(win, tm.n), padded = lattice_padded(win, tm.n);
    const int n_bins = g.n_bins, n_win = (n_bins + win - 1) / win;      // (2,084,864 bins at most)
    const float far = (float)(n_bins + 2);
    const double inv_d = 1.0 / (double)h;
    for (int c = tm.t; c < g.n_cand; c += tm.n) sm.curve[c] = 0.f;      // explained share of E, per candidate
    double e_inv = 0.0, root = 0.0;
    int windows = 0;
    for (int side = 0; side < (g.flo < 0 ? 2 : 1); ++side) {
        const int levels = side == 0 ? g.fhi : -g.flo;
        const float sg = side == 0 ? pre : -pre;
        // values beyond the last bin: number and sum of T - (n_bins + 1), the state of the scan above the top window
        double e = 0.0, over_n = 0.0, over_s = 0.0;
        for (int i4 = tm.t; i4 < k4; i4 += tm.n) {
            const float4 v = xs4[i4];
            const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float a = x[j] * sg;
                const double t = (double)a * inv_d;                // (may leave binary32: the grid can end anywhere below max|x|)
                e = fma(t, t, e);
                const float td = a * inv_up;                       // not below |x|/h, and above it by less than a bin
                if (td >= (float)(n_bins + 1)) {
                    int m = n_bins + 1;
                    if (td < far) lattice_bin(a, h, inv_up, m);
                    if (m > n_bins) {
                        over_n += 1.0;
                        over_s += t - (double)(n_bins + 1);
                    }
                }
            }
        }
        e = warp_sum(e);
        over_n = warp_sum(over_n);
        over_s = warp_sum(over_s);
        __syncthreads();
        if (lane == 0) {
            ts->wide_n[warp] = over_n;
            ts->wide_s[warp] = over_s;
            ts->wide_e[warp] = e;
        }
        __syncthreads();
        double cn = 0.0, cs = 0.0, cf = 0.0, et = 0.0;   // N, S, F of the scan at bin `pos`
        long long pos = n_bins + 1;
        for (int w = 0; w < nwarp; ++w) {
            cn += ts->wide_n[w];
            cs += ts->wide_s[w];
            et += ts->wide_e[w];
        }
        e_inv = 1.0 / et;
        root = sqrt(e_inv);                                        // P is kept as P/sqrt(E): at most sqrt(K)
        for (int wi = n_win - 1; wi >= 0; --wi) {
            const int base = wi * win;                             // bins m = base+1 .. base+win
            ++windows;
            __syncthreads();
            for (int i = tm.t; i < padded; i += tm.n) sm.n[i] = sm.f[i] = 0u;
            __syncthreads();
            for (int i4 = tm.t; i4 < k4; i4 += tm.n) {
                const float4 v = xs4[i4];
                const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float a = x[j] * sg, td = a * inv_up;
                    if (!(td >= (float)(base + 1) && td < (float)(base + win + 2) && td < far)) continue;
                    int m;
                    const float r = lattice_bin(a, h, inv_up, m);
                    if (m > base && m <= base + win && m <= n_bins) {
                        const int w = lattice_word(m - 1 - base, lb);
                        atomicAdd(sm.n + w, 1u);
                        atomicAdd(sm.f + w, (unsigned)magic_int(fmaf(r, inv_fix, kMagic)));
                    }
                }
            }
            __syncthreads();
            const int first = tm.t << lb, run = first < padded ? 1 << lb : 0;
            ScanPart p = scan_run<false>(sm.n, sm.f, first, run, lb);
            scan_warp(p, lb);
            if (lane == 0) {
                ts->scan_n[warp] = p.n;
                ts->scan_s[warp] = p.s;
                ts->scan_f[warp] = p.f;
            }
            const ScanPart x = scan_exclusive(p);
            __syncthreads();
            // the state moved to the end of the last thread's run (sum of T - position is linear in the position)
            double an = cn, as = cs - (double)((long long)base + ((long long)tm.n << lb) + 1 - pos) * cn, af = cf;
            double mn = 0.0, ms = 0.0, mf = 0.0;
            for (int w = nwarp - 1; w >= 0; --w) {
                if (w == warp) {
                    mn = an;
                    ms = as;
                    mf = af;
                }
                as += (double)ts->scan_s[w] + (double)(32 << lb) * an;
                an += (double)ts->scan_n[w];
                af += (double)ts->scan_f[w];
            }
            cn = an;                                               // the next window continues from this one's first bin
            cs = as;
            cf = af;
            pos = base + 1;
            const double fq = __longlong_as_double((long long)(1023 - fbits) << 52);
            double dn = (double)x.n + mn, ds = (double)x.s + ms + (double)((31 - lane) << lb) * mn, df = (double)x.f + mf;
            for (int i = run - 1; i >= 0; --i) {
                const int w = lattice_word(first + i, lb);
                ds += dn;
                dn += (double)sm.n[w];
                df += (double)sm.f[w];
                reinterpret_cast<float*>(sm.f)[w] = (float)(fma(df, fq, ds) * root);
            }
            __syncthreads();
            const int top = min(base + win, n_bins);
            for (int c = tm.t; c < g.n_cand; c += tm.n) {
                const int a1 = c + 1;
                int j = (base + a1) / (2 * a1) + 1;                // smallest j with (2j-1)*a1 > base
                double acc = 0.0;
                for (; j <= levels && (2 * j - 1) * a1 <= top; ++j)
                    acc += (double)reinterpret_cast<const float*>(sm.f)[lattice_word((2 * j - 1) * a1 - 1 - base, lb)];
                sm.curve[c] += (float)(4.0 * (double)a1 * acc * root);
            }
        }
    }
    float bv = INFINITY;
    int bi = 0x7fffffff;
    for (int c = tm.t; c < g.n_cand; c += tm.n) {
        float v = 1.0f - sm.curve[c];
        if (!usable_scale(__fmul_rn((float)(c + 1), gr.step))) v = INFINITY;
        sm.curve[c] = v;
        if (v < bv) {
            bv = v;
            bi = c;
        }
    }
    team_argmin(tm, bv, bi, ts, 0);
    if (bi == 0x7fffffff) return res;
    res.degenerate = false;
    res.best = bi;
    res.dmin = bv;
    res.lo = 0;
    res.hi = g.n_cand - 1;
    res.band = lattice_band(bv, 1.0f, (float)sqrt((double)k * e_inv), __int_as_float((127 - fbits) << 23), 0.f, 0.f) +
               1.2e-7f * (float)(windows + 4);
    return res;
}

// -------------------------------------------------------------------------------------------------
// The same without a histogram, by evaluating candidates: for rows of so few values that clearing and scanning 2C bins costs more
// (lattice_coarse), and for grids that end so far below max|x| that their bins would take many windows (lattice_split).
// -------------------------------------------------------------------------------------------------
// team_argmin for values that are not negative (nor NaN): they order like their bit patterns
__device__ __forceinline__ void team_argmin_error(const BlockTeam& tm, float& v, int& idx, TeamScratch* ts, int slot) {
    const unsigned int least = __reduce_min_sync(0xffffffffu, __float_as_uint(v));
    idx = __reduce_min_sync(0xffffffffu, __float_as_uint(v) == least ? idx : 0x7fffffff);
    v = __uint_as_float(least);
    if ((tm.t & 31) == 0) {
        ts->dmin[slot][tm.t >> 5] = v;
        ts->didx[slot][tm.t >> 5] = idx;
    }
    __syncthreads();
    for (int w = 0; w < (tm.n >> 5); ++w) {
        const float ov = ts->dmin[slot][w];
        const int oi = ts->didx[slot][w];
        if (ov < v || (ov == v && oi < idx)) {
            v = ov;
            idx = oi;
        }
    }
}
template <bool SCALED>
__device__ __forceinline__ float direct_part(const float4* xs4, int k4, int first, int stride, float al, float sc, float flo, float fhi) {
    const float inv = __fdiv_rn(1.0f, al), clo = kMagic + flo, chi = kMagic + fhi;
    const u64 M2 = pack2(kMagic, kMagic), NM2 = pack2(-kMagic, -kMagic), inv2 = pack2(inv, inv), na2 = pack2(-al, -al), sc2 = pack2(sc, sc),
              z2 = pack2(-0.f, -0.f);
    auto pair = [&](u64 x, u64 acc) {
        if (SCALED) x = fma2(x, sc2, z2);
        float a, b;
        unpack2(fma2(x, inv2, M2), a, b);
        const u64 d = fma2(na2, add2(pack2(fminf(fmaxf(a, clo), chi), fminf(fmaxf(b, clo), chi)), NM2), x);
        return fma2(d, d, acc);
    };
    u64 total = 0ull;
    for (int i = first; i < k4;) {                          // folds of 128 values: rounding noise near 1e-7
        const int stop = min(k4, i + kFlushEvery4 * stride);
        u64 acc_a = 0ull, acc_b = 0ull;
#pragma unroll 4
        for (; i < stop; i += stride) {
            const float4 v = xs4[i];
            acc_a = pair(pack2(v.x, v.y), acc_a);
            acc_b = pair(pack2(v.z, v.w), acc_b);
        }
        total = add2(total, add2(acc_a, acc_b));
    }
    float a, b;
    unpack2(total, a, b);
    return a + b;
}

// Grid, scaling and energy of a row; false where there is nothing to search.
struct DirectRow {
    float step, sc;       // sc: a power of two that keeps squares in binary32
    __device__ __forceinline__ float scale(int c) const { return fmaxf(__fmul_rn((float)(c + 1), step) * sc, FLT_MIN); }
    __device__ __forceinline__ bool usable(int c) const { return usable_scale(__fmul_rn((float)(c + 1), step)); }
};
__device__ __forceinline__ bool direct_begin(const BlockTeam& tm, const LatticeShape& g, const float4* xs4, int k4, unsigned int amax_bits,
                                             TeamScratch* ts, LatticeResult& res, DirectRow& row) {
    res.degenerate = true;
    res.best = -1;
    res.step = 0.f;
    res.dmin = res.band = 0.f;
    res.lo = 0;
    res.hi = -1;
    res.evaluated = 0;
    const unsigned int mb = team_umax(tm, amax_bits, ts);
    const Grid gr = grid_of(__uint_as_float(mb), g.hi_frac, g.n_cand);
    res.bad = mb >= 0x7f800000u;
    if (res.bad || !gr.usable) return false;
    res.step = row.step = gr.step;
    const int ex = (int)(mb >> 23) - 127;
    row.sc = ex < -40 || ex > 40 ? __int_as_float((127 - max(min(ex, 126), -126)) << 23) : 1.0f;
    double e = 0.0;                                         // the warps' sums now, the row's after the next barrier
    for (int i = tm.t; i < k4; i += tm.n) {
        const float4 v = xs4[i];
        const float y[4] = {v.x * row.sc, v.y * row.sc, v.z * row.sc, v.w * row.sc};
#pragma unroll
        for (int u = 0; u < 4; ++u) e = fma((double)y[u], (double)y[u], e);
    }
    e = warp_sum(e);
    if ((tm.t & 31) == 0) ts->energy[tm.t >> 5] = e;
    return true;
}
__device__ __forceinline__ double direct_energy(const BlockTeam& tm, const TeamScratch* ts) {
    double e = 0.0;
    for (int w = 0; w < (tm.n >> 5); ++w) e += ts->energy[w];
    return e;
}
__device__ __forceinline__ float direct_error(const float4* xs4, int k4, int first, int stride, const DirectRow& r, int c, int flo, int fhi) {
    return r.sc != 1.0f ? direct_part<true>(xs4, k4, first, stride, r.scale(c), r.sc, (float)flo, (float)fhi)
                        : direct_part<false>(xs4, k4, first, stride, r.scale(c), r.sc, (float)flo, (float)fhi);
}

// The coarse candidates, then all of the stretch of the grid that the chords between them leave open.  2^lanes neighbouring lanes
// share a candidate: with fewer lanes there are more candidates under way than are wanted, with more the short rows leave lanes
// without values.
__device__ __forceinline__ LatticeResult lattice_coarse(const BlockTeam& tm, const LatticeShape& g, float* curve, const float4* xs4, int k4,
                                                        unsigned int amax_bits, TeamScratch* ts) {
    LatticeResult res;
    DirectRow row;
    if (!direct_begin(tm, g, xs4, k4, amax_bits, ts, res, row)) return res;
    const int lanes = g.direct, groups = tm.n >> lanes, group = tm.t >> lanes, j = tm.t & ((1 << lanes) - 1);
    float bv = INFINITY;
    int bi = 0x7fffffff;
    auto evaluate = [&](int c, bool wanted) {               // every lane of the warp takes part
        float v = direct_error(xs4, wanted ? k4 : 0, j, 1 << lanes, row, c, g.flo, g.fhi);
        for (int o = 1; o < 1 << lanes; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (!row.usable(c)) v = INFINITY;
        if (!wanted || j != 0) return;
        curve[c] = v;
        if (v < bv || (v == bv && c < bi)) {
            bv = v;
            bi = c;
        }
    };
    const int n_coarse = coarse_count(g.n_cand);
    for (int i0 = 0; i0 < n_coarse; i0 += groups)
        evaluate(coarse_a1(min(i0 + group, n_coarse - 1), g.n_cand) - 1, i0 + group < n_coarse);
    float cv = bv;
    int ci = bi;
    team_argmin_error(tm, cv, ci, ts, 0);
    if (ci == 0x7fffffff) return res;                       // every error is Inf
    const float e = (float)direct_energy(tm, ts), keep = cv * 1.00001f + 2e-6f * e;    // binary32 in the sums and in the bound
    int lo = g.n_cand, hi = -1;
    for (int i = tm.t; i + 1 < n_coarse; i += tm.n) {
        const int a0 = coarse_a1(i, g.n_cand), a1 = coarse_a1(i + 1, g.n_cand);
        if (a1 - a0 >= 2 && !(chord_bound(e, a0, curve[a0 - 1], a1, curve[a1 - 1]) > keep)) {      // (an unusable end keeps the interval)
            lo = min(lo, a0);
            hi = max(hi, a1 - 2);
        }
    }
    team_range(tm, lo, hi, ts);
    for (int c0 = lo; c0 <= hi; c0 += groups) evaluate(min(c0 + group, hi), c0 + group <= hi);
    team_argmin_error(tm, bv, bi, ts, 1);
    res.degenerate = false;
    res.best = bi;
    res.dmin = bv;
    res.lo = lo;
    res.hi = hi;
    res.evaluated = n_coarse + max(0, hi - lo + 1);
    res.band = bv * (1.0f + (float)kRescoreBand);
    return res;
}

// The powers of two of the grid, then splits of the intervals that their chord leaves open, near the minimum of its bound, depth
// first (as in omse_rows_short.cuh): 30 to 60 evaluations by the whole block, one after the other, whatever C is.  The chords are
// drawn in binary64 at the binary32 scales themselves, since the errors of fine grids are a millionth of E.
// stack: kSplitSlots entries; a split leaves at most three quarters of an interval, below the fifth half.
struct __align__(16) SplitPoint {
    double w;             // (E - error)/scale
    int c;
    float v;
};
constexpr int kSplitSlots = 48, kSplitFree = 5;
__device__ __forceinline__ LatticeResult lattice_split(const BlockTeam& tm, const LatticeShape& g, float* curve, SplitPoint* stack, const float4* xs4,
                                                       int k4, unsigned int amax_bits, TeamScratch* ts) {
    LatticeResult res;
    DirectRow row;
    if (!direct_begin(tm, g, xs4, k4, amax_bits, ts, res, row)) return res;
    for (int c = tm.t; c < g.n_cand; c += tm.n) curve[c] = INFINITY;
    __syncthreads();
    const double e = direct_energy(tm, ts);
    const int nwarp = tm.n >> 5;
    float cv = INFINITY;
    int ci = 0x7fffffff, slot = 0;
    auto evaluate = [&](int c) -> SplitPoint {              // the same in all threads
        const float part = warp_allsum(direct_error(xs4, k4, tm.t, tm.n, row, c, g.flo, g.fhi));
        if ((tm.t & 31) == 0) ts->dmin[slot][tm.t >> 5] = part;
        __syncthreads();
        float v = 0.f;
        for (int w = 0; w < nwarp; ++w) v += ts->dmin[slot][w];
        slot ^= 1;
        if (!row.usable(c)) v = INFINITY;
        if (tm.t == 0) curve[c] = v;
        if (v < cv || (v == cv && c < ci)) {
            cv = v;
            ci = c;
        }
        ++res.evaluated;
        return SplitPoint{(e - (double)v) / (double)row.scale(c), c, v};
    };
    const int n_first = 33 - __clz(g.n_cand - 1);           // 2^i below n_cand, and n_cand
    for (int i = 0; i < n_first; ++i) {
        const SplitPoint p = evaluate(min(1 << i, g.n_cand) - 1);
        if (tm.t == 0) stack[i] = p;
    }
    __syncthreads();
    SplitPoint top = stack[n_first - 1];
    int sp = n_first - 2;
    while (sp >= 0) {
        const SplitPoint low = stack[sp];
        const int width = top.c - low.c;
        bool open = width >= 2;
        double at = 0.0;
        if (open) {
            const double a0 = (double)row.scale(low.c), a1 = (double)row.scale(top.c), slope = (low.w - top.w) / (a1 - a0);
            at = slope > 0.0 ? fmin(fmax(0.5 * (low.w / slope + a0), a0), a1) : a1;
            const double bound = e - at * (low.w - slope * (at - a0)), most = (double)fmaxf(low.v, top.v);
            // what the chord has to be above: the best value so far, the noise of the sums, and values on the other side of a
            // threshold (lattice_band); an unusable end keeps the interval
            open = !(bound > (double)cv * 1.00001 + 4e-6 * most + 2.5e-7 * sqrt(e * most) + 1e-12 * e);
            at = (at - a0) / (a1 - a0) * (double)width;
        }
        if (open) {
            const int q = max(1, sp < n_first - 2 + kSplitFree ? width >> 2 : width >> 1);
            const int c = low.c + min(max(__double2int_rn(at), q), width - q);
            const SplitPoint p = evaluate(c);               // (its barrier lies between the reads of the stack above and the write)
            ++sp;
            if (tm.t == 0) stack[sp] = p;
            __syncthreads();
        } else {
            top = low;
            --sp;
        }
    }
    if (ci == 0x7fffffff) return res;                       // every error is Inf
    res.degenerate = false;
    res.best = ci;
    res.dmin = cv;
    res.lo = 0;                                             // the candidates that were not evaluated read as Inf
    res.hi = g.n_cand - 1;
    res.band = cv * (1.0f + (float)kRescoreBand);
    return res;
}

}  // namespace omse
