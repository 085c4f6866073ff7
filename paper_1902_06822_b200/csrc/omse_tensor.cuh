// Per-tensor MMSE scale (Section 3.7, first equation): one scale for a whole activation tensor.
//
// The error curve comes from one histogram of |x|/h, h half a grid step, as for rows (see omse_lattice.cuh), kept in
// binary64 here because the curve is an output: with N(m), P(m) the number and the summed excess of the values above
// m*h,  <x,q> = h*sum_j (P(m_j) + m_j*N(m_j)),  <q,q> = sum_j (2j-1)*N(m_j),  m_j = (2j-1)*(c+1), and
// SSE = sum x^2 - 2*alpha*<x,q> + alpha^2*<q,q> at the binary32 scale alpha.  Candidates near the minimum, and those
// whose error is so small against sum x^2 that the difference loses digits, are re-scored element by element.
//
// A tensor that fits in the shared memory of the GPU goes through one kernel whose blocks keep their slices on chip
// (tensor_resident_kernel).  Larger ones, and grids of many candidates, go through a pipeline of grid-wide kernels
// ordered by the stream:
//   init -> maxima -> histogram -> scan -> levels (<x,q> and <q,q> of every candidate) -> argmin and list of candidates
//   to re-score -> re-score -> polish x R -> final error.
// Grid-wide sums there use "the last block to arrive reduces" (a ticket from atomicAdd, no waiting).
// Measured on one B200 against a sweep of the candidates over the values each does not code as 0: 51,380,224 post-ReLU
// values with 2048 candidates 655 -> 322 us, 25,088 with 50 candidates 53 -> 19 us, 1,605,633 values of both signs with
// offset and 500 candidates 229 -> 33 us.
#pragma once
#include <type_traits>

#include "omse_lattice.cuh"

namespace omse {

constexpr int kHistThreads = 512, kScanThreads = 512, kResidentThreads = 512;
constexpr int kHistChunk = 8160;     // values a block inserts between two folds of its 32-bit words (see hist_put)
constexpr int kHotBins = 32, kHotCopies = 8;   // the first bins are kept in copies: small values come in large numbers
constexpr int kHotWords = kHotBins * kHotCopies;
constexpr double kTinyShare = 1e-8;  // candidates with an error below this share of sum x^2 are re-scored for the curve

struct TensorState {          // lives in the context workspace
    unsigned int mpos_bits, mneg_bits;   // max of positive / negative part as float bits (atomicMax)
    unsigned int ticket;                 // arrivals for last-block reductions (reset by the last block)
    unsigned int bad;                    // a value was not finite
    int best_idx;
    float alpha;
    float step;
    int n_list;                      // candidates to re-score in fp64 (0: the winner of the curve needs none)
    unsigned int n_near;             // values next to an edge of a bin, listed (more than TensorArgs::near_cap: not all of them)
    int first_done;                  // the first polish step came out of the histogram
    int polish_done;                 // set when a polish step stops or reaches a fixed point: later steps return at once
    int key_min, key_max;                // offset mode: order-preserving integer keys of min and max of the tensor
    float delta;                         // offset subtracted from every element (0 without offset)
    double sum_sq;                       // sum x^2
    double near;                         // sum of floor(|x|/h) over the values next to an edge of a bin (see tensor_noise)
    // state N, S, F of the scan at the bin `pos`, below which the next window lies (bins are taken in windows from the top down);
    // windows read one of the two and write the other
    struct Scan {
        double n, s, f;
        long long pos;
    } scan[2];
};

struct TensorArgs {
    const float* x;
    long long n;
    int n_cand;
    float hi_frac;
    int lo, hi;
    int n_bins, n_bins2;    // bins of the fine histogram and of the extra negative level's
    int clipped;            // values above the last bin exist (the grid ends below max|x|)
    int win, win_base;      // this launch's bins: m = win_base+1 .. win_base+win
    int shared_win;         // so many of them, from the first on, are kept in shared memory; the others in the global histogram
    int first_window;       // 1: topmost window (sum x^2, values above the bins and the coarse histogram are taken with it)
    int which;              // parity of the window: the scan state it reads
    TensorState* st;
    unsigned long long* hist;   // [2][win] counts and fractional sums, then [2][n_bins2]
    double* above;          // [2][win] N and P of the window, then [2][n_bins2] (may alias hist)
    double* chunks;         // [n_chunks][3] sums of the chunks of a window
    int n_chunks;
    double* block_sums;     // [grid][kBlockSums]: sum x^2, number and excess of the values above the bins, the same for the coarse
                            // ones, sum of the bins of the values next to an edge (the bits of an integer)
    int n_blocks;           // blocks of the histogram launch
    double* levels;         // [2][n_cand] <x,q>/h and <q,q>
    double* partials;       // passes: [blocks][listed candidates] doubles + [blocks] int64
    long long partial_doubles;   // capacity of `partials`
    int* list;              // [n_cand] candidates to re-score (workspace)
    float* near;            // [near_cap] values next to an edge of a bin, less the offset and times HistGeometry::pre (workspace)
    int near_cap;
    int refine_iters;
    int first_pass;         // polish pass 0, which the histogram may have made unnecessary
    double* curve;          // [n_cand] error per candidate (workspace)
    double* curve_out;      // user copy, nullable
    float* alpha_out;
    float* sse_out;
    int* idx_out;
    float* delta_out;       // offset mode: receives delta; nullptr = no offset
    unsigned long long* evals;   // executed evaluations (instrumentation), nullable
    unsigned int* status;
    unsigned int* status_out;    // receives the status word at the end, nullable
};

__device__ __forceinline__ void tensor_state_init(TensorState* st) {
    st->mpos_bits = 0u;
    st->mneg_bits = 0u;
    st->ticket = 0u;
    st->bad = 0u;
    st->best_idx = -1;
    st->alpha = 0.f;
    st->step = 0.f;
    st->n_list = 0;
    st->n_near = 0u;
    st->first_done = 0;
    st->polish_done = 0;
    st->key_min = 0x7fffffff;
    st->key_max = (int)0x80000000;
    st->delta = 0.f;
    st->sum_sq = 0.0;
    st->near = 0.0;
}
__global__ void tensor_init_kernel(TensorState* st) {
    if (threadIdx.x == 0) tensor_state_init(st);
}

// order-preserving map float -> int (finite values)
__device__ __forceinline__ int float_key(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

// Offset mode (Section 3.1 scheme with offset): delta = min, and the search range is that of the shifted tensor.
__global__ void tensor_offset_kernel(TensorState* st) {
    if (threadIdx.x == 0 && st->key_min <= st->key_max) {
        const float lo = key_float(st->key_min), hi = key_float(st->key_max);
        st->delta = lo;
        st->mpos_bits = __float_as_uint(hi - lo);    // max of fl(x - delta): subtraction is monotone
        st->mneg_bits = 0u;
    }
}

__global__ void __launch_bounds__(256) tensor_absmax_kernel(const float* __restrict__ x, long long n,
                                                             TensorState* st, unsigned int* status,
                                                             unsigned long long* hist, int hist_words) {
    __shared__ double scratch[64];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < hist_words; i += gridDim.x * blockDim.x) hist[i] = 0ull;
    float lo = INFINITY, hi = -INFINITY;          // extremes of the finite values this thread saw
    bool bad = false;
    const long long n4 = n >> 2;
    const float4* x4 = reinterpret_cast<const float4*>(x);
    const long long stride = (long long)gridDim.x * blockDim.x;
    auto one = [&](float e) {
        const bool finite = fabsf(e) <= FLT_MAX;
        bad |= !finite;
        lo = fminf(lo, finite ? e : lo);
        hi = fmaxf(hi, finite ? e : hi);
    };
    auto four = [&](const float4& v) {
        one(v.x);
        one(v.y);
        one(v.z);
        one(v.w);
    };
    // four 128-bit loads in flight per thread before any of them is used
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n4; i += 4 * stride) {
        const float4 v0 = __ldg(x4 + i), v1 = __ldg(x4 + i + stride), v2 = __ldg(x4 + i + 2 * stride),
                     v3 = __ldg(x4 + i + 3 * stride);
        four(v0);
        four(v1);
        four(v2);
        four(v3);
    }
    for (; i < n4; i += stride) four(__ldg(x4 + i));
    for (long long e = (n4 << 2) + (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) one(x[e]);
    // maxima of the positive and of the negative part follow from the extremes (both 0 when nothing finite was seen)
    float mpos = fmaxf(hi, 0.f), mneg = fmaxf(-lo, 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0 && lo <= hi) {   // the warp saw a finite value: integer atomics on order-preserving keys
        atomicMin(&st->key_min, float_key(lo));
        atomicMax(&st->key_max, float_key(hi));
    }
    block_max2(mpos, mneg, scratch);
    if (threadIdx.x == 0) {
        atomicMax(&st->mpos_bits, __float_as_uint(mpos));   // non-negative floats order like their bits
        atomicMax(&st->mneg_bits, __float_as_uint(mneg));
    }
    if (bad) {
        atomicOr(status, 1u);
        atomicOr(&st->bad, 1u);
    }
}

// Bins and fractional parts are exact: h = H*2^e with an integer 2^23 <= H < 2^24, so |x|/h = a/H with a = |x|*2^-e, and a - m*H,
// which fma() forms without rounding, is an integer k for every a >= H.  inv_up exceeds 1/H by 2.3e-7 to 4.8e-7 of it, so
// floor(a*inv_up) is the value's bin m or, for a value just below an edge, the bin above; a negative k tells.
// hist_near: the rare values that need the correction, or lie above an edge by so little that a scale's rounding or the rounding
// of x/alpha could put them below it (1.2e-7*|x|, up to 2.1*m units of k): their bins are added up for tensor_noise.
__device__ __forceinline__ bool hist_near(int k, int m) { return k < 3 * m; }       // (false for a bin below the first)
__device__ __forceinline__ void hist_correct(int& k, int& m, unsigned int hk) {
    if (k < 0) {
        k += (int)hk;
        --m;
    }
}

// hist_put adds one value to bin word `w`: k is spread over two 32-bit words, count and low six bits in the first, the rest
// in the second.  Up to kHistChunk values fit in one bin without overflow (8160*63 < 2^19, 8160 < 2^13,
// 8160*2^18 < 2^32), and an insertion costs two shared-memory atomics instead of three.
__device__ __forceinline__ void hist_put(unsigned int* w1, unsigned int* w2, int w, unsigned int k) {
    atomicAdd(w1 + w, (1u << 19) + (k & 63u));
    atomicAdd(w2 + w, k >> 6);
}
__device__ __forceinline__ unsigned int hist_count(unsigned int a) { return a >> 19; }
__device__ __forceinline__ unsigned long long hist_frac(unsigned int a, unsigned int b) {
    return ((unsigned long long)b << 6) + (a & 0x7ffffu);
}
// Where there are more values per bin, or larger fractions, than that: count, low and high half of k in three words.
__device__ __forceinline__ void hist_put3(unsigned int* c, unsigned int* lo, unsigned int* hi, int w, unsigned int k) {
    atomicAdd(c + w, 1u);
    atomicAdd(lo + w, k & 0xffffu);
    atomicAdd(hi + w, k >> 16);
}

// What the insertions need to know about the grid.
struct HistGeometry {
    float pre, scale, h, inv_up;  // a = |x*pre*scale|, h = H; bin floor(a*inv_up)
    float far;                    // bins from here on are above all histograms
    int sgn, d, d_from, n_bins, n_bins2, base, top, shared_win;
    unsigned long long *far_n, *far_f;   // the window's bins in global memory
    unsigned int rd, hk;          // 2^32/D; H
};
__device__ __forceinline__ HistGeometry hist_geometry(float step, const TensorArgs& a) {
    HistGeometry g;
    g.pre = step > 1e-30f ? 1.0f : 18446744073709551616.0f;      // 2^64: keeps the powers of two finite for the smallest steps
    const int hb = __float_as_int(__fmul_rn(__fmul_rn(step, g.pre), 0.5f));
    g.hk = (hb & 0x7fffff) | 0x800000;
    g.scale = __int_as_float((277 - (hb >> 23)) << 23);           // 2^-e: h*pre = hk*2^e with e = (hb >> 23) - 150
    g.h = (float)g.hk;
    g.inv_up = __fdiv_rn(1.0f, g.h) * (1.0f + 3.0e-7f);           // never below 1/H
    g.sgn = a.lo < 0;
    g.d = a.n_bins2 > 0 ? -2 * a.lo - 1 : 0;
    g.d_from = g.d > 0 ? g.d : 0x7fffffff;
    g.rd = g.d > 0 ? (unsigned)((0x100000000ull + g.d - 1) / g.d) : 0u;
    g.n_bins = a.n_bins;
    g.n_bins2 = a.n_bins2;
    g.base = a.win_base;
    g.top = a.win_base + a.win;
    g.shared_win = a.shared_win;
    g.far_n = a.hist;
    g.far_f = a.hist + a.win;
    g.far = (float)(max(a.n_bins, g.d * (a.n_bins2 + 1)) + 2);    // (2,084,866 at most: 4.8e-7 of it is less than a bin)
    return g;
}
// one unit 2^e in units of h, as the factor of the fractional sums
__device__ __forceinline__ double hist_unit(float step) {
    const float h = __fmul_rn(__fmul_rn(step, step > 1e-30f ? 1.0f : 18446744073709551616.0f), 0.5f);
    return 1.0 / (double)((__float_as_int(h) & 0x7fffff) | 0x800000);
}
struct HistSums {
    double sq, over_n, over_s, over2_n, over2_s;
    long long near;
};
constexpr int kBlockSums = 6;
// Values next to an edge of a bin, on their way to the list of the tensor.  The count is looked at before it is added to: a tensor
// whose values all lie on edges would queue for it.
template <unsigned int CAP>
struct NearList {
    unsigned int n;
    float v[CAP];
    __device__ __forceinline__ void add(float x) {
        if (*(volatile unsigned int*)&n > CAP) return;
        const unsigned int at = atomicAdd(&n, 1u);
        if (at < CAP) v[at] = x;
    }
    // the block's values to the tensor's list, by all threads, between barriers
    __device__ __forceinline__ void flush(unsigned int* n_all, float* all, unsigned int cap, unsigned int& s_at) {
        const unsigned int mine = n;
        if (mine == 0u) return;                             // (the same in all threads)
        if (threadIdx.x == 0) s_at = atomicAdd(n_all, mine > CAP ? cap + 1u : mine);
        __syncthreads();
        const unsigned int at = s_at;
        if (mine <= CAP && at <= cap && mine <= cap - at)
            for (unsigned int i = threadIdx.x; i < mine; i += blockDim.x) all[at + i] = v[i];
    }
};
// Words of a block's histograms.
constexpr unsigned int kHistNear = 1024;
struct HistWords {
    NearList<kHistNear>* near;
    unsigned int *w1, *w2;            // fine window, hot copies first (two-word form)
    unsigned int *c2, *lo2, *hi2;     // coarse histogram (three-word form)
};

// One value, its bin and remainder known, into the words of the fine window (bins base+1 ...) and of the coarse histogram.
__device__ __forceinline__ void hist_put_fine(const HistGeometry& g, const HistWords& w, int i, int k) {
    hist_put(w.w1, w.w2, g.base == 0 && i < kHotBins ? i * kHotCopies + (threadIdx.x & (kHotCopies - 1)) : kHotWords + i, (unsigned)k);
}
__device__ __forceinline__ void hist_put_coarse(const HistGeometry& g, const HistWords& w, int m, int k) {
    const unsigned int m2 = __umulhi((unsigned)m, g.rd), rem = (unsigned)m - m2 * (unsigned)g.d;
    hist_put3(w.c2, w.lo2, w.hi2, min((int)m2, g.n_bins2) - 1, rem * g.hk + (unsigned)k);
}

// The same into the global histogram: the lanes that meet in a bin add once.  Values that repeat would queue for one address (51M
// values, a twelfth of them equal: 3.2 ms, 1.5 so); uniform ones pay for it (0.8 ms, 1.45 so), heavy-tailed ones have few there.
__device__ __forceinline__ void hist_put_far(const HistGeometry& g, int i, int k) {
    const unsigned int peers = __match_any_sync(__activemask(), i);
    const unsigned int sum = __reduce_add_sync(peers, (unsigned)k);            // at most 32*2^24
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) {
        atomicAdd(g.far_n + i, (unsigned long long)__popc(peers));
        atomicAdd(g.far_f + i, (unsigned long long)sum);
    }
}

// Four values x*pre where the window holds all bins and no value lies above them (the common case).  One branch for the rare
// values next to an edge, instead of four.  SIGNED: the range has negative codes; an unsigned one codes negative values as 0.
template <bool SIGNED>
__device__ __forceinline__ void hist_insert4(const float (&x)[4], const HistGeometry& g, const HistWords& w, HistSums& s) {
    float u[4], r[4], least = 0.f;                        // M + bin, remainder (an integer)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float y = x[j] * g.scale, a = SIGNED ? fabsf(y) : y;
        s.sq = fma((double)x[j], (double)x[j], s.sq);
        u[j] = __fmaf_rd(a, g.inv_up, kMagic);
        const float mf = u[j] - kMagic;
        r[j] = fmaf(-mf, g.h, a);
        least = fminf(least, fmaf(-3.0f, mf, r[j]));      // (not negative for a bin below the first)
    }
    if (least < 0.f) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int m = magic_int(u[j]), k = (int)r[j];
            if (m >= 1 && hist_near(k, m)) {
                s.near += m;
                w.near->add(x[j]);
                hist_correct(k, m, g.hk);
                u[j] = kMagic + (float)m;
                r[j] = (float)k;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int m = magic_int(u[j]);
        if (m < 1) continue;
        const int k = __float2int_rz(r[j]);
        hist_put_fine(g, w, min(m, g.n_bins) - 1, k);
        if (SIGNED && x[j] < 0.f && m >= g.d_from) hist_put_coarse(g, w, m, k);
    }
}
// One value x*pre where values may lie above the last bin or outside the window.
template <bool SIGNED>
__device__ __forceinline__ void hist_insert(float x, const HistGeometry& g, const HistWords& w, bool first, HistSums& s) {
    const float y = x * g.scale, a = SIGNED ? fabsf(y) : y, td = a * g.inv_up;
    if (first) s.sq = fma((double)x, (double)x, s.sq);
    if (!(td >= 1.0f)) return;
    int m = 0x7fffffff, k = 0;                            // far above the bins
    if (td < g.far) {
        const float u = __fmaf_rd(a, g.inv_up, kMagic);
        m = magic_int(u);
        k = __float2int_rz(fmaf(-(u - kMagic), g.h, a));
        if (hist_near(k, m)) {
            if (first) s.near += m;
            hist_correct(k, m, g.hk);
            if (m < 1) return;
        }
    }
    if (m > g.n_bins) {
        if (first) {
            s.over_n += 1.0;
            s.over_s += (double)a / (double)g.h - (double)(g.n_bins + 1);
        }
    } else if (m > g.base && m <= g.top) {
        const int i = m - 1 - g.base;
        if (i < g.shared_win) hist_put_fine(g, w, i, k);
        else hist_put_far(g, i, k);
    }
    if (SIGNED && first && x < 0.f && g.d > 0 && m >= g.d) {
        if (m >= g.d * (g.n_bins2 + 1)) {
            s.over2_n += 1.0;
            s.over2_s += (double)a / ((double)g.h * (double)g.d) - (double)(g.n_bins2 + 1);
        } else {
            hist_put_coarse(g, w, m, k);
        }
    }
}

// Histogram of one window of bins.  A block takes chunks of the tensor in turn; after each the 32-bit words are folded into
// the block's 64-bit sums, and at the end those go to the global histogram by integer atomics (any order, same result).
// Bound: one read of the tensor from HBM beside two shared-memory atomics per value (2.7 clocks per warp each).
template <bool FULL, bool SIGNED>
__global__ void __launch_bounds__(kHistThreads, 2) tensor_hist_kernel(const TensorArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double dscratch[64];
    __shared__ NearList<kHistNear> s_near;
    __shared__ unsigned int s_near_at;
    TensorState* st = a.st;
    const int tid = threadIdx.x, swin = a.shared_win, words = kHotWords + swin;         // swin is a multiple of 4
    unsigned long long* acc_f = reinterpret_cast<unsigned long long*>(smem_raw);       // [swin]
    HistWords w;
    w.near = &s_near;
    if (tid == 0) s_near.n = FULL ? 0u : kHistNear + 1u;           // (not listed by windows)
    w.w1 = reinterpret_cast<unsigned int*>(acc_f + swin);
    w.w2 = w.w1 + words;
    w.c2 = w.w2 + words;
    w.lo2 = w.c2 + a.n_bins2;
    w.hi2 = w.lo2 + a.n_bins2;
    unsigned int* acc_n = w.hi2 + a.n_bins2;
    const float m = fmaxf(__uint_as_float(st->mpos_bits), __uint_as_float(st->mneg_bits));
    const Grid gr = grid_of(m, a.hi_frac, a.n_cand);
    HistSums s = {0.0, 0.0, 0.0, 0.0, 0.0, 0ll};
    if (gr.usable && !st->bad) {
        const HistGeometry g = hist_geometry(gr.step, a);
        const float delta = st->delta, off = -delta * g.pre;        // fmaf(x, pre, off) = pre*fl(x - delta): pre is a power of two
        const bool first = a.first_window != 0;
        for (int i = tid; i < 2 * words + 3 * a.n_bins2; i += kHistThreads) w.w1[i] = 0u;      // all words
        for (int i = tid; i < swin; i += kHistThreads) {
            acc_f[i] = 0ull;
            acc_n[i] = 0u;
        }
        const float4* x4 = reinterpret_cast<const float4*>(a.x);
        const long long n4 = a.n >> 2, n4_all = (a.n + 3) >> 2;
        constexpr int chunk4 = kHistChunk / 4, per = (chunk4 + kHistThreads - 1) / kHistThreads;
        float4 v[per];
        auto fetch = [&](long long c0) {                            // this thread's values of a chunk; absent ones read as delta
#pragma unroll
            for (int j = 0; j < per; ++j) {
                const int o = tid + j * kHistThreads;
                v[j] = o < chunk4 && c0 + o < n4 ? __ldg(x4 + c0 + o) : make_float4(delta, delta, delta, delta);
            }
        };
        long long c0 = (long long)blockIdx.x * chunk4;
        if (c0 < n4_all) fetch(c0);
        int coarse_room = 0xffff;                                   // values until the coarse words could overflow
        for (; c0 < n4_all; c0 += (long long)gridDim.x * chunk4) {
            __syncthreads();                                        // words are clear
#pragma unroll
            for (int j = 0; j < per; ++j) {
                const float x[4] = {fmaf(v[j].x, g.pre, off), fmaf(v[j].y, g.pre, off), fmaf(v[j].z, g.pre, off), fmaf(v[j].w, g.pre, off)};
                if (FULL) {
                    hist_insert4<SIGNED>(x, g, w, s);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) hist_insert<SIGNED>(x[e], g, w, first, s);
                }
            }
            if (c0 + (long long)gridDim.x * chunk4 < n4_all) fetch(c0 + (long long)gridDim.x * chunk4);   // next chunk on its way
            if (c0 + chunk4 > n4 && tid < (int)(a.n - 4 * n4)) {    // the last one to three values
                const float x[4] = {fmaf(a.x[4 * n4 + tid], g.pre, off), 0.f, 0.f, 0.f};
                if (FULL) hist_insert4<SIGNED>(x, g, w, s);
                else hist_insert<SIGNED>(x[0], g, w, first, s);
            }
            __syncthreads();
            if (a.win_base == 0 && tid < kHotBins && tid < swin) {
                unsigned int c = 0u;
                unsigned long long f = 0ull;
#pragma unroll
                for (int j = 0; j < kHotCopies; ++j) {
                    const int i = tid * kHotCopies + j;
                    c += hist_count(w.w1[i]);
                    f += hist_frac(w.w1[i], w.w2[i]);
                    w.w1[i] = w.w2[i] = 0u;
                }
                acc_n[tid] += c;
                acc_f[tid] += f;
            }
            const uint4* q1 = reinterpret_cast<const uint4*>(w.w1 + kHotWords);
            for (int b = tid + (a.win_base == 0 ? kHotBins / 4 : 0); b < (swin >> 2); b += kHistThreads) {
                const uint4 q = q1[b];
                if ((q.x | q.y | q.z | q.w) == 0u) continue;        // most bins of a heavy-tailed tensor stay empty
                const unsigned int p[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = 4 * b + e;
                    if (!p[e]) continue;
                    acc_n[i] += hist_count(p[e]);
                    acc_f[i] += hist_frac(p[e], w.w2[kHotWords + i]);
                    w.w1[kHotWords + i] = w.w2[kHotWords + i] = 0u;
                }
            }
            coarse_room -= kHistChunk + 4;
            if (first && a.n_bins2 > 0 && coarse_room < kHistChunk + 4) {
                coarse_room = 0xffff;
                for (int b = tid; b < a.n_bins2; b += kHistThreads)
                    if (w.c2[b]) {
                        atomicAdd(a.hist + 2 * a.win + b, (unsigned long long)w.c2[b]);
                        atomicAdd(a.hist + 2 * a.win + a.n_bins2 + b, ((unsigned long long)w.hi2[b] << 16) + w.lo2[b]);
                        w.c2[b] = w.lo2[b] = w.hi2[b] = 0u;
                    }
            }
        }
        __syncthreads();
        for (int b = tid; b < swin; b += kHistThreads)
            if (acc_n[b]) {
                atomicAdd(a.hist + b, (unsigned long long)acc_n[b]);
                atomicAdd(a.hist + a.win + b, acc_f[b]);
            }
        if (first)
            for (int b = tid; b < a.n_bins2; b += kHistThreads)
                if (w.c2[b]) {
                    atomicAdd(a.hist + 2 * a.win + b, (unsigned long long)w.c2[b]);
                    atomicAdd(a.hist + 2 * a.win + a.n_bins2 + b, ((unsigned long long)w.hi2[b] << 16) + w.lo2[b]);
                }
        s.sq *= 1.0 / ((double)g.pre * (double)g.pre);
        if (first) s_near.flush(&st->n_near, a.near, (unsigned)a.near_cap, s_near_at);
        if (blockIdx.x == 0 && tid == 0 && a.evals && first) atomicAdd(a.evals, (unsigned long long)a.n);
    }
    if (a.first_window) {
        double v[5] = {s.sq, s.over_n, s.over_s, s.over2_n, s.over2_s};
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            long long near = j == 0 ? s.near : 0ll;
            block_sum2(v[j], near, dscratch);
            if (tid == 0) a.block_sums[kBlockSums * blockIdx.x + j] = v[j];
            if (tid == 0 && j == 0) a.block_sums[kBlockSums * blockIdx.x + 5] = __longlong_as_double(near);
        }
    }
}

// Suffix scan of bins 0 .. n-1 of (count, fractional sum) by a block of kScanThreads threads: above_n[i] = N, above_p[i] = P at
// the position of bin i, in units of h.  (cn, cs, cf): the state N, S, F at the position `gap` bins above bin 0, replaced by
// the state at bin 0's position.  `unit` turns fractional sums into units of h.  part: exchange words.
constexpr int kScanHeld = 8;
__device__ __forceinline__ void tensor_scan(const unsigned long long* hn, const unsigned long long* hf, int n, double unit,
                                            double& cn, double& cs, double& cf, double gap, double* above_n, double* above_p,
                                            double (*part)[3]) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = (n + kScanThreads - 1) / kScanThreads, first = tid * run;
    // Runs of up to kScanHeld bins are loaded once and stay in registers (4096 bins; a second trip to L2 is 1500 cycles).
    double hc[kScanHeld], hf8[kScanHeld];
    auto load = [&](int i0) {                               // eight bins' loads in flight
        unsigned long long c[kScanHeld], f[kScanHeld];
#pragma unroll
        for (int j = 0; j < kScanHeld; ++j) {
            const bool in = i0 + j < run && first + i0 + j < n;
            c[j] = in ? __ldcg(hn + first + i0 + j) : 0ull;
            f[j] = in ? __ldcg(hf + first + i0 + j) : 0ull;
        }
#pragma unroll
        for (int j = 0; j < kScanHeld; ++j) {
            hc[j] = (double)c[j];
            hf8[j] = (double)f[j];
        }
    };
    double pn = 0.0, ps = 0.0, pf = 0.0;
    for (int i0 = (run - 1) & ~(kScanHeld - 1); i0 >= 0; i0 -= kScanHeld) {
        load(i0);
#pragma unroll
        for (int j = kScanHeld - 1; j >= 0; --j) {
            if (i0 + j < run) ps += pn;
            pn += hc[j];
            pf += hf8[j];
        }
    }
    // suffix sums over the lanes' runs, then over the warps' (each warp for itself)
    auto suffix = [](double& vn, double& vs, double& vf, int l, int items, int width) {
#pragma unroll
        for (int o = 1; o < items; o <<= 1) {
            const double n2 = __shfl_down_sync(0xffffffffu, vn, o), s2 = __shfl_down_sync(0xffffffffu, vs, o),
                         f2 = __shfl_down_sync(0xffffffffu, vf, o);
            if (l + o < items) {
                vs += s2 + (double)(o * width) * n2;
                vn += n2;
                vf += f2;
            }
        }
    };
    suffix(pn, ps, pf, lane, 32, run);
    __syncthreads();                                        // exchange words free
    if (lane == 0) {
        part[warp][0] = pn;
        part[warp][1] = ps;
        part[warp][2] = pf;
    }
    double xn = __shfl_down_sync(0xffffffffu, pn, 1), xs = __shfl_down_sync(0xffffffffu, ps, 1), xf = __shfl_down_sync(0xffffffffu, pf, 1);
    if (lane == 31) xn = xs = xf = 0.0;
    __syncthreads();
    constexpr int nwarp = kScanThreads / 32;
    double wn = 0.0, ws = 0.0, wf = 0.0;
    if (lane < nwarp) {
        wn = part[lane][0];
        ws = part[lane][1];
        wf = part[lane][2];
    }
    suffix(wn, ws, wf, lane, nwarp, 32 * run);
    // the state above moved to the end of this warp's last run, and to bin 0 (a sum of T - position is linear in the position)
    const int behind = (warp + 1) & 31;                     // (lane 16 and above hold zeros)
    double mn = __shfl_sync(0xffffffffu, wn, behind), ms = __shfl_sync(0xffffffffu, ws, behind), mf = __shfl_sync(0xffffffffu, wf, behind);
    if (warp == nwarp - 1) mn = ms = mf = 0.0;
    ms += cs + ((double)(nwarp - 1 - warp) * (32 * run) - ((double)run * kScanThreads - gap)) * cn;
    mn += cn;
    mf += cf;
    cs += __shfl_sync(0xffffffffu, ws, 0) + gap * cn;
    cn += __shfl_sync(0xffffffffu, wn, 0);
    cf += __shfl_sync(0xffffffffu, wf, 0);
    double dn = xn + mn, ds = xs + ms + (double)((31 - lane) * run) * mn, df = xf + mf;
    for (int i0 = (run - 1) & ~(kScanHeld - 1); i0 >= 0; i0 -= kScanHeld) {
        if (run > kScanHeld) load(i0);
#pragma unroll
        for (int j = kScanHeld - 1; j >= 0; --j) {
            if (i0 + j >= run) continue;
            ds += dn;
            dn += hc[j];
            df += hf8[j];
            if (first + i0 + j < n) {
                above_n[first + i0 + j] = dn;
                above_p[first + i0 + j] = fma(df, unit, ds);
            }
        }
    }
}

// <x,q>/h and <q,q> of candidate c from the window [base, base+win) of N and P, shared by `stride` threads.
__device__ __forceinline__ void tensor_levels(const double* above_n, const double* above_p, int base, int top, int a1, int levels,
                                              int first, int stride, double& sx, double& sq) {
    int j = base > 0 ? (base + a1) / (2 * a1) + first : first;      // (2j+1)*a1 > base
    const int end = min(levels, (top / a1 + 1) >> 1);               // (2j+1)*a1 <= top
#pragma unroll 4
    for (; j < end; j += stride) {
        const int m = (2 * j + 1) * a1;                     // (below 2^21)
        const double nn = above_n[m - 1 - base];
        sx += fma((double)m, nn, above_p[m - 1 - base]);
        sq = fma((double)(2 * j + 1), nn, sq);
    }
}
// Eight threads per candidate; i: this thread among all of them.  Later windows add to what earlier ones left.
__device__ __forceinline__ void tensor_levels_of(const TensorArgs& a, int i) {
    const int c = i >> 3, part = i & 7;
    double sx = 0.0, sq = 0.0;
    if (c < a.n_cand) {
        const int top = min(a.win_base + a.win, a.n_bins);
        tensor_levels(a.above, a.above + a.win, a.win_base, top, c + 1, a.hi, part, 8, sx, sq);
        if (a.first_window && part == 0 && c < a.n_bins2) {
            const double d = (double)(-2 * a.lo - 1), nn = a.above[2 * a.win + c];
            sx += d * (a.above[2 * a.win + a.n_bins2 + c] + (double)(c + 1) * nn);
            sq += d * nn;
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    if (part == 0 && c < a.n_cand) {
        if (!a.first_window) {
            sx += a.levels[c];
            sq += a.levels[a.n_cand + c];
        }
        a.levels[c] = sx;
        a.levels[a.n_cand + c] = sq;
    }
}
__global__ void __launch_bounds__(256) tensor_levels_kernel(const TensorArgs a) { tensor_levels_of(a, blockIdx.x * 256 + threadIdx.x); }

// What the histogram's blocks left beside the bins, by one block: sum x^2, the sum of the values next to an edge, the state of the
// scan above the topmost window, N and P of the coarse bins.
__device__ __forceinline__ void tensor_scan_begin(const TensorArgs& a, double unit, double (*part)[3], double* scratch) {
    double t[kBlockSums - 1];
    long long near = 0;
#pragma unroll
    for (int j = 0; j < kBlockSums - 1; ++j) {             // the blocks' sums, in a fixed order
        t[j] = 0.0;
        for (int b = threadIdx.x; b < a.n_blocks; b += kScanThreads) {
            t[j] += __ldcg(a.block_sums + kBlockSums * b + j);
            if (j == 0) near += __double_as_longlong(__ldcg(a.block_sums + kBlockSums * b + 5));
        }
        long long zero = 0;
        if (j == 0) block_sum2(t[0], near, scratch);
        else if (a.clipped) block_sum2(t[j], zero, scratch);
    }
    if (threadIdx.x == 0) {
        a.st->sum_sq = t[0];
        a.st->near = (double)near;
        a.st->scan[a.which] = TensorState::Scan{a.clipped ? t[1] : 0.0, a.clipped ? t[2] : 0.0, 0.0, a.n_bins};
    }
    if (a.n_bins2 > 0) {
        const double d = (double)(-2 * a.lo - 1);
        double dn = a.clipped ? t[3] : 0.0, ds = a.clipped ? t[4] : 0.0, df = 0.0;
        tensor_scan(a.hist + 2 * a.win, a.hist + 2 * a.win + a.n_bins2, a.n_bins2, unit / d, dn, ds, df, (double)a.n_bins2,
                    a.above + 2 * a.win, a.above + 2 * a.win + a.n_bins2, part);
    }
}
__device__ __forceinline__ double tensor_unit(const TensorArgs& a) {
    const float m = fmaxf(__uint_as_float(a.st->mpos_bits), __uint_as_float(a.st->mneg_bits));
    return hist_unit(grid_of(m, a.hi_frac, a.n_cand).step);
}

// A window that a block scans by itself; with few candidates it goes on to their sums.
constexpr int kLevelsHere = 128;
__global__ void __launch_bounds__(kScanThreads) tensor_scan_kernel(const TensorArgs a) {
    __shared__ double part[32][3];
    __shared__ double scratch[64];
    const double unit = tensor_unit(a);
    if (a.first_window) tensor_scan_begin(a, unit, part, scratch);
    __syncthreads();
    const TensorState::Scan above = a.st->scan[a.which];
    double cn = above.n, cs = above.s, cf = above.f;
    tensor_scan(a.hist, a.hist + a.win, a.win, unit, cn, cs, cf, (double)(above.pos - a.win_base), a.above, a.above + a.win, part);
    if (threadIdx.x == 0) a.st->scan[a.which ^ 1] = TensorState::Scan{cn, cs, cf, a.win_base};
    if (a.n_cand > kLevelsHere) return;
    __syncthreads();                                       // N and P
    for (int i0 = 0; i0 < 8 * a.n_cand; i0 += kScanThreads) tensor_levels_of(a, i0 + threadIdx.x);
}

// Windows of more bins, in two launches: the sums of chunks of kScanChunk bins, then the scan of every chunk from what lies above it.
// (One more block of the first launch does what is beside the bins.)
constexpr int kScanChunk = 4096;
__global__ void __launch_bounds__(kScanThreads) tensor_chunks_kernel(const TensorArgs a) {
    __shared__ double part[32][3];
    __shared__ double scratch[64];
    if ((int)blockIdx.x == a.n_chunks) {
        tensor_scan_begin(a, tensor_unit(a), part, scratch);
        return;
    }
    const int first = blockIdx.x * kScanChunk, n = min(kScanChunk, a.win - first);
    double cn = 0.0, cs = 0.0, cf = 0.0;
    for (int i = threadIdx.x; i < n; i += kScanThreads) {
        const double c = (double)__ldcg(a.hist + first + i);
        cn += c;
        cs = fma((double)i, c, cs);
        cf += (double)__ldcg(a.hist + a.win + first + i);
    }
    long long zero = 0;
    block_sum2(cn, zero, scratch);
    block_sum2(cs, zero, scratch);
    block_sum2(cf, zero, scratch);
    if (threadIdx.x == 0) {
        a.chunks[3 * blockIdx.x] = cn;
        a.chunks[3 * blockIdx.x + 1] = cs;
        a.chunks[3 * blockIdx.x + 2] = cf;
    }
}
__global__ void __launch_bounds__(kScanThreads) tensor_chunk_scan_kernel(const TensorArgs a) {
    __shared__ double part[32][3];
    __shared__ double scratch[64];
    const TensorState::Scan above = a.st->scan[a.which];
    const int first = blockIdx.x * kScanChunk, n = min(kScanChunk, a.win - first);
    // the state at this chunk's end: sums of T - position are linear in the position
    double cn = 0.0, cs = 0.0, cf = 0.0;
    const double end = (double)(first + n);
    for (int c = blockIdx.x + 1 + threadIdx.x; c < a.n_chunks; c += kScanThreads) {
        const double nn = __ldcg(a.chunks + 3 * c);
        cn += nn;
        cs += __ldcg(a.chunks + 3 * c + 1) + ((double)c * kScanChunk - end) * nn;
        cf += __ldcg(a.chunks + 3 * c + 2);
    }
    long long zero = 0;
    block_sum2(cn, zero, scratch);
    block_sum2(cs, zero, scratch);
    block_sum2(cf, zero, scratch);
    cn += above.n;
    cs += above.s + ((double)(above.pos - a.win_base) - end) * above.n;
    cf += above.f;
    tensor_scan(a.hist + first, a.hist + a.win + first, n, tensor_unit(a), cn, cs, cf, (double)n, a.above + first, a.above + a.win + first, part);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->scan[a.which ^ 1] = TensorState::Scan{cn, cs, cf, a.win_base};
}

// squared error of a candidate from its sums; INFINITY when its scale is not usable
__device__ __forceinline__ double tensor_error(float step, int c, double sum_sq, double sx, double sq) {
    const float ac = __fmul_rn((float)(c + 1), step);
    if (!usable_scale(ac)) return INFINITY;
    const double al = (double)ac, h = 0.5 * (double)step;
    return fmax(fma(al * al, sq, fma(-2.0 * al * h, sx, sum_sq)), 0.0);
}
// What separates the curve at candidate c from the error that exact_code's codes give.  The curve counts a value above the
// threshold m*h, m = (2j-1)*(c+1); the codes follow the IEEE quotient by alpha_c = fl((c+1)*step), whose threshold lies within
// 2^-23 of m*h.  A value in between is coded to the other neighbour, which moves its error by 2*alpha_c times its distance from
// the midpoint, 1.8e-7*m*h at most.  Such values are next to an edge of a bin; `near` is the sum of their m, so the sum of these
// terms is at most 4*(c+1)*1.8e-7*h^2*near.  Among values drawn from a density one in a million lies there and the bound is far
// below the band; among values on a lattice of their own all may.
__device__ __forceinline__ double tensor_noise(float step, int c, double near) {
    const double h = 0.5 * (double)step;
    return 8e-7 * (double)(c + 1) * h * h * near;
}
// Candidates whose value less their noise is up to this may be the minimum (bv: the smallest value, its noise added): near-ties,
// and what the rounding of the binary64 sums can amount to.
__device__ __forceinline__ double tensor_band(double bv, double sum_sq) {
    return bv * (1.0 + kRescoreBand) + 1e-13 * sum_sq;
}

// The first polish step, alpha <- <x,q>/<q,q> at candidate c, needs no look at the tensor: at a scale of the grid the thresholds are
// edges of bins, and <x,q>, <q,q> are the sums that the curve was made of, exact integers but for a last rounding in binary64.  Only
// the values next to an edge may be coded differently by the IEEE quotient; they are listed, and here is what such a value
// changes.  (51,380,224 values: a step less is 47 us of 366; 1,605,633 in one kernel: an exchange and a pass, 4 us of 37.)  The values come in
// the order in which atomics listed them, so the sums of their changes have to be exact: in the histogram's units (h is hk of them, below
// 2^24) a value is an integer.  512 of them in 4096 bins stay below 2^53, a quarter of a million in 8192 bins below 2^63.
// y: the value times HistGeometry::pre; hi: levels of a side.
struct NearChange {
    float x, units;          // magnitude, and the same in the histogram's units
    int q, qq;               // change of its code's magnitude and of the square
};
__device__ __forceinline__ NearChange near_change(float y, const HistGeometry& g, int c, int hi, float alpha, float inv, float flo, float fhi, float thr) {
    const float s = y * g.scale, v = g.sgn ? fabsf(s) : s, u = __fmaf_rd(v, g.inv_up, kMagic);
    int m = magic_int(u), k = __float2int_rz(fmaf(-(u - kMagic), g.h, v));
    if (hist_near(k, m)) hist_correct(k, m, g.hk);
    int counted = min(hi, (min(m, g.n_bins) / (c + 1) + 1) >> 1);
    if (y < 0.f && g.d > 0 && min(m / g.d, g.n_bins2) >= c + 1) ++counted;
    const float x = y * __fdiv_rn(1.0f, g.pre);
    const int coded = abs(exact_code(x, alpha, inv, flo, fhi, thr));
    return NearChange{fabsf(x), fabsf(s), coded - counted, coded * coded - counted * counted};
}
// The step by one block at candidate c (same in all threads): sx, sq are <x,q>/h and <q,q> there as the bins have it.
__device__ __forceinline__ void tensor_first_step(const TensorArgs& a, float step, int c, double* scratch) {
    TensorState* st = a.st;
    const unsigned int n_near = __ldcg(&st->n_near);
    if (a.refine_iters < 1 || n_near > (unsigned)a.near_cap) return;
    const HistGeometry g = hist_geometry(step, a);
    const float alpha = __fmul_rn((float)(c + 1), step), inv = __fdiv_rn(1.0f, alpha), flo = (float)a.lo, fhi = (float)a.hi,
                thr = ambiguity_threshold(flo, fhi);
    double dq = 0.0;
    long long dx = 0;
    for (unsigned int i = threadIdx.x; i < n_near; i += blockDim.x) {
        const NearChange v = near_change(__ldcg(a.near + i), g, c, a.hi, alpha, inv, flo, fhi, thr);
        dx += (long long)v.units * v.q;
        dq += (double)v.qq;
    }
    block_sum2(dq, dx, scratch);
    if (threadIdx.x == 0) {
        const double sxq = fma(0.5 * (double)step, __ldcg(a.levels + c), (double)dx / ((double)g.scale * (double)g.pre));
        const long long sqq = (long long)__ldcg(a.levels + a.n_cand + c) + (long long)dq;
        const float a_new = sqq != 0 ? (float)(sxq / (double)sqq) : 0.f;
        if (a_new >= FLT_MIN && a_new <= FLT_MAX && a_new != alpha) st->alpha = a_new;
        else st->polish_done = 1;                           // as a polish pass would
        st->first_done = 1;
    }
}

// One block: the curve, its minimum and the list of candidates to re-score.
__global__ void __launch_bounds__(1024) tensor_finish_kernel(const TensorArgs a) {
    __shared__ double scratch[64];
    __shared__ int cnt;
    TensorState* st = a.st;
    const float m = fmaxf(__uint_as_float(st->mpos_bits), __uint_as_float(st->mneg_bits));
    const Grid g = grid_of(m, a.hi_frac, a.n_cand);
    const bool usable = g.usable && !st->bad;
    const double sum_sq = st->sum_sq;
    double bv = INFINITY;
    int bi = 0x7fffffff;
    for (int c = threadIdx.x; c < a.n_cand; c += blockDim.x) {
        const double v = usable ? tensor_error(g.step, c, sum_sq, a.levels[c], a.levels[a.n_cand + c]) : INFINITY;
        a.curve[c] = v;
        if (a.curve_out) a.curve_out[c] = v;
        if (v < bv) {
            bv = v;
            bi = c;
        }
    }
    if (threadIdx.x == 0) cnt = 0;
    block_argmin(bv, bi, scratch);
    if (bi == 0x7fffffff) {
        if (threadIdx.x == 0) {
            st->best_idx = -1;
            st->alpha = 0.f;
            st->n_list = 0;
            atomicOr(a.status, 2u);
        }
        return;
    }
    const double near = st->near, band = tensor_band(bv + tensor_noise(g.step, bi, near), sum_sq);
    const double tiny = a.curve_out ? kTinyShare * sum_sq : 0.0;
    for (int c = threadIdx.x; c < a.n_cand; c += blockDim.x) {
        const double v = a.curve[c];
        if (v - tensor_noise(g.step, c, near) <= band || v < tiny) a.list[atomicAdd(&cnt, 1)] = c;   // at most n_cand entries: the list holds them all
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        st->step = g.step;
        st->best_idx = bi;
        st->alpha = __fmul_rn((float)(bi + 1), g.step);
        st->n_list = cnt > 1 || bv < tiny ? cnt : 0;   // a single candidate in the band needs no re-scoring
    }
    if (!(cnt > 1 || bv < tiny)) tensor_first_step(a, g.step, bi, scratch);
}

// Grid-wide pass over the tensor; sums in fp64, codes equal to those of the IEEE division (see magic_code).
//   MODE 0 (rescore): squared error at each listed candidate; the last block picks the best.
//   MODE 1 (refine):  <x,q> and <q,q> at st->alpha; the last block sets alpha <- <x,q>/<q,q>.
//   MODE 2 (final):   squared error at st->alpha; the last block writes the outputs.
// Every block keeps its partial sums in its own slot of `partials`; blocks without a slot (a long list of
// candidates on a small scratch) leave at once and the others stride over the whole tensor.
template <int MODE>
__global__ void __launch_bounds__(256) tensor_pass_kernel(const TensorArgs a) {
    __shared__ double scratch[64];
    __shared__ bool is_last;
    TensorState* st = a.st;
    const float flo = (float)a.lo, fhi = (float)a.hi;
    const float clo = kMagic + flo, chi = kMagic + fhi;
    const float amb_thr = ambiguity_threshold(flo, fhi);
    const int n_list = MODE == 0 ? st->n_list : 1;
    if (MODE == 0 && n_list == 0) return;
    const float alpha_now = st->alpha;
    const float delta = st->delta;
    if (MODE == 1 && (!(alpha_now > 0.f) || st->polish_done || (a.first_pass && st->first_done))) return;
    const int slot = MODE == 0 ? ((n_list + 3) & ~3) : 1;                  // doubles per block
    double* const room = MODE == 0 ? a.levels + 2 * a.n_cand : a.partials;   // (the first polish step still needs <x,q> and <q,q>)
    const long long fit = (a.partial_doubles - (room - a.partials)) / (slot + 1);
    const unsigned int nblk = (long long)gridDim.x < fit ? gridDim.x : (unsigned int)fit;
    if (blockIdx.x >= nblk) return;
    double* part_d = room;                                                 // [nblk][slot]
    long long* part_q = reinterpret_cast<long long*>(room + (size_t)nblk * slot);   // [nblk]
    const long long stride = (long long)nblk * blockDim.x;
    const long long tid0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n4 = a.n >> 2;
    const float4* x4 = reinterpret_cast<const float4*>(a.x);

    for (int l0 = 0; l0 < n_list; l0 += 4) {
        float al[4], inv[4];
        double ald[4];
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        long long sqq = 0;
        int sqq32 = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (MODE == 0) {
                const int c = (l0 + j < n_list) ? a.list[l0 + j] : a.list[l0];
                al[j] = __fmul_rn((float)(c + 1), st->step);
            } else {
                al[j] = alpha_now;
            }
            inv[j] = al[j] > 0.f ? __fdiv_rn(1.0f, al[j]) : 0.f;
            ald[j] = (double)al[j];
        }
        const int nj = MODE == 0 ? 4 : 1;
        auto element = [&](float x) {
            const double xd = (double)x;
#pragma unroll
            for (int j = 0; j < nj; ++j) {
                bool amb;
                float tc = magic_code(x, inv[j], clo, chi, amb_thr, amb);
                if (amb) tc = kMagic + (float)(al[j] > 0.f ? code_of(x, al[j], flo, fhi) : 0);   // rare: the division decides
                const int q = magic_int(tc);
                const double qd = int_double(q);
                if (MODE == 1) {
                    sqq32 += q * q;          // folded into the 64-bit sum after every float4 (q*q <= 2^14)
                    acc[j] = fma(xd, qd, acc[j]);
                } else {
                    const double d = fma(-ald[j], qd, xd);
                    acc[j] = fma(d, d, acc[j]);
                }
            }
        };
        auto four = [&](const float4& v) {
            element(v.x - delta);
            element(v.y - delta);
            element(v.z - delta);
            element(v.w - delta);
            sqq += sqq32;
            sqq32 = 0;
        };
        // four 128-bit loads in flight per thread before any of them is used
        long long i = tid0;
        for (; i + 3 * stride < n4; i += 4 * stride) {
            const float4 v0 = __ldg(x4 + i), v1 = __ldg(x4 + i + stride), v2 = __ldg(x4 + i + 2 * stride),
                         v3 = __ldg(x4 + i + 3 * stride);
            four(v0);
            four(v1);
            four(v2);
            four(v3);
        }
        for (; i < n4; i += stride) four(__ldg(x4 + i));
        for (long long e = (n4 << 2) + tid0; e < a.n; e += stride) element(a.x[e] - delta);
        sqq += sqq32;
        for (int j = 0; j < nj; ++j) {
            long long q = sqq;
            block_sum2(acc[j], q, scratch);
            if (threadIdx.x == 0) {
                part_d[(size_t)blockIdx.x * slot + l0 + j] = acc[j];
                if (MODE == 1) part_q[blockIdx.x] = q;
            }
        }
    }
    // ---- last block to arrive reduces the per-block partials (fixed order: thread t takes blocks t, t+256, ...,
    //      then the block-wide sum in lane and warp order)
    __threadfence();
    if (threadIdx.x == 0) {
        const unsigned int tk = atomicAdd(&st->ticket, 1u);
        is_last = (tk == nblk - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double best_sse = INFINITY;     // MODE 0: this thread's best listed candidate
    int best = 0x7fffffff;
    double total = 0.0;             // MODE 1, 2
    long long total_q = 0;
    if (MODE == 0) {
        for (int l = threadIdx.x; l < n_list; l += blockDim.x) {
            double s = 0.0;
            for (unsigned int b = 0; b < nblk; ++b) s += __ldcg(&part_d[(size_t)b * slot + l]);
            const int c = a.list[l];
            if (a.curve_out && s < kTinyShare * st->sum_sq) a.curve_out[c] = s;   // the difference of sums had lost digits
            if (s < best_sse || (s == best_sse && c < best)) {
                best_sse = s;
                best = c;
            }
        }
        block_argmin(best_sse, best, scratch);
    } else {
        for (unsigned int b = threadIdx.x; b < nblk; b += blockDim.x) {
            total += __ldcg(&part_d[b]);
            if (MODE == 1) total_q += __ldcg(&part_q[b]);
        }
        block_sum2(total, total_q, scratch);
    }
    if (threadIdx.x == 0) {
        st->ticket = 0u;
        if (MODE == 0) {
            st->best_idx = best;
            st->alpha = __fmul_rn((float)(best + 1), st->step);
        } else if (MODE == 1) {
            bool moved = false;
            if (total_q != 0) {
                const float a_new = (float)(total / (double)total_q);
                if (a_new >= FLT_MIN && a_new <= FLT_MAX && a_new != st->alpha) {
                    st->alpha = a_new;
                    moved = true;
                }
            }
            if (!moved) st->polish_done = 1;   // stopped or fixed point: the remaining polish launches have nothing to do
        } else {
            *a.alpha_out = st->alpha;
            if (a.delta_out) *a.delta_out = st->delta;
            *a.sse_out = (float)total;
            if (a.idx_out) *a.idx_out = st->best_idx;
            if (a.status_out) *a.status_out = *a.status;
        }
    }
    if (MODE == 0) {
        __syncthreads();                                    // best_idx and alpha before the step replaces alpha
        tensor_first_step(a, st->step, best, scratch);
    }
}

// -------------------------------------------------------------------------------------------------
// The whole search in one kernel, for a tensor whose values fit in the shared memory of the GPU: every block stages its
// slice once and keeps it for all passes, the blocks exchange sums through slots in global memory (a cooperative launch
// guarantees that all of them run), and what has to be known everywhere - the scan of the histogram, the curve, the
// polish - every block computes for itself.
// Bound: latency.  A search with R polish steps is a chain of 1 + R exchanges (extremes, histogram, every polish step but the first;
// one more where candidates are re-scored) of a microsecond or two each; the pipeline of launches pays a launch and a trip of the
// values from L2 for each of them.
// -------------------------------------------------------------------------------------------------
constexpr int kResidentBlocks = 160;     // blocks the exchange area has room for
constexpr int kResidentBins = 4096;      // bins of the histogram in the exchange area (and as many coarse ones)
constexpr int kResidentCands = 1024;
constexpr int kResidentNear = 512;       // values next to an edge of a bin in the list, a thread's each
constexpr unsigned int kSpinLimit = 1u << 22;   // polls of a slot before a block gives up (seconds), by default

struct __align__(128) ResidentSlot {     // one block's contribution to an exchange: 64 bits, and 40 bits under a 24-bit tag
    unsigned long long a, b;             // (a line of its own: see below)
};
struct ResidentExchange {                // in the context workspace; all zero between calls
    ResidentSlot slot[2][kResidentBlocks];
    unsigned int ticket;
    unsigned int n_near;                 // as TensorState::n_near
    unsigned int pad_[2];
    double fin[kResidentBlocks];
    float near[kResidentNear];
    unsigned long long hist[4 * kResidentBins];
};

struct ResidentArgs {
    ResidentExchange* ex;
    int slice4;                          // float4s per block
    double* rescore;                     // [listed candidates][gridDim.x]
    unsigned int spin_limit;             // polls of a slot before a block gives up
};

// An exchange between the blocks: every block publishes a slot, data and tag in one 16-byte store, and the first warp of every
// block polls all of them, up to five slots a lane.  No counter that all blocks would have to add to one after the other, no fence
// between data and flag, and one trip to L2 each way.  One warp polls and not a thread for each slot, and every slot has a
// line of L2 to itself: the polls of all blocks queue at the lines that slots share, and the slots of the last blocks to arrive
// wait behind them (148 blocks that arrive within 0.75 us: 148 threads of each poll 5.4 us, a warp 3.7, a warp and a line per slot
// 2.2).  The warp has the sums in its lanes, so that a barrier on either side of it is all that the block waits for.  Slots
// alternate between two sets: a block can only be one exchange ahead, since it waits for everybody's slot of this one.  Tags count
// the exchanges of a call from 1; the last block of a call clears the slots.  Slots are stored and loaded with relaxed order.  Where
// an exchange stands for more than its slots (DATA: the histogram, the errors of the re-scored candidates), thread 0 fences between
// the barrier behind which the block's writes lie and its slot, and the polling warp fences between its polls and the barrier that
// lets the block read.  A block that does not see a slot within the limit of polls sets s_bad, goes on to the end without further
// exchanges, and reports it.
struct ResidentPart {                // shared words of a block's part in an exchange
    double d[kResidentThreads / 32], d_all;
    long long q[kResidentThreads / 32], q_all;
};
struct ResidentTeam {
    ResidentExchange* ex;
    unsigned int step;               // exchanges so far
    int* s_bad;                      // shared: some slot did not appear
    unsigned int spin_limit;
};
__device__ __forceinline__ void slot_store(ResidentSlot* p, unsigned long long a, unsigned long long b) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void slot_load(const ResidentSlot* p, unsigned long long& a, unsigned long long& b) {
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// The first warp publishes the block's slot (a, b40: the same in all lanes, known after a barrier) and polls; use(a, b40) is called
// for every block's slot, the slots lane, lane + 32, ... by a lane in increasing order.
template <bool DATA, class F>
__device__ __forceinline__ void resident_gather(const ResidentTeam& t, unsigned long long a, unsigned long long b40, F use) {
    const int lane = threadIdx.x & 31, nblk = gridDim.x;
    ResidentSlot* set = t.ex->slot[t.step & 1];
    if (lane == 0) {
        if (DATA) fence_gpu();
        slot_store(set + blockIdx.x, a, ((unsigned long long)t.step << 40) | b40);
    }
    constexpr int per = (kResidentBlocks + 31) / 32;
    unsigned long long va[per], vb[per];
    unsigned int open = 0u;
#pragma unroll
    for (int j = 0; j < per; ++j) {
        va[j] = vb[j] = 0ull;
        if (lane + 32 * j < nblk) open |= 1u << j;
    }
    for (unsigned int polls = 0u; open && polls < t.spin_limit; ++polls) {
#pragma unroll
        for (int j = 0; j < per; ++j)
            if (open >> j & 1u) slot_load(set + lane + 32 * j, va[j], vb[j]);
#pragma unroll
        for (int j = 0; j < per; ++j)
            if ((unsigned int)(vb[j] >> 40) == t.step) open &= ~(1u << j);
    }
    if (open) *t.s_bad = 1;
    if (DATA) fence_gpu();
    __syncwarp();
#pragma unroll
    for (int j = 0; j < per; ++j)
        if ((unsigned int)(vb[j] >> 40) == t.step) use(va[j], vb[j] & 0xffffffffffull);
}
// Sum of a double and of a non-negative integer below 2^40 over all threads of all blocks, in a fixed order; every thread
// gets it.  False: see above.  The words of `part` are for this function and resident_extremes() alone: their barriers order its uses.
template <bool DATA>
__device__ __forceinline__ bool resident_sum(ResidentTeam& t, double& d, long long& q, ResidentPart* part) {
    constexpr int nwarp = kResidentThreads / 32;
    const int lane = threadIdx.x & 31;
    d = warp_sum(d);
    q = warp_sum(q);
    if (lane == 0) {
        part->d[threadIdx.x >> 5] = d;
        part->q[threadIdx.x >> 5] = q;
    }
    __syncthreads();
    ++t.step;
    if (threadIdx.x < 32) {
        d = part->d[lane & (nwarp - 1)];
        q = part->q[lane & (nwarp - 1)];
#pragma unroll
        for (int o = 1; o < nwarp; o <<= 1) {      // (all lanes end with the same bits: a + b == b + a)
            d += __shfl_xor_sync(0xffffffffu, d, o);
            q += __shfl_xor_sync(0xffffffffu, q, o);
        }
        double dt = 0.0;
        long long qt = 0;
        resident_gather<DATA>(t, (unsigned long long)__double_as_longlong(d), (unsigned long long)q, [&](unsigned long long va, unsigned long long vb) {
            dt += __longlong_as_double((long long)va);
            qt += (long long)vb;
        });
        dt = warp_allsum(dt);
        qt = warp_allsum(qt);
        if (lane == 0) {
            part->d_all = dt;
            part->q_all = qt;
        }
    }
    __syncthreads();
    d = part->d_all;
    q = part->q_all;
    return *t.s_bad == 0;
}
// Smallest key, largest key and the union of flags over all threads of all blocks; every thread gets them.
__device__ __forceinline__ bool resident_extremes(ResidentTeam& t, int& kmin, int& kmax, unsigned int& flags, ResidentPart* part) {
    constexpr int nwarp = kResidentThreads / 32;
    const int lane = threadIdx.x & 31;
    const auto both = [](int hi, int lo) { return (long long)(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo); };
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (lane == 0) {
        part->q[threadIdx.x >> 5] = both(kmax, kmin);
        part->d[threadIdx.x >> 5] = (double)flags;
    }
    __syncthreads();
    ++t.step;
    if (threadIdx.x < 32) {
        const long long k = part->q[lane & (nwarp - 1)];
        kmin = __reduce_min_sync(0xffffffffu, (int)(unsigned)k);
        kmax = __reduce_max_sync(0xffffffffu, (int)(k >> 32));
        flags = __reduce_or_sync(0xffffffffu, (unsigned)part->d[lane & (nwarp - 1)]);
        resident_gather<false>(t, (unsigned long long)both(kmax, kmin), flags, [&](unsigned long long va, unsigned long long vb) {
            kmin = min(kmin, (int)(unsigned)va);
            kmax = max(kmax, (int)(unsigned)(va >> 32));
            flags |= (unsigned)vb;
        });
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        flags = __reduce_or_sync(0xffffffffu, flags);
        if (lane == 0) {
            part->q_all = both(kmax, kmin);
            part->d_all = (double)flags;
        }
    }
    __syncthreads();
    kmin = (int)(unsigned)part->q_all;
    kmax = (int)(part->q_all >> 32);
    flags = (unsigned)part->d_all;
    return *t.s_bad == 0;
}

__global__ void __launch_bounds__(kResidentThreads) tensor_resident_kernel(const TensorArgs a, const ResidentArgs r, int refine_iters) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double scratch[64];
    __shared__ double part[32][3];
    __shared__ ResidentPart exchanged;
    __shared__ NearList<256> s_near;
    __shared__ unsigned int s_near_at;
    __shared__ int s_bad, s_last, s_count[33];
    ResidentExchange* ex = r.ex;
    ResidentTeam team = {ex, 0u, &s_bad, r.spin_limit};
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nblk = gridDim.x;
    const int bins = a.win;                                         // n_bins rounded up to a multiple of 4
    // shared memory: the slice | N, P of the bins and coarse bins (the words of the histogram before that) | the curve | the list
    float4* data = reinterpret_cast<float4*>(smem_raw);
    double* above = reinterpret_cast<double*>(data + r.slice4);
    double* above2 = above + 2 * bins;
    double* curve = above2 + 2 * a.n_bins2;
    int* list = reinterpret_cast<int*>(curve + a.n_cand);
    bool ok = true;
    if (tid == 0) {
        s_bad = 0;
        s_near.n = 0u;
    }
    // ---- the slice, its extremes
    const float4* x4 = reinterpret_cast<const float4*>(a.x);
    const long long n4 = a.n >> 2, begin = (long long)blockIdx.x * r.slice4;
    const int mine4 = (int)max(0ll, min((long long)r.slice4, ((a.n + 3) >> 2) - begin));      // float4s of this block, the last one perhaps partial
    float lo = INFINITY, hi = -INFINITY;
    bool bad = false;
    auto extremes = [&](float e) {
        const bool finite = fabsf(e) <= FLT_MAX;
        bad |= !finite;
        lo = fminf(lo, finite ? e : lo);
        hi = fmaxf(hi, finite ? e : hi);
    };
    const int full4 = (int)max(0ll, min((long long)mine4, n4 - begin));
    int i = tid;
    for (; i + 3 * kResidentThreads < full4; i += 4 * kResidentThreads) {      // four loads in flight
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __ldg(x4 + begin + i + j * kResidentThreads);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            data[i + j * kResidentThreads] = v[j];
            extremes(v[j].x);
            extremes(v[j].y);
            extremes(v[j].z);
            extremes(v[j].w);
        }
    }
    for (; i < full4; i += kResidentThreads) {
        const float4 v = __ldg(x4 + begin + i);
        data[i] = v;
        extremes(v.x);
        extremes(v.y);
        extremes(v.z);
        extremes(v.w);
    }
    const int tail = mine4 > full4 ? (int)(a.n - 4 * n4) : 0;       // one to three values in the block that holds the end
    if (tid < tail) {
        const float v = a.x[4 * n4 + tid];
        reinterpret_cast<float*>(data + full4)[tid] = v;
        extremes(v);
    }
    for (int j = tid; j < 3 * (bins + a.n_bins2); j += kResidentThreads) reinterpret_cast<unsigned int*>(above)[j] = 0u;
    // ---- extremes of the tensor, in every block
    int kmin = lo <= hi ? float_key(lo) : 0x7fffffff, kmax = lo <= hi ? float_key(hi) : (int)0x80000000;
    unsigned int nonfinite = bad ? 1u : 0u;
    ok = resident_extremes(team, kmin, kmax, nonfinite, &exchanged);
    const float vmin = kmin <= kmax ? key_float(kmin) : 0.f, vmax = kmin <= kmax ? key_float(kmax) : 0.f;
    float delta = 0.f, m = fmaxf(fmaxf(vmax, 0.f), fmaxf(-vmin, 0.f));
    if (a.delta_out && kmin <= kmax) {
        delta = vmin;
        m = vmax - vmin;                                            // max of fl(x - delta): subtraction is monotone
    }
    const Grid gr = grid_of(m, a.hi_frac, a.n_cand);
    const bool usable = ok && gr.usable && !nonfinite;
    int best = -1;
    float alpha = 0.f;
    const float flo = (float)a.lo, fhi = (float)a.hi, thr = ambiguity_threshold(flo, fhi);
    const int per = mine4 - (tail ? 1 : 0);                         // complete float4s
    const float* tailp = reinterpret_cast<const float*>(data + full4);
    if (usable) {
        // ---- histogram of the slice; the offset is subtracted from the staged values on the way
        const HistGeometry g = hist_geometry(gr.step, a);
        unsigned int* wc = reinterpret_cast<unsigned int*>(above);
        unsigned int *wl = wc + bins, *wh = wl + bins, *c2 = wh + bins, *l2 = c2 + a.n_bins2, *h2 = l2 + a.n_bins2;
        double sq = 0.0;
        long long near = 0;
        auto insert = [&](float x) {
            const float y = x * g.pre * g.scale, v = g.sgn ? fabsf(y) : y;
            sq = fma((double)x, (double)x, sq);
            const float u = __fmaf_rd(v, g.inv_up, kMagic);
            int mm = magic_int(u);
            if (mm < 1) return;
            int ks = __float2int_rz(fmaf(-(u - kMagic), g.h, v));
            if (hist_near(ks, mm)) {
                near += mm;
                s_near.add(x * g.pre);
                hist_correct(ks, mm, g.hk);
                if (mm < 1) return;
            }
            const unsigned int k = (unsigned)ks;
            hist_put3(wc, wl, wh, min(mm, g.n_bins) - 1, k);
            if (y < 0.f && mm >= g.d_from) {
                const unsigned int m2 = __umulhi((unsigned)mm, g.rd), rem = (unsigned)mm - m2 * (unsigned)g.d;
                hist_put3(c2, l2, h2, min((int)m2, g.n_bins2) - 1, rem * g.hk + k);
            }
        };
        for (int j = tid; j < per; j += kResidentThreads) {
            float4 v = data[j];
            if (delta != 0.f) {
                v.x -= delta;
                v.y -= delta;
                v.z -= delta;
                v.w -= delta;
                data[j] = v;
            }
            insert(v.x);
            insert(v.y);
            insert(v.z);
            insert(v.w);
        }
        if (tid < tail) {
            const float x = tailp[tid] - delta;
            reinterpret_cast<float*>(data + full4)[tid] = x;
            insert(x);
        }
        __syncthreads();
        unsigned long long* gh = ex->hist;
        for (int j = tid; j < bins + a.n_bins2; j += kResidentThreads) {
            const bool coarse = j >= bins;
            const int b = coarse ? j - bins : j;
            const unsigned int c = coarse ? c2[b] : wc[b];
            if (!c) continue;
            const unsigned long long f = coarse ? ((unsigned long long)h2[b] << 16) + l2[b] : ((unsigned long long)wh[b] << 16) + wl[b];
            atomicAdd(gh + (coarse ? 2 * kResidentBins : 0) + b, (unsigned long long)c);
            atomicAdd(gh + (coarse ? 3 * kResidentBins : kResidentBins) + b, f);
        }
        s_near.flush(&ex->n_near, ex->near, kResidentNear, s_near_at);
        // With more than a few values per thread the additions take longer than the block's sums: every thread waits for its own
        // beside them, which leaves thread 0's fence little to wait for (601,676 values 27.5 -> 26.5 us; 11,552 values 15.1 and 16.0)
        if (r.slice4 > kResidentThreads) fence_gpu();
        long long none = 0;
        double sum_sq = sq;
        ok = resident_sum<true>(team, sum_sq, near, &exchanged) && ok; // every block's additions are known after this (near < 2^29 per block)
        // ---- N, P and the curve, in every block
        const unsigned int n_near = ok ? __ldcg(&ex->n_near) : kResidentNear + 1u;      // (for the polish; on their way meanwhile)
        const float near_y = __ldcg(ex->near + tid);
        const double unit = hist_unit(gr.step);
        double cn = 0.0, cs = 0.0, cf = 0.0;
        if (a.n_bins2 > 0) {
            tensor_scan(gh + 2 * kResidentBins, gh + 3 * kResidentBins, a.n_bins2, unit / (double)g.d, cn, cs, cf, (double)a.n_bins2,
                        above2, above2 + a.n_bins2, part);
            cn = cs = cf = 0.0;
        }
        tensor_scan(gh, gh + kResidentBins, bins, unit, cn, cs, cf, (double)a.n_bins, above, above + bins, part);
        __syncthreads();
        double bv = INFINITY;
        int bi = 0x7fffffff;
        // The smallest scales have the most levels: a warp for each of 16 candidates, eight threads for each of the next 64, then
        // a thread (500 candidates on 8 bits 11,600 cycles with eight threads for all of them, 5300 so).
        auto candidates = [&](auto lanes_tag, int from, int to) {
            constexpr int lanes = decltype(lanes_tag)::value;
            for (int c0 = from; c0 < to; c0 += kResidentThreads / lanes) {
                const int c = c0 + tid / lanes, p = tid & (lanes - 1);
                double sx = 0.0, sn = 0.0;
                if (c < to) tensor_levels(above, above + bins, 0, a.n_bins, c + 1, a.hi, p, lanes, sx, sn);
                if (p == 0 && c < min(to, a.n_bins2)) {
                    const double nn = above2[c], d = (double)g.d;
                    sx += d * (above2[a.n_bins2 + c] + (double)(c + 1) * nn);
                    sn += d * nn;
                }
#pragma unroll
                for (int o = 1; o < lanes; o <<= 1) {
                    sx += __shfl_xor_sync(0xffffffffu, sx, o);
                    sn += __shfl_xor_sync(0xffffffffu, sn, o);
                }
                if (p == 0 && c < to) {
                    const double v = tensor_error(gr.step, c, sum_sq, sx, sn);
                    curve[c] = v;
                    if (a.curve_out && blockIdx.x == 0) a.curve_out[c] = v;
                    if (v < bv) {
                        bv = v;
                        bi = c;
                    }
                }
            }
        };
        candidates(std::integral_constant<int, 32>(), 0, min(16, a.n_cand));
        candidates(std::integral_constant<int, 8>(), 16, min(80, a.n_cand));
        candidates(std::integral_constant<int, 1>(), 80, a.n_cand);
        block_argmin_error(bv, bi, scratch);
        best = bi;
        const double near_sum = (double)near, tiny = a.curve_out ? kTinyShare * sum_sq : 0.0;
        const double band = tensor_band(bv + tensor_noise(gr.step, bi, near_sum), sum_sq);
        // ---- candidates to re-score, in increasing order: thread t looks at candidates 2t and 2t+1
        static_assert(kResidentNear == kResidentThreads, "a listed value per thread");
        static_assert(kResidentCands <= 2 * kResidentThreads, "two candidates per thread");
        auto wanted = [&](int c) { return c < a.n_cand && (curve[c] - tensor_noise(gr.step, c, near_sum) <= band || curve[c] < tiny); };
        const bool in0 = wanted(2 * tid), in1 = wanted(2 * tid + 1);
        const unsigned int b0 = __ballot_sync(0xffffffffu, in0), b1 = __ballot_sync(0xffffffffu, in1), below = (1u << lane) - 1u;
        if (lane == 0) s_count[warp] = __popc(b0) + __popc(b1);
        __syncthreads();
        const int listed = s_count[lane & (kResidentThreads / 32 - 1)], n_list = (int)__reduce_add_sync(0xffffffffu, (unsigned)listed) / (1024 / kResidentThreads);
        if (n_list > 1 || bv < tiny) {
            int at = __popc(b0 & below) + __popc(b1 & below) + (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)listed : 0u);
            if (in0) list[at++] = 2 * tid;
            if (in1) list[at] = 2 * tid + 1;
            __syncthreads();
        }
        auto slice_error = [&](float al) -> double {                // squared error of the slice at one scale, exact codes
            const float inv = __fdiv_rn(1.0f, al);
            const double ad = (double)al;
            double ss = 0.0;
            auto one = [&](float x) {
                const double e = fma(-ad, int_double(exact_code(x, al, inv, flo, fhi, thr)), (double)x);
                ss = fma(e, e, ss);
            };
            for (int j = tid; j < per; j += kResidentThreads) {
                const float4 v = data[j];
                one(v.x);
                one(v.y);
                one(v.z);
                one(v.w);
            }
            if (tid < tail) one(tailp[tid]);
            long long zero = 0;
            block_sum2(ss, zero, scratch);
            return ss;
        };
        if (ok && best != 0x7fffffff && (n_list > 1 || bv < tiny)) {
            for (int l = 0; l < n_list; ++l) {
                const double ss = slice_error(__fmul_rn((float)(list[l] + 1), gr.step));
                if (tid == 0) r.rescore[(size_t)l * nblk + blockIdx.x] = ss;
            }
            double nothing = 0.0;
            none = 0;
            ok = resident_sum<true>(team, nothing, none, &exchanged) && ok;     // (only its waiting is wanted)
            double best_sse = INFINITY;
            int bc = 0x7fffffff;
            for (int l = warp; l < n_list; l += kResidentThreads / 32) {
                double v = 0.0;
                for (int b = lane; b < nblk; b += 32) v += __ldcg(r.rescore + (size_t)l * nblk + b);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                const int c = list[l];
                if (a.curve_out && v < tiny && blockIdx.x == 0 && lane == 0) a.curve_out[c] = v;   // the difference of sums had lost digits
                if (v < best_sse || (v == best_sse && c < bc)) {
                    best_sse = v;
                    bc = c;
                }
            }
            block_argmin(best_sse, bc, scratch);
            if (bc != 0x7fffffff) best = bc;
        }
        if (best == 0x7fffffff) best = -1;
        if (best >= 0) alpha = __fmul_rn((float)(best + 1), gr.step);
        // ---- polish: alpha <- <x,q>/<q,q>.  The first step from the bins (see tensor_first_step), the others by a look at the slice.
        int from = 0;
        if (best >= 0 && refine_iters > 0 && n_near <= kResidentNear) {
            double sx = 0.0, sn = 0.0, dx = 0.0;
            long long dq = 0;
            tensor_levels(above, above + bins, 0, a.n_bins, best + 1, a.hi, lane, 32, sx, sn);
            sx = warp_allsum(sx);
            sn = warp_allsum(sn);
            if (best < a.n_bins2) {
                const double nn = above2[best], d = (double)g.d;
                sx += d * (above2[a.n_bins2 + best] + (double)(best + 1) * nn);
                sn += d * nn;
            }
            if (tid < (int)n_near) {
                const NearChange v = near_change(near_y, g, best, a.hi, alpha, __fdiv_rn(1.0f, alpha), flo, fhi, thr);
                dx = (double)v.x * (double)v.q;
                dq = v.qq;
            }
            if (__syncthreads_or(dq != 0)) block_sum2(dx, dq, scratch);
            else dx = 0.0;
            const double sxq = fma(0.5 * (double)gr.step, sx, dx);
            const long long sqq = (long long)sn + dq;
            const float a_new = sqq != 0 ? (float)(sxq / (double)sqq) : 0.f;
            const bool moved = a_new >= FLT_MIN && a_new <= FLT_MAX && a_new != alpha;
            if (moved) alpha = a_new;
            from = moved ? 1 : refine_iters;
        }
        for (int it = from; ok && best >= 0 && it < refine_iters; ++it) {
            const float inv = __fdiv_rn(1.0f, alpha);
            double sxq = 0.0;
            long long sqq = 0;
            int s32 = 0;
            auto one = [&](float x) {
                const int q = exact_code(x, alpha, inv, flo, fhi, thr);
                s32 += q * q;
                sxq = fma((double)x, int_double(q), sxq);
            };
            for (int j = tid; j < per; j += kResidentThreads) {
                const float4 v = data[j];
                one(v.x);
                one(v.y);
                one(v.z);
                one(v.w);
                sqq += s32;                                         // four squares of at most 2^16
                s32 = 0;
            }
            if (tid < tail) one(tailp[tid]);
            sqq += s32;
            ok = resident_sum<false>(team, sxq, sqq, &exchanged) && ok;
            if (sqq == 0) break;
            const float a_new = (float)(sxq / (double)sqq);
            if (!(a_new >= FLT_MIN) || !(a_new <= FLT_MAX) || a_new == alpha) break;
            alpha = a_new;
        }
    }
    // ---- final error of the slice; the last block to arrive adds up and writes the outputs
    double ss = 0.0;
    {
        const bool shifted = usable;                                // the staged values have the offset subtracted already
        const float inv = alpha > 0.f ? __fdiv_rn(1.0f, alpha) : 0.f;
        const double ad = (double)alpha;
        auto one = [&](float x) {
            if (!shifted) x -= delta;
            const double e = alpha > 0.f ? fma(-ad, int_double(exact_code(x, alpha, inv, flo, fhi, thr)), (double)x) : (double)x;
            ss = fma(e, e, ss);
        };
        for (int j = tid; j < per; j += kResidentThreads) {
            const float4 v = data[j];
            one(v.x);
            one(v.y);
            one(v.z);
            one(v.w);
        }
        if (tid < tail) one(tailp[tid]);
    }
    long long zero = 0;
    block_sum2(ss, zero, scratch);
    if (tid == 0) {
        ex->fin[blockIdx.x] = ss;
        if (!ok) atomicOr(a.status, 4u);                            // any block's: its share of the outputs is not of this search
        __threadfence();
        s_last = atomicAdd(&ex->ticket, 1u) == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (warp == 0) {
        double v = 0.0;
        for (int b = lane; b < nblk; b += 32) v += __ldcg(ex->fin + b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            *a.alpha_out = alpha;
            *a.sse_out = (float)v;
            if (a.idx_out) *a.idx_out = best;
            if (a.delta_out) *a.delta_out = delta;
            const unsigned int st = (nonfinite ? 1u : 0u) | (best < 0 ? 2u : 0u);
            if (st) atomicOr(a.status, st);
            if (a.evals && usable) atomicAdd(a.evals, (unsigned long long)a.n);
        }
    }
    if (a.curve_out && best < 0)
        for (int c = tid; c < a.n_cand; c += kResidentThreads) a.curve_out[c] = INFINITY;
    // the exchange area as the next call expects it
    for (int j = tid; j < bins; j += kResidentThreads) ex->hist[j] = ex->hist[kResidentBins + j] = 0ull;
    for (int j = tid; j < a.n_bins2; j += kResidentThreads) ex->hist[2 * kResidentBins + j] = ex->hist[3 * kResidentBins + j] = 0ull;
    if (tid < kResidentBlocks) {
        slot_store(&ex->slot[0][tid], 0ull, 0ull);
        slot_store(&ex->slot[1][tid], 0ull, 0ull);
    }
    if (tid == 0) ex->ticket = ex->n_near = 0u;
}

// Key layers (Section 3.5): MSE of each layer = sum of its kernels' squared errors / elements, compared
// with the threshold tau.  One block per layer, fixed-order sum in fp64.
struct LayerError {
    const float* sse;        // [n_kernels] squared error per kernel, as the quantize calls output it
    long long n_kernels, kernel_len;
};

__global__ void __launch_bounds__(256) layer_mse_kernel(const LayerError* __restrict__ layers, float tau,
                                                         double* __restrict__ mse, int* __restrict__ is_key) {
    __shared__ double scratch[64];
    const LayerError L = layers[blockIdx.x];
    double s = 0.0;
    for (long long i = threadIdx.x; i < L.n_kernels; i += blockDim.x) s += (double)L.sse[i];
    long long zero = 0;
    block_sum2(s, zero, scratch);
    if (threadIdx.x == 0) {
        const double m = s / ((double)L.n_kernels * (double)L.kernel_len);
        mse[blockIdx.x] = m;
        if (is_key) is_key[blockIdx.x] = m > (double)tau ? 1 : 0;
    }
}

// Compression ratio of Section 3.5 for layers that hold one quantized tensor, or two where is_key is set:
// (codes at `bits` per element plus one binary32 scale per kernel, per quantized tensor) over the binary32 size.
__global__ void compression_ratio_kernel(const LayerError* __restrict__ layers, int n_layers, int bits,
                                         const int* __restrict__ is_key, double* __restrict__ cr) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double q = 0.0, f = 0.0;
    for (int l = 0; l < n_layers; ++l) {
        const double n = (double)layers[l].n_kernels * (double)layers[l].kernel_len;
        q += (is_key[l] ? 2.0 : 1.0) * (n * (double)bits + 32.0 * (double)layers[l].n_kernels);
        f += 32.0 * n;
    }
    *cr = f > 0.0 ? q / f : 0.0;
}

// INT4 emission: byte e/2 holds element e (even) in bits 0-3 and element e+1 in bits 4-7.
__global__ void __launch_bounds__(256) pack_int4_kernel(const signed char* __restrict__ codes, long long n,
                                                         unsigned char* __restrict__ packed) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long tid0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool aligned = ((reinterpret_cast<unsigned long long>(codes) & 15ull) == 0) &&
                         ((reinterpret_cast<unsigned long long>(packed) & 7ull) == 0);
    const long long n16 = aligned ? (n >> 4) : 0;
    for (long long i = tid0; i < n16; i += stride) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(codes) + i);
        const unsigned int w[4] = {(unsigned)v.x, (unsigned)v.y, (unsigned)v.z, (unsigned)v.w};
        unsigned int out[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            unsigned int r = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const unsigned int u = w[2 * h + j];   // four codes -> two bytes
                const unsigned int b0 = (u & 0xf) | ((u >> 4) & 0xf0);
                const unsigned int b1 = ((u >> 16) & 0xf) | ((u >> 20) & 0xf0);
                r |= (b0 | (b1 << 8)) << (16 * j);
            }
            out[h] = r;
        }
        reinterpret_cast<uint2*>(packed)[i] = make_uint2(out[0], out[1]);
    }
    const long long nb = (n + 1) >> 1;
    for (long long b = (n16 << 3) + tid0; b < nb; b += stride) {
        const unsigned int lo = (unsigned char)codes[2 * b] & 0xf;
        const unsigned int hi = (2 * b + 1 < n) ? ((unsigned char)codes[2 * b + 1] & 0xf) : 0u;
        packed[b] = (unsigned char)(lo | (hi << 4));
    }
}

}  // namespace omse
