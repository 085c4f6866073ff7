// Short kernels (up to 1280 weights, e.g. 3x3x3 or 64x3x3): a group of G = 1, 2, 4, ... 32 lanes of a warp owns a row, which
// sits in their registers, and looks for the best candidate by evaluating a few of them, one after the other.  (The longer ones of
// them, and rows of up to 2304 weights, by a histogram: hist_search.)
//
// W(alpha) = sum_i sum_j (|x_i| - (j - 1/2)*alpha)_+ is convex, and the error is E - 2*alpha*W, so the errors at two
// candidates bound it from below at all candidates between them (the chord of W).  The powers of two of the grid are tried
// first, from the top down, until no smaller scale can win: the largest value, saturated, alone errs by more than the best
// candidate so far, or the chord from alpha = 0 says so.  An interval between two candidates that its chord does not exclude
// is split near the minimum of that bound, and so on, depth first: 20 evaluations for 27 Student-t values and 1024
// candidates, 25 for 576 Laplace values (49 on 8 bits), where one round of eight candidates per octave and everything
// between the open ones takes 60 to 90.  What stays open to the end are the candidates within 1e-5 of the minimum, so every
// candidate near enough to be decided in fp64 has been evaluated.
//
// Every lane of a group keeps the search's state; what differs between the groups of a warp is how many steps they take.
// As many values per lane as fit (40) before a group grows: a step of the search costs about as much as the evaluation of
// ten pairs of values, whatever the number of rows that share it (228,261 rows of 147 values: 476 us with 4 lanes of 40
// values, 604 with 8 of 20; 58,254 of 576 on 8 bits: 526 with 16 lanes of 36, 738 with 32 of 20).  Bound: issue of
// instructions; per evaluation and pair of values 4 packed FP32 operations and 4 more to saturate.
// Measured on one B200 with 1024 candidates, against a thread per row (up to 32 values) or a warp per row with a candidate
// per lane: 2,485,513 rows of 27 Student-t values 2.86 -> 1.11 ms (11.9 with the whole grid), 116,508 of 576 on 3 bits
// 1.72 -> 0.74; 1000 candidates, Laplace values: 1,000,000 rows of 33 1.96 -> 0.53 ms, 516,222 of 64 1.16 -> 0.48, 228,261 of
// 147 0.89 -> 0.48, 58,254 of 576 on 8 bits 0.70 -> 0.53, 40,000 of 1000 (against a block per row) 0.84 -> 0.52.
// A launch of few rows is bound by the chain of a row's steps instead (about 14 us); it takes the second search below.
#pragma once
#include "omse_lattice.cuh"

namespace omse {

constexpr int kShortThreads = 128;       // blocks of four warps: five per SM at 96 registers, against four at 128 and six at 80
constexpr int kShortBlocks = 5;          // (rows of 147 values 492 us, 503 and 514; of 27 values 1148, 1172 and 1267)
// Searches of rows_short_kernel; the last two take all lanes of a warp for one row.
constexpr int kBySplits = 0, kByLanes = 1, kByHistogram = 2;
constexpr int kShortMinQuads = 3;
constexpr int kShortQuads = 10;          // float4s of a row per lane, at most

// Lanes per row (log2) for rows of k values.
inline int short_lanes(long long k) {
    const long long quads = (k + 3) >> 2;
    int lg = 0;
    while (lg < 5 && quads > (long long)kShortQuads << lg) ++lg;
    return lg;
}
// Float4s from one row to the next in shared memory: 16-byte accesses of a quarter warp, 8/G rows, meet different banks.
__host__ __device__ inline int short_stride4(int k4, int lg) {
    const int g = 1 << lg;
    return lg >= 3 || (k4 & (2 * g - 1)) == g ? k4 : ((k4 + g - 1) & ~(2 * g - 1)) + g;
}
// Candidates tried first: n_cand and the powers of two below it.
__host__ __device__ inline int short_first(int n_cand) {
    int n = 1;
    for (int p = 1; p < n_cand; p <<= 1) ++n;
    return n;
}
// Slots of a group's stack of candidates: those, and one for each split of an interval whose upper part is split again.  A
// split leaves at most w - max(1, w/4) of a width w on either side, below the top kShortFree of them half.
constexpr int kShortFree = 5;
inline int short_slots(int n_cand) {
    int depth = 0;
    for (int w = n_cand; w >= 2; ++depth) {
        const int q = depth < kShortFree ? w / 4 : w / 2;
        w -= q > 1 ? q : 1;
    }
    return short_first(n_cand) + depth;
}

// Sums and maxima over the lanes of a group: every lane ends with the same bits (a + b == b + a).
template <class V>
__device__ __forceinline__ V group_sum(V v, int lg) {
    if (lg == 0) return v;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const V other = __shfl_xor_sync(0xffffffffu, v, 1 << s);
        v = s < lg ? v + other : v;
    }
    return v;
}
__device__ __forceinline__ float group_max(float v, int lg) {
    if (lg == 0) return v;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const float other = __shfl_xor_sync(0xffffffffu, v, 1 << s);
        v = s < lg ? fmaxf(v, other) : v;
    }
    return v;
}

// Shared memory of one warp.
struct ShortSmem {
    float4* xs;            // [group][short_stride4] the rows of a step, zero padded
    float2* stack;         // [slot][group] a candidate's index + 1 and 2*step*W there; or the histogram
    signed char* qs;       // the rows' codes on the way out, in the same place
    unsigned short* close; // [kShortClose][group] candidates within the noise band of the smallest error
};
// A row with one value far above the others has equal errors at every candidate that divides it without remainder, and
// decides among them in fp64.  Four places (and the whole stretch of the grid between them otherwise) let a few such rows in a
// hundred thousand hold up the launch: 116,508 rows of 576 Student-t values on 3 bits 1.55 -> 0.97 ms.
constexpr int kShortClose = 12;

__device__ __forceinline__ float quick_reciprocal(float a) {      // to an ulp, one instruction; subnormal numbers count as zero
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// Upper bound of E - error on (a0, a1) by the chord of W, that is the maximum of a*(c - s*a); at: where it lies.  A value
// that is not finite gives a bound that is not either (and then compares as open).
__device__ __forceinline__ float chord_gain(float a0, float w0, float a1, float w1, float& at) {
    const float s = (w0 - w1) * quick_reciprocal(a1 - a0), c = fmaf(s, a0, w0);
    at = s > 0.f ? fminf(fmaxf(0.5f * c * quick_reciprocal(s), a0), a1) : a1;
    return at * fmaf(-s, at, c);
}

struct ShortRow {
    int k4, lg, g, j;      // float4s; lanes per row (log2); group of this lane, lane of its group
    bool search;
    float step, sc;        // grid; power of two that the values are multiplied by where their squares would leave binary32
    float mpos, mneg, e, l1, w_zero;    // scaled: maxima of the positive and negative part, sums of squares and magnitudes, 2*step*W at alpha = 0
    float flo, fhi;
};
// The candidates that may be the minimum, by their index + 1: the one with the smallest binary32 error, the others within the
// noise band of that error (a list or, where they are too many, the window [w_lo, w_hi] of the indexes), evaluations.
struct ShortResult {
    float best, w_lo, w_hi, n_eval;
    int n_close;
};

template <int NQ>
__device__ __forceinline__ ShortResult short_search(const ShortSmem& sm, const ShortRow& r, int n_cand) {
    const int lg = r.lg, groups = 32 >> lg;
    const float step = r.step * r.sc, e = r.e, slack = 2e-6f * e;          // rounding of E and of the binary32 bounds
    u64 x2[2 * NQ];
    {
        const float4* src = sm.xs + r.g * short_stride4(r.k4, lg);
        const u64 sc2 = pack2(r.sc, r.sc), zero2 = pack2(-0.f, -0.f);
#pragma unroll
        for (int t = 0; t < NQ; ++t) {
            const int q4 = r.j + (t << lg);
            const float4 v = r.search && q4 < r.k4 ? src[q4] : make_float4(0.f, 0.f, 0.f, 0.f);
            x2[2 * t] = fma2(pack2(v.x, v.y), sc2, zero2);
            x2[2 * t + 1] = fma2(pack2(v.z, v.w), sc2, zero2);
        }
    }
    const float sat_alpha = r.search ? fmaxf(__fdividef(r.mpos, r.fhi + 0.5f), __fdividef(r.mneg, 0.5f - r.flo)) * 1.00002f : 0.f;
    const u64 M2 = pack2(kMagic, kMagic), NM2 = pack2(-kMagic, -kMagic);
    const float clo = kMagic + r.flo, chi = kMagic + r.fhi;
    // squared error of the row at candidate a1 - 1; the reciprocal by one step of Newton's method from the quick one
    auto error_at = [&](float a1) -> float {
        const float ac = __fmul_rn(a1, r.step);
        const float al = ac * r.sc, rough = quick_reciprocal(al), inv = fmaf(fmaf(-al, rough, 1.0f), rough, rough);
        const u64 inv2 = pack2(inv, inv), na2 = pack2(-al, -al);
        u64 acc_a = 0ull, acc_b = 0ull;                  // two accumulators: shorter dependency chain
        if (__any_sync(0xffffffffu, al < sat_alpha)) {   // some value saturates
#pragma unroll
            for (int p = 0; p < 2 * NQ; ++p) {
                float t0, t1;
                unpack2(fma2(x2[p], inv2, M2), t0, t1);
                t0 = fminf(fmaxf(t0, clo), chi);
                t1 = fminf(fmaxf(t1, clo), chi);
                const u64 d = fma2(na2, add2(pack2(t0, t1), NM2), x2[p]);
                if (p & 1) acc_b = fma2(d, d, acc_b);
                else acc_a = fma2(d, d, acc_a);
            }
        } else {
#pragma unroll
            for (int p = 0; p < 2 * NQ; ++p) {
                const u64 d = fma2(na2, add2(fma2(x2[p], inv2, M2), NM2), x2[p]);
                if (p & 1) acc_b = fma2(d, d, acc_b);
                else acc_a = fma2(d, d, acc_a);
            }
        }
        float p0, p1;
        unpack2(add2(acc_a, acc_b), p0, p1);
        const float v = group_sum(p0 + p1, lg);
        return usable_scale(ac) ? v : INFINITY;
    };
    // The candidates are not met in order of their index.  Beside the smallest error the search keeps those that may lie
    // within the noise band of the final minimum: a candidate inside the band of the final minimum is inside the band of
    // the running minimum when it is seen (the running minimum only falls), and when the running minimum falls by more than
    // the band everything seen before drops out.
    ShortResult res = {0.f, 0.f, 0.f, 0.f, 0};
    float best_v = INFINITY;
    const float band_f = 1.0f + 1.25f * (float)kRescoreBand;
    // first candidate i (0: the top of the grid) goes to slot n_first - 1 - i, so that the next lower one is always on top
    const int n_first = short_first(n_cand);
    float2* stack = sm.stack + r.g;
    unsigned short* close = sm.close + r.g;
    int sp = n_first - 1, bottom = 0;
    const float top = (float)n_cand;
    float a1 = top, w1 = 0.f, at = top;                  // upper end of the interval, candidate to evaluate
    bool busy = r.search, first = true;
    while (__any_sync(0xffffffffu, busy)) {
        const float v = error_at(at), w = (e - v) * quick_reciprocal(at);
        if (busy && v <= best_v * band_f) {
            const bool fresh = v * band_f < best_v, better = v < best_v || (v == best_v && at < res.best);
            res.n_close = fresh ? 0 : res.n_close;
            res.w_lo = fresh ? at : fminf(res.w_lo, at);
            res.w_hi = fresh ? at : fmaxf(res.w_hi, at);
            best_v = better ? v : best_v;
            res.best = better ? at : res.best;
            close[min(res.n_close, kShortClose - 1) * groups] = (unsigned short)at;
            ++res.n_close;
        }
        res.n_eval += busy ? 1.f : 0.f;
        const float room = e - fmaf(best_v, 1.00001f, slack);
        sp += busy && !first ? 1 : 0;
        if (busy) stack[sp * groups] = make_float2(at, w);
        if (busy && first) {
            if (at == top) w1 = w;
            const float low = (at - 1.f) * step, over = fmaxf(r.mpos - r.fhi * low, r.flo < 0.f ? r.mneg + r.flo * low : 0.f);
            float unused;
            if (sp == 0 || (over > 0.f && over * over > e - room) ||
                chord_gain(0.f, r.w_zero, at, w, unused) < room - 1e-5f * e) {
                first = false;
                bottom = sp;
                sp = n_first - 2;
            } else {
                --sp;
                at = (float)(1 << sp);
            }
        }
        bool pop = busy && !first;
        busy = busy && first;
        while (pop && sp >= bottom) {
            const float2 lower = stack[sp * groups];
            float peak;
            const float gain = chord_gain(lower.x, lower.y, a1, w1, peak), width = a1 - lower.x;
            const float q = fmaxf(1.f, floorf((sp < n_first - 2 + kShortFree ? 0.25f : 0.5f) * width));
            busy = width >= 2.f && !(gain < room);
            pop = !busy;
            at = fminf(fmaxf(rintf(peak), lower.x + q), a1 - q);
            a1 = busy ? a1 : lower.x;
            w1 = busy ? w1 : lower.y;
            sp -= busy ? 0 : 1;
        }
    }
    return res;
}

template <int NQ>
__device__ __forceinline__ ShortResult short_dispatch(int quads, const ShortSmem& sm, const ShortRow& r, int n_cand) {
    if constexpr (NQ > kShortMinQuads) {
        if (quads < NQ) return short_dispatch<NQ - 1>(quads, sm, r, n_cand);
    }
    return short_search<NQ>(sm, r, n_cand);
}

// ---- The search for the longer ones of the short rows: a warp makes one histogram of its row, as the block path does (see
// omse_lattice.cuh), and looks the candidates up.  What is different: the count and the fractional sum of a bin share one word
// (random words of shared memory take an atomic of a warp eight clocks, whatever is added), the fraction has eight to twelve bits, so
// that bin and fraction are bit fields of one multiply-add's result, and the extra negative level has no histogram: counting it on both
// sides gives a lower bound of the error, the largest negative value alone an upper one, and only the candidates that these leave
// open (some 40 of 1024) get the exact sum over the few values that lie beyond it.  If more than one is within the noise of the
// fractions, they are evaluated in binary32, as the splits do.
// Bound: chains of dependent instructions (12 to 20 warps per SM, 0.54 to 0.59 of an instruction per clock and scheduler) and fetching
// them: of some 7.3 cycles between two instructions of a warp (39,062 rows of 1024 values on 4 bits) 1.9 are the fixed latency, 1.45 missing
// instructions (1.9 at 576 values, 0.7 on 8 bits), 1.0 shared memory.  Measured on one B200, 1024 candidates, 67M Laplace values, against
// splits (up to 1024 values) and a block per row: 4 bits, 512 values a row 888 -> 821 us, 1024 838 -> 642, 1280 1013 -> 611, 2304 705 -> 580;
// 8 bits, 1024 1007 -> 781, 2304 786 -> 565.
struct HistShape {
    int n_bins, lb, fbits, cshift;        // bins; log2 of a lane's run of them; bits of a fraction; the count's place in the word
};
constexpr int kHistOpen = 4;              // open candidates per lane at a time
__device__ __forceinline__ bool hist_search(const ShortSmem& sm, const ShortRow& r, int k, int n_cand, const HistShape& g, ShortResult& res) {
    const int lane = threadIdx.x & 31;
    unsigned int* P = reinterpret_cast<unsigned int*>(sm.stack);
    float* coarse = reinterpret_cast<float*>(P + (32 << g.lb));
    res = ShortResult{0.f, 0.f, 0.f, 0.f, 0};
    if (!r.search) return true;                               // (the same in all lanes)
    if (r.sc != 1.0f) return false;
    const int lb = g.lb, run = 1 << lb, levels = (int)r.fhi, n_bins = g.n_bins;
    const bool sgn = r.flo < 0.f;
    const int d = sgn ? 2 * (int)(-r.flo) - 1 : 0;
    for (int i = lane; i < (8 << lb); i += 32) reinterpret_cast<uint4*>(P)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    // ---- insertion
    const float h = 0.5f * r.step, inv = __fdiv_rn(1.0f, h);
    {
        const float inv_b = inv * (float)(1 << g.fbits), base = 8388608.0f - (float)(1 << g.fbits);      // 2^23: bin 1 is word 0
        const unsigned int mask = (1u << g.fbits) - 1u, one = 1u << g.cshift;
        const int s1 = g.fbits, s2 = g.fbits + lb - 2;
        const unsigned int at = (unsigned)__cvta_generic_to_shared(P) - 4u * (0x4B000000u >> s1);
#pragma unroll 2
        for (int i = lane; i < r.k4; i += 32) {
            const float4 v = sm.xs[i];
            const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float u = fmaf(sgn ? fabsf(y[j]) : y[j], inv_b, base);
                const unsigned int bits = __float_as_uint(u);
                if (u >= 8388608.0f) shared_add(at + 4u * ((bits >> s1) ^ ((bits >> s2) & 0x1cu)), (bits & mask) | one);
            }
        }
    }
    __syncwarp();
    // ---- P(m) at word m - 1, in units of 2^-shift.  Counts and fractions of all bins together stay in their fields, so one addition
    //      does for both.
    int shift;
    {
        const int first = lane << lb;
        const unsigned int fmask = (1u << g.cshift) - 1u;
        unsigned int a = 0u, s = 0u;
        for (int q = run - 4; q >= 0; q -= 4) {
            const uint4 w = *reinterpret_cast<const uint4*>(P + lattice_word(first + q, lb));
            s += a >> g.cshift;
            a += w.w;
            s += a >> g.cshift;
            a += w.z;
            s += a >> g.cshift;
            a += w.y;
            s += a >> g.cshift;
            a += w.x;
        }
        const unsigned int own_a = a, own_s = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int a2 = __shfl_down_sync(0xffffffffu, a, o), s2 = __shfl_down_sync(0xffffffffu, s, o);
            if (lane + o < 32) {
                s += s2 + ((unsigned)o << lb) * (a2 >> g.cshift);
                a += a2;
            }
        }
        const unsigned int total_a = __shfl_sync(0xffffffffu, a, 0), total_s = __shfl_sync(0xffffffffu, s, 0);
        shift = scan_shift(total_a >> g.cshift, total_s, g.fbits);
        // what lies behind this lane's run, at the run's end
        a -= own_a;
        s -= own_s + (unsigned)run * (a >> g.cshift);
        const int drop = g.fbits - shift;
        for (int q = run - 4; q >= 0; q -= 4) {
            uint4* at = reinterpret_cast<uint4*>(P + lattice_word(first + q, lb));
            uint4 w = *at;
            auto put = [&](unsigned int x) {
                s += a >> g.cshift;
                a += x;
                return (s << shift) + ((a & fmask) >> drop);
            };
            w.w = put(w.w);
            w.z = put(w.z);
            w.y = put(w.y);
            w.x = put(w.x);
            *at = w;
        }
    }
    __syncwarp();
    // ---- errors in units of h^2, E less its share of the levels
    const double e = (double)r.e * (double)inv * (double)inv, scale = -4.0 * __longlong_as_double((long long)(1023 - shift) << 52);
    const float ef = (float)e, q = __int_as_float((127 - shift) << 23), qn = shift < g.fbits ? (2.0f * (float)n_bins + 8.0f * (float)n_cand) * q : 0.f;
    const float s1 = r.l1 * inv, inv_f = __int_as_float((127 - g.fbits) << 23);
    auto upper_sum = [&](int a1, int first, int stride) -> unsigned long long {
        unsigned long long acc = 0ull;
        const int last = min(n_bins, (2 * levels - 1) * a1);
        for (int m = (2 * first + 1) * a1; m <= last; m += 2 * stride * a1) acc += P[lattice_word(m - 1, lb)];
        return acc;
    };
    auto usable = [&](int a1) { return usable_scale(__fmul_rn((float)a1, r.step)); };
    auto error = [&](int a1, unsigned long long p) { return usable(a1) ? (float)fma(scale * (double)a1, u52_double(p), e) : INFINITY; };
    // The extra level's sum lies between what the largest negative value alone gives and what all values give less the largest
    // positive one's.
    const float t_pos = r.mpos * inv, t_neg = r.mneg * inv;
    auto alone = [&](float t, int m) -> unsigned int {
        return d > 0 ? (unsigned int)(fmaxf(t * 0.999999f - (float)m - 0.01f, 0.f) * (float)(1 << shift)) : 0u;
    };
    auto beyond = [&](int a1) -> unsigned int {
        const int m = d * a1;
        if (d == 0 || !(t_neg > (float)m) || m > n_bins) return 0u;
        const unsigned int all = P[lattice_word(m - 1, lb)];
        return all - min(all, alone(t_pos, m));
    };
    // ---- coarse candidates: upper bounds give the threshold, lower bounds are kept
    const int n_coarse = coarse_count(n_cand);
    float least = INFINITY;
    auto note = [&](int i, int a1, unsigned long long p) {
        least = fminf(least, error(a1, p + alone(t_neg, d * a1)));
        coarse[i] = error(a1, p + beyond(a1));
    };
    int done = 0;
    if (levels > 8) {
        // The smallest scales have the most levels: 8 lanes share each of the first 16, 4 each of the next 8.  The smallest of all, which
        // leave the largest value further away than the whole error is at the first scale that reaches it, are not looked at.  (Of the values
        // that the range reaches: on an unsigned one the negative values err by as much at every scale.)
        const float t_max = sgn ? fmaxf(t_pos, t_neg) : t_pos, reach = ceilf(__fdividef(t_max, (float)(2 * levels + 1)) * 1.00001f) * 1.0001f;
        const int skip = reach <= (float)n_cand ? max(0, (int)floorf(__fdividef(t_max - sqrtf((float)k) * reach, (float)(2 * levels + 2)) * 0.9999f) - 1) : 0;
        for (int i = lane; i < min(min(skip, 16), n_coarse); i += 32) coarse[i] = 3e38f;
        auto shared = [&](int from, int to, int lanes) {
            for (int i0 = from; i0 < to; i0 += 32 / lanes) {
                const int i = i0 + lane / lanes, a1 = coarse_a1(i, n_cand);
                unsigned long long p = i < to ? upper_sum(a1, lane & (lanes - 1), lanes) : 0ull;
                for (int o = 1; o < lanes; o <<= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
                if (i < to && (lane & (lanes - 1)) == 0) note(i, a1, p);
            }
        };
        shared(min(skip, 16), min(16, n_coarse), 8);
        shared(16, min(24, n_coarse), 4);
        done = 24;
    }
    for (int i = done + lane; i < n_coarse; i += 32) {
        const int a1 = coarse_a1(i, n_cand);
        note(i, a1, upper_sum(a1, 0, 1));
    }
    __syncwarp();
    // (values may be below zero by what E is off)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
    if (!(least < INFINITY)) return true;                     // no usable scale
    // What a candidate may be off by.  The fractions: 2^-(F+1) per value and level, at most T/(2*a1) + 1/2 levels of 4*a1 each for the values
    // from T = a1 on, so 2^-F times twice the sum of those.  The truncation of P, where there is any.  And, as in lattice_band, what the
    // scales' and the quotients' rounding move (the reciprocal's, the same for all values, among them).
    auto band = [&](float v, float fractions) {
        const float dv = fmaxf(v, 0.f) + 2e-6f * ef;
        return v + (float)kRescoreBand * dv + 2.0f * (fractions + qn + 6e-7f * sqrtf(dv * ef) + 1e-9f * ef);
    };
    float fractions = 2.0f * inv_f * s1;
    int lo, hi;
    // Where much of the grid is open, which is where one value lies far above the others, few values lie beyond the smallest open candidate
    // `lo`: P(lo) + lo*(P(lo - 1) - P(lo)) is at least their sum.  Once more with that.  (Such a row held up a launch of few rows per warp: 1776
    // rows of 2304 Student-t values, 4 bits, 1024 candidates 55 us by blocks, 92 with the sum of all values and a truncation that does
    // not take place, 58 so; 2400 rows on 5 bits 70, 99, 75; 12,000 on 4 bits 298, 260, 227.)
#pragma unroll 1
    for (bool again = false;; again = true) {
        const float keep = band(least, fractions) + 1e-6f * ef;            // 1e-6: binary32 in the bounds below
        lo = 0x7fffffff;
        hi = -1;
        for (int i = lane; i < n_coarse; i += 32) {
            const int a0 = coarse_a1(i, n_cand);
            if (!(coarse[i] > keep)) {
                lo = min(lo, a0);
                hi = max(hi, a0);
            }
            if (i + 1 >= n_coarse) continue;
            const int a1 = coarse_a1(i + 1, n_cand);
            if (a1 - a0 >= 2 && !(chord_bound(ef, a0, coarse[i], a1, coarse[i + 1]) > keep)) {      // (an unusable end keeps the interval)
                lo = min(lo, a0 + 1);
                hi = max(hi, a1 - 1);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (again || hi - lo < 32 * kHistOpen) break;
        if (lo > 1 && lo <= n_bins) {
            const unsigned int here = P[lattice_word(lo - 1, lb)], before = P[lattice_word(lo - 2, lb)];
            fractions = 2.0f * inv_f * q * fmaf((float)lo, (float)(before - here + 1u), (float)here + 1.0f);
        }
    }
    // ---- the open candidates, four to a lane at a time, with the extra level as it is: the negative values beyond it are met one by
    //      one.  First the smallest error, then the candidates within the noise (found again where there were more than one lot).
    float value[kHistOpen], best = INFINITY, most = 0.f, limit = 0.f, single = 0.f, best_v = INFINITY;
    int met = 0, n_left = 0;
    // a candidate within the noise by its binary32 error (the same in all lanes); what is kept is what short_search keeps
    auto consider = [&](float a1) {
        const float v = warp_allsum(direct_part<false>(sm.xs, r.k4, lane, 32, __fmul_rn(a1, r.step), 1.0f, r.flo, r.fhi));
        const float band_f = 1.0f + 1.25f * (float)kRescoreBand;
        res.n_eval += 1.f;
        if (!(v <= best_v * band_f)) return;
        const bool fresh = v * band_f < best_v;
        res.n_close = fresh ? 0 : res.n_close;
        res.w_lo = fresh ? a1 : res.w_lo;
        res.w_hi = a1;
        if (v < best_v) {                                     // (increasing scales: the lowest one keeps a tie)
            best_v = v;
            res.best = a1;
        }
        sm.close[min(res.n_close, kShortClose - 1)] = (unsigned short)a1;
        ++res.n_close;
    };
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int first = lo; first <= hi; first += 32 * kHistOpen) {
            const int last = min(hi, first + 32 * kHistOpen - 1);
            if (pass == 0 || hi - lo >= 32 * kHistOpen) {
                float extra[kHistOpen] = {0.f, 0.f, 0.f, 0.f};
                if (d > 0 && t_neg > (float)(d * first)) {
                    const float from = -((float)(d * first) * h);
#pragma unroll 1
                    for (int i0 = 0; i0 < r.k4; i0 += 32) {
                        const float4 v = i0 + lane < r.k4 ? sm.xs[i0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
                        const float y[4] = {v.x, v.y, v.z, v.w};
                        if (!__any_sync(0xffffffffu, fminf(fminf(fminf(y[0], y[1]), y[2]), y[3]) < from)) continue;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            unsigned int some = __ballot_sync(0xffffffffu, y[j] < from);
                            met += __popc(some);
                            while (some) {
                                const float t = -__shfl_sync(0xffffffffu, y[j], __ffs(some) - 1) * inv;
                                some &= some - 1;
#pragma unroll
                                for (int c = 0; c < kHistOpen; ++c) {
                                    if (first + 32 * c > last) break;
                                    extra[c] += fmaxf(t - (float)(d * (first + lane + 32 * c)), 0.f);
                                }
                            }
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < kHistOpen; ++c) {
                    const int a1 = first + lane + 32 * c;
                    value[c] = INFINITY;
                    if (a1 <= last) {
                        const float gain = 4.0f * (float)a1 * extra[c];
                        value[c] = error(a1, upper_sum(a1, 0, 1)) - gain;
                        most = fmaxf(most, gain);
                    }
                    best = fminf(best, value[c]);
                }
            }
            if (pass == 0) continue;
            unsigned int within[kHistOpen];
#pragma unroll
            for (int c = 0; c < kHistOpen; ++c) within[c] = __ballot_sync(0xffffffffu, value[c] <= limit);
            // One copy of the evaluation in the code, not eight: the warps of this kernel wait for instructions (30,000 rows of 1152 values, 4
            // bits, no polish step 255 -> 238 us, with three 325 -> 318).
            static_assert(kHistOpen == 4, "a ballot for each candidate of a lane");
#pragma unroll 1
            for (int c = 0; c < kHistOpen; ++c) {
                unsigned int some = c == 0 ? within[0] : c == 1 ? within[1] : c == 2 ? within[2] : within[3];
#pragma unroll 1
                while (some) {
                    const float a1 = (float)(first + __ffs(some) - 1 + 32 * c);
                    some &= some - 1;
                    if (n_left == 0) single = a1;             // (left as it is if it is the only one)
#pragma unroll 1
                    for (int i = n_left == 1 ? 0 : n_left == 0 ? 2 : 1; i < 2; ++i) consider(i == 0 ? single : a1);
                    ++n_left;
                }
            }
        }
        if (pass == 1) break;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
            most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
        }
        if (!(best < INFINITY)) return true;
        // (binary32 in the sums of `extra`: values by 1.2e-7, the additions by half of that each)
        limit = band(best, fractions) + 2.0f * (1.2e-7f + 6e-8f * (float)met) * most + 2.5e-7f * ef / (float)max(d, 1);
    }
    res.n_eval += 1.f;
    if (n_left == 1) {
        res.best = res.w_lo = res.w_hi = single;
        res.n_close = 1;
    }
    __syncwarp();                                             // the list
    return true;
}

// ---- The search for small launches, where a row's chain of evaluations is what counts: the whole warp on one row, a
// candidate per lane.  Eight candidates per octave first, then everything between the ones whose chord excludes nothing: two
// or three rounds (2400 rows of 64 values 27 -> 15 us).
constexpr int kMaxCoarse = 80;           // coarse_count(OMSE_MAX_CANDIDATES)
constexpr int kHullValues = 256;         // errors of the neighbourhood of the minimum that are kept

// The candidates that are tried first, from the top of the grid down (s = 0, 1, ...): eight per octave, all below 16.  The
// top two octaves hold two and four when the range has at least seven codes on a side and the row 192 values: the best
// scale then lies below them (4 bits: max|x|/9 on average), and the 32 lanes of a warp reach down to C/36 at once (30,000
// rows of 576 values 426 -> 310 us).  2 and 3 bits keep all eight (best scale at max|x|/3 and max|x|/5), and so do shorter
// rows, whose largest value alone can make a large scale good: the wide intervals are then not excluded (147 values 135 ->
// 168 us with two and four, 256 values 218 -> 178).
struct CoarseGrid {
    int n_cand, full, n;         // candidates, coarse_count, how many of them are tried
    __device__ __forceinline__ CoarseGrid(int n_cand_, float fhi, int k) : n_cand(n_cand_), full(coarse_count(n_cand_)) {
        n = fhi >= 7.f && k >= 192 && full >= 42 ? full - 10 : full;
    }
    __device__ __forceinline__ int a1(int s) const {
        const int off = n == full ? s : s < 2 ? 4 * s : s < 6 ? 4 + 2 * s : s + 10;
        return coarse_a1(max(full - 1 - off, 0), n_cand);
    }
};
// Squared error of the row at one scale per lane; packed pairs, folded every 128 values so that the rounding noise stays
// near 1e-7 relative.  CL: some lane's scale saturates some value.
template <bool CL, bool SC>
__device__ __forceinline__ float direct_sum(const float4* xs4, const ShortRow& r, float alpha) {
    const float inv = __fdiv_rn(1.0f, alpha), clo = kMagic + r.flo, chi = kMagic + r.fhi;
    const u64 M2 = pack2(kMagic, kMagic), NM2 = pack2(-kMagic, -kMagic), inv2 = pack2(inv, inv), na2 = pack2(-alpha, -alpha);
    const u64 sc2 = pack2(r.sc, r.sc), z2 = pack2(-0.f, -0.f);
    u64 tot = 0ull;
    for (int i = 0; i < r.k4;) {
        const int stop = min(r.k4, i + kFlushEvery4);
        u64 acc_a = 0ull, acc_b = 0ull;
#pragma unroll 4
        for (; i < stop; ++i) {
            const float4 v = xs4[i];
            u64 xa = pack2(v.x, v.y), xb = pack2(v.z, v.w);
            if (SC) {
                xa = fma2(xa, sc2, z2);
                xb = fma2(xb, sc2, z2);
            }
            u64 ta = fma2(xa, inv2, M2), tb = fma2(xb, inv2, M2);
            if (CL) {
                float a0, a1, b0, b1;
                unpack2(ta, a0, a1);
                unpack2(tb, b0, b1);
                ta = pack2(fminf(fmaxf(a0, clo), chi), fminf(fmaxf(a1, clo), chi));
                tb = pack2(fminf(fmaxf(b0, clo), chi), fminf(fmaxf(b1, clo), chi));
            }
            const u64 ea = fma2(na2, add2(ta, NM2), xa), eb = fma2(na2, add2(tb, NM2), xb);
            acc_a = fma2(ea, ea, acc_a);
            acc_b = fma2(eb, eb, acc_b);
        }
        tot = add2(tot, add2(acc_a, acc_b));
    }
    float p0, p1;
    unpack2(tot, p0, p1);
    return p0 + p1;
}
// Out of line: inlined wherever candidates are evaluated, its loops would be most of the code.
__device__ __noinline__ float direct_error_at(const float4* xs4, int k4, float step, float sc, float sat_alpha, float flo, float fhi, int c) {
    ShortRow r;
    r.k4 = k4;
    r.sc = sc;
    r.flo = flo;
    r.fhi = fhi;
    const float ac = __fmul_rn((float)(c + 1), step);
    const bool ok = usable_scale(ac);
    const float al = ok ? ac * sc : 1.0f;
    float v;
    if (sc != 1.0f) v = direct_sum<true, true>(xs4, r, al);
    else if (__any_sync(0xffffffffu, al < sat_alpha)) v = direct_sum<true, false>(xs4, r, al);
    else v = direct_sum<false, false>(xs4, r, al);
    return ok ? v : INFINITY;
}
// errors are not negative: they order like their bit patterns
__device__ __forceinline__ float warp_min_error(float v) { return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v))); }

__device__ __forceinline__ ShortResult direct_search(const ShortSmem& sm, const ShortRow& r, int n_cand) {
    const int lane = threadIdx.x & 31;
    ShortResult res = {0.f, 0.f, 0.f, 0.f, 0};
    if (!r.search) return res;                                // (the same in all lanes)
    float* coarse = reinterpret_cast<float*>(sm.stack);
    float* hull = coarse + kMaxCoarse;
    const float e = r.e, slack = 2e-6f * e;
    const float sat_alpha = fmaxf(__fdividef(r.mpos, r.fhi + 0.5f), __fdividef(r.mneg, 0.5f - r.flo)) * 1.00002f;   // margin for the rounding of x*inv
    auto direct_error = [&](int c) { return direct_error_at(sm.xs, r.k4, r.step, r.sc, sat_alpha, r.flo, r.fhi, c); };
    // ---- coarse candidates from the top down, 32 at a time, until no smaller scale can win
    const CoarseGrid cg(n_cand, r.fhi, 4 * r.k4);
    int tried = 0, bi = 0x7fffffff;
    float bv = INFINITY, best = INFINITY;
    for (;;) {
        const int i = tried + lane, a1 = cg.a1(min(i, cg.n - 1));
        const float v = direct_error(a1 - 1);
        bool below = false;                                   // no scale below this one can win
        if (i < cg.n) {
            coarse[i] = v;
            if (v < bv || (v == bv && a1 - 1 < bi)) {
                bv = v;
                bi = a1 - 1;
            }
        }
        res.n_eval += (float)min(32, cg.n - tried);
        tried = min(cg.n, tried + 32);
        best = warp_min_error(bv);
        if (tried == cg.n) break;
        if (lane == 31) {
            const float al = __fmul_rn((float)(a1 - 1), r.step) * r.sc, keep = best * 1.00001f + slack;
            const float over = fmaxf(r.mpos - r.fhi * al, r.flo < 0.f ? r.mneg + r.flo * al : 0.f);
            below = (over > 0.f && over * over > keep) ||
                    chord_bound_w(e, 0.f, r.w_zero, (float)a1, __fdividef(e - v, (float)a1)) > keep + 1e-5f * e;
        }
        if (__any_sync(0xffffffffu, below)) break;
    }
    __syncwarp();
    // ---- the stretch of the grid that the chords do not exclude
    const float keep = best * 1.00001f + slack;
    int lo = 0x7fffffff, hi = -1;
    for (int i = lane; i + 1 < tried; i += 32) {
        const int a0 = cg.a1(i + 1), a1 = cg.a1(i);
        if (a1 - a0 >= 2 && !(chord_bound(e, a0, coarse[i + 1], a1, coarse[i]) > keep)) {   // (an unusable end keeps the interval)
            lo = min(lo, a0);
            hi = max(hi, a1 - 2);
        }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    for (int c0 = lo; c0 <= hi; c0 += 32) {
        const int c = min(c0 + lane, hi);
        const float v = direct_error(c);
        if (c0 + lane <= hi && c - lo < kHullValues) hull[c - lo] = v;
        if (v < bv || (v == bv && c < bi)) {
            bv = v;
            bi = c;
        }
        res.n_eval += (float)min(32, hi - c0 + 1);
    }
    best = warp_min_error(bv);
    if (!(best < INFINITY)) return res;                       // every error is Inf or NaN
    res.best = (float)__reduce_min_sync(0xffffffffu, (unsigned)(bv == best ? bi : 0x7fffffff)) + 1.f;
    // ---- the candidates within the band
    const float band = (float)((double)best * (1.0 + kRescoreBand));
    int c_lo = 0x7fffffff, c_hi = -1;
    __syncwarp();
    auto meet = [&](float v, int c) {                         // one candidate per lane, Inf for none
        const bool close = v <= band;
        const unsigned int mask = __ballot_sync(0xffffffffu, close);
        const int at = res.n_close + __popc(mask & ((1u << lane) - 1u));
        if (close) {
            if (at < kShortClose) sm.close[at] = (unsigned short)(c + 1);
            c_lo = min(c_lo, c);
            c_hi = max(c_hi, c);
        }
        res.n_close += __popc(mask);
    };
    for (int i0 = 0; i0 < tried; i0 += 32) {
        const int i = i0 + lane, c = cg.a1(min(i, tried - 1)) - 1;
        meet(i < tried && (c < lo || c > hi) ? coarse[i] : INFINITY, c);
    }
    for (int c0 = lo; c0 <= hi; c0 += 32) {
        const int c = min(c0 + lane, hi);
        const float v = hi - lo < kHullValues ? hull[c - lo] : direct_error(c);
        meet(c0 + lane <= hi ? v : INFINITY, c);
    }
    res.w_lo = (float)__reduce_min_sync(0xffffffffu, c_lo) + 1.f;
    res.w_hi = (float)__reduce_max_sync(0xffffffffu, c_hi) + 1.f;
    __syncwarp();                                             // the list
    return res;
}

// One step of a warp: nrows rows from row0 on, one per group.  carry: code of the element before the step's first one (only
// where that shares a byte of packed codes with it); more: the warp goes on with the next rows of the same tensor.
// Outside the search the rows are read from shared memory in loops that are not unrolled: the code of the passes, unrolled
// over registers, was most of the kernel, and warps waited for instructions (rows of 27 values 1.42 -> 1.20 ms).
template <int BY>
__device__ __forceinline__ void short_step(const RowArgs& a, const RowTensor& T, const ShortSmem& sm, int lg, long long row0, int nrows,
                                           bool more, int& carry, unsigned int& st, unsigned long long& ev) {
    const int lane = threadIdx.x & 31;
    ShortRow r;
    r.lg = lg;
    r.g = lane >> lg;
    r.j = lane & ((1 << lg) - 1);
    const int k = (int)T.K, k4 = (k + 3) >> 2, stride4 = short_stride4(k4, lg), n = nrows * k;
    r.k4 = k4;
    const bool active = r.g < nrows;
    const int own = active ? k4 : 0;                     // float4s r.j, r.j + G, ... below this are this lane's
    const long long row = row0 + r.g, flat0 = row0 * T.K;
    r.flo = (float)a.lo[0];
    r.fhi = (float)a.hi[0];
    const float flo = r.flo, fhi = r.fhi, thr = ambiguity_threshold(flo, fhi);

    // ---- the rows into shared memory
    __syncwarp();                                        // the previous step's rows and codes have been read
    const float* src = T.w + flat0;
    float* xs = reinterpret_cast<float*>(sm.xs);
    if ((k & 3) == 0 && (reinterpret_cast<unsigned long long>(src) & 15ull) == 0) {
        if (stride4 == k4) {
            for (int i = lane; i < (n >> 2); i += 32) cp_async16(xs + 4 * i, src + 4 * i);
        } else {
            const unsigned int rd = 0xffffffffu / (unsigned)k4 + 1u;      // i/k4 = (i*rd) >> 32 for i < 2^16 (k4 > 1)
            for (int i = lane; i < (n >> 2); i += 32) {
                const int rr = k4 == 1 ? i : (int)__umulhi((unsigned)i, rd);
                cp_async16(xs + 4 * (i + rr * (stride4 - k4)), src + 4 * i);
            }
        }
    } else {
        const unsigned int rd = 0xffffffffu / (unsigned)k + 1u;
        for (int i = lane; i < n; i += 32) {
            const int rr = k == 1 ? i : (int)__umulhi((unsigned)i, rd);
            cp_async4(xs + i + rr * (4 * stride4 - k), src + i);
        }
        if (lane < nrows)
            for (int i = k; i < 4 * k4; ++i) xs[lane * 4 * stride4 + i] = 0.f;
    }
    cp_async_wait();
    __syncwarp();
    float4* mine = sm.xs + r.g * stride4;
    if (T.delta) {                                       // quantization with offset: the row minimum is subtracted first
        float m = -INFINITY;
        const float* y = reinterpret_cast<const float*>(mine);
#pragma unroll 1
        for (int i = r.j; i < own; i += 1 << lg)
            for (int u = 4 * i; u < min(4 * i + 4, k); ++u)
                if (fabsf(y[u]) <= FLT_MAX) m = fmaxf(m, -y[u]);
        m = -group_max(m, lg);
        const float off = m < INFINITY ? m : 0.f;
#pragma unroll 1
        for (int i = r.j; i < own; i += 1 << lg)
            for (int u = 4 * i; u < min(4 * i + 4, k); ++u) reinterpret_cast<float*>(mine)[u] = y[u] - off;
        if (active && r.j == 0) T.delta[row] = off;
    } else if (T.prior_alpha) {                          // second tensor of a key layer: the residual of the first one
        const float a1 = active ? T.prior_alpha[row] : 0.f, inv = a1 > 0.f ? __fdiv_rn(1.0f, a1) : 0.f;
        if (a1 > 0.f)
#pragma unroll 1
            for (int i = r.j; i < own; i += 1 << lg) {
                const float4 v = mine[i];
                const float y[4] = {v.x, v.y, v.z, v.w};
                int q[4];
                exact_codes4(y, a1, inv, flo, fhi, thr, q);
                mine[i] = make_float4(fmaf(-a1, (float)q[0], y[0]), fmaf(-a1, (float)q[1], y[1]),
                                      fmaf(-a1, (float)q[2], y[2]), fmaf(-a1, (float)q[3], y[3]));
            }
    }
    // ---- maxima and sums; a power of two against overflow and underflow of the squares
    unsigned int abits = 0u;                             // largest bit pattern without the sign: tells non-finite values
    float mpos = 0.f, mneg = 0.f, e = 0.f, l1 = 0.f, l0 = 0.f;
#pragma unroll 1
    for (int i = r.j; i < own; i += 1 << lg) {
        const float4 v = mine[i];
        const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            abits = max(abits, __float_as_uint(y[u]) & 0x7fffffffu);
            mpos = fmaxf(mpos, y[u]);
            mneg = fmaxf(mneg, -y[u]);
            e = fmaf(y[u], y[u], e);
            l1 += fabsf(y[u]);
            l0 += y[u];
        }
    }
    if (abits >= 0x7f800000u) st |= 1u;
    mpos = group_max(mpos, lg);
    mneg = group_max(mneg, lg);
    const bool finite = group_max(abits >= 0x7f800000u ? 1.f : 0.f, lg) == 0.f;
    const Grid grid = grid_of(fmaxf(mpos, mneg), a.hi_frac, a.n_cand);
    r.search = active && finite && grid.usable;
    r.step = grid.step;
    const int ex = (int)(__float_as_uint(fmaxf(mpos, mneg)) >> 23) - 127;
    r.sc = 1.f;
    if (r.search && (ex < -40 || ex > 40)) {
        r.sc = __int_as_float((127 - max(min(ex, 126), -126)) << 23);
        e = l1 = l0 = 0.f;
#pragma unroll 1
        for (int i = r.j; i < own; i += 1 << lg) {
            const float4 v = mine[i];
            const float y[4] = {v.x * r.sc, v.y * r.sc, v.z * r.sc, v.w * r.sc};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                e = fmaf(y[u], y[u], e);
                l1 += fabsf(y[u]);
                l0 += y[u];
            }
        }
    }
    r.mpos = mpos * r.sc;
    r.mneg = mneg * r.sc;
    r.e = group_sum(e, lg);
    l1 = group_sum(l1, lg);
    l0 = group_sum(l0, lg);
    r.l1 = l1;
    r.w_zero = r.step * r.sc * (fhi * (l1 + l0) - flo * (l1 - l0));         // every level counts |x| in full

    ShortResult s;
    if constexpr (BY == kBySplits) {
        s = short_dispatch<kShortQuads>((k4 + (1 << lg) - 1) >> lg, sm, r, a.n_cand);
    } else {
        __syncwarp();                                    // the other lanes' part of the row
        bool found = false;
        if constexpr (BY == kByHistogram) {
            found = hist_search(sm, r, k, a.n_cand, HistShape{a.n_bins, a.hist_lb, T.hist_fbits, T.hist_cshift}, s);
            __syncwarp();
        }
        if (!found) s = direct_search(sm, r, a.n_cand);
    }

    // ---- candidates within the fp32 noise band of the minimum: decide in fp64 with exact codes
    const bool found = r.search && s.best > 0.f;
    {
        bool open = found && s.n_close > 1;
        const bool listed = s.n_close <= kShortClose;
        double best_sse = INFINITY;
        float win = 0.f;
        for (int i = 0; __any_sync(0xffffffffu, open); ++i) {
            float a1 = s.w_lo + (float)i;
            if (open && listed) a1 = (float)sm.close[(i << (5 - lg)) + r.g];
            const float ac = __fmul_rn(a1, r.step), inv = __fdiv_rn(1.0f, ac);
            const double ad = (double)ac;
            double ss = 0.0;
            const bool ok = open && usable_scale(ac);
#pragma unroll 1
            for (int q4 = r.j; q4 < (ok ? own : 0); q4 += 1 << lg) {    // the padding zeros code to 0 and add nothing
                const float4 v = mine[q4];
                const float y[4] = {v.x, v.y, v.z, v.w};
                int q[4];
                exact_codes4(y, ac, inv, flo, fhi, thr, q);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const double d = fma(-ad, int_double(q[u]), (double)y[u]);
                    ss = fma(d, d, ss);
                }
            }
            ss = group_sum(ss, lg);
            if (open) {
                s.n_eval += 1.f;
                if (ok && (ss < best_sse || (ss == best_sse && a1 < win))) {
                    best_sse = ss;
                    win = a1;
                }
                open = listed ? i + 1 < s.n_close : a1 < s.w_hi;
            }
        }
        if (win > 0.f) s.best = win;
    }
    if (r.j == 0) ev += (unsigned long long)s.n_eval * (4ull * k4);
    // ---- polish
    float alpha = found ? __fmul_rn(s.best, r.step) : 0.f;
    if (active && !found) st |= 2u;
    {
        bool open = found;
        for (int it = 0; it < a.refine_iters && __any_sync(0xffffffffu, open); ++it) {
            const float inv = found ? __frcp_rn(alpha) : 0.f;
            double sxq = 0.0;
            int sqq = 0;
#pragma unroll 1
            for (int q4 = r.j; q4 < (open ? own : 0); q4 += 1 << lg) {
                const float4 v = mine[q4];
                const float y[4] = {v.x, v.y, v.z, v.w};
                int q[4];
                exact_codes4(y, alpha, inv, flo, fhi, thr, q);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sqq += q[u] * q[u];
                    sxq = fma((double)y[u], int_double(q[u]), sxq);
                }
            }
            sxq = group_sum(sxq, lg);
            sqq = group_sum(sqq, lg);
            const float a_new = (float)(sxq / (double)sqq);
            open = open && sqq != 0 && a_new >= FLT_MIN && a_new <= FLT_MAX && a_new != alpha;   // a fixed point would repeat exactly
            if (open) alpha = a_new;
        }
    }
    // ---- final codes and error; the codes leave through shared memory, at the same offset from 8 elements.  They lie where the stack
    //      and the list have been: every lane's last look at those comes before any lane's first code (votes do not order memory).
    const int o = (int)(flat0 & 7);
    signed char* qs = sm.qs;
    __syncwarp();
    {
        const float inv = alpha > 0.f ? __fdiv_rn(1.0f, alpha) : 0.f;
        const double ad = (double)alpha;
        double ss = 0.0;
#pragma unroll 1
        for (int q4 = r.j; q4 < own; q4 += 1 << lg) {
            const float4 v = mine[q4];
            const float y[4] = {v.x, v.y, v.z, v.w};
            int q[4] = {0, 0, 0, 0};
            if (alpha > 0.f) exact_codes4(y, alpha, inv, flo, fhi, thr, q);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double d = fma(-ad, int_double(q[u]), (double)y[u]);
                ss = fma(d, d, ss);
            }
            signed char* dst = qs + o + r.g * k + 4 * q4;
            if ((k & 3) == 0) {
                *reinterpret_cast<unsigned int*>(dst) =
                    (q[0] & 0xff) | ((q[1] & 0xff) << 8) | ((q[2] & 0xff) << 16) | ((unsigned)(q[3] & 0xff) << 24);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (4 * q4 + u < k) dst[u] = (signed char)q[u];
            }
        }
        ss = group_sum(ss, lg);
        if (active && r.j == 0) {
            T.alpha[row] = alpha;
            T.sse[row] = (float)ss;
            if (T.best_idx) T.best_idx[row] = found ? (int)s.best - 1 : -1;
        }
    }
    const int end = o + n;
    if (lane == 0) {
        if (o & 1) qs[o - 1] = (signed char)carry;
        qs[end] = 0;
    }
    __syncwarp();
    if (T.codes) {
        signed char* dst = T.codes + (flat0 - o);
        int from = (o + 3) & ~3, to = end & ~3;
        if ((reinterpret_cast<unsigned long long>(T.codes) & 3ull) != 0 || from > to) from = to = end;
        for (int i = o + lane; i < from; i += 32) dst[i] = qs[i];
        for (int i = from + 4 * lane; i < to; i += 128) *reinterpret_cast<unsigned int*>(dst + i) = *reinterpret_cast<const unsigned int*>(qs + i);
        if (to + lane < end) dst[to + lane] = qs[to + lane];
    }
    if (T.packed) {
        unsigned char* dst = T.packed + ((flat0 - o) >> 1);
        const int b0 = o >> 1, b1 = more ? end >> 1 : (end + 1) >> 1;      // (a byte shared with the next rows is left to them)
        int from = (b0 + 3) & ~3, to = b1 & ~3;
        if ((reinterpret_cast<unsigned long long>(T.packed) & 3ull) != 0 || from > to) from = to = b1;
        auto byte_of = [&](int b) { return (unsigned char)((qs[2 * b] & 0xf) | ((qs[2 * b + 1] & 0xf) << 4)); };
        for (int b = b0 + lane; b < from; b += 32) dst[b] = byte_of(b);
        for (int b = from + 4 * lane; b < to; b += 128) {
            const uint2 u = *reinterpret_cast<const uint2*>(qs + 2 * b);
            auto nibbles = [](unsigned int v) { return (v & 0xfu) | ((v >> 4) & 0xf0u) | ((v >> 8) & 0xf00u) | ((v >> 12) & 0xf000u); };
            *reinterpret_cast<unsigned int*>(dst + b) = nibbles(u.x) | (nibbles(u.y) << 16);
        }
        if (to + lane < b1) dst[to + lane] = byte_of(to + lane);
        carry = qs[end - 1];
    }
}

template <int BY>
__global__ void __launch_bounds__(kShortThreads, BY == kByLanes ? 6 : kShortBlocks) rows_short_kernel(const RowArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ShortSmem sm;
    sm.xs = reinterpret_cast<float4*>(smem_raw + (size_t)warp * a.short_bytes);
    sm.stack = reinterpret_cast<float2*>(sm.xs + a.short_rows4);
    sm.close = reinterpret_cast<unsigned short*>(sm.stack + a.short_slots);
    sm.qs = reinterpret_cast<signed char*>(sm.xs) + a.short_codes;
    unsigned int st = 0;
    unsigned long long ev = 0ull;
    for (;;) {
        long long unit = 0;
        if (lane == 0) unit = (long long)atomicAdd(a.ticket, 1ull);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= a.n_units) break;
        const RowTensor& T = a.tensors ? a.tensors[tensor_of_unit(a, unit)] : a.one;
        if (T.gate && *T.gate == 0) continue;
        const int lg = BY == kBySplits ? T.lanes : 5, groups = 32 >> lg;
        const long long row0 = (unit - T.unit_begin) * T.rows_per_unit;
        const int nrows = (int)min((long long)T.rows_per_unit, T.S - row0);
        int carry = 0;
        for (int r = 0; r < nrows; r += groups) {
            const int now = min(groups, nrows - r);
            const bool more = r + groups < nrows;
            short_step<BY>(a, T, sm, lg, row0 + r, now, more, carry, st, ev);
        }
    }
    rows_done(a, st, ev);
}

}  // namespace omse
