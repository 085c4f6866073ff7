// Dual line search (Section 3.5, n = 2): a two-dimensional grid over (alpha1, alpha2); for every pair
// each element picks its first code t in Z_p1 by enumeration, the second code being the rounding of
// the rest:  min_t ( x - alpha1*t - alpha2*[ (x - alpha1*t)/alpha2 ]_Zp2 )^2.
//
// One thread block owns one kernel (row) in shared memory.  Pairs are spread over threads: a thread
// holds one alpha1 and DPT consecutive alpha2 in registers, so x - alpha1*t is formed once per t and
// shared by its alpha2's; elements are broadcast from shared memory.  The enumeration over t is
// restricted, exactly, to a window around round(x/alpha1).  A first code whose rest saturates the second
// code errs by more than alpha2/2, one whose rest does not by at most alpha2/2, and the latter all lie
// within (max|Z_p2| + 1/2)*alpha2/alpha1 of x/alpha1; when every rest saturates, the error grows with
// the distance from x/alpha1 up to the asymmetry of Z_p2, which can only move the winner to the other
// neighbour of x/alpha1.  So the codes within (max|Z_p2| + 1/2)*alpha2/alpha1 + 1/2 of round(x/alpha1),
// and at least the two neighbours, hold the minimum (codes beyond Z_p1 collapse onto its ends).
// Grid values are compared in fp32 (blocks of 64 elements folded into fp64); pairs within the fp32 noise band of the minimum
// are re-scored in the reference arithmetic.  dual_kernel does that, and the final codes, with the full enumeration,
// dual_bound_kernel below with the window, except for rows at the ends of binary32, where equal squares decide.
#pragma once
#include "omse_rows.cuh"

namespace omse {

constexpr int kDualDpt = 8;        // alpha2 candidates per thread
constexpr int kDualThreads = 128;
constexpr int kDualListCap = 256;  // near-minimal pairs listed at a time for re-scoring with the full enumeration

struct DualArgs {
    const float* t;          // [S][K]
    long long S, K;
    int n_cand1, n_cand2;
    float hi_frac1, hi_frac2;
    int lo1, hi1, lo2, hi2;
    float* alpha;            // [2][S]
    float* sse;              // [S]
    int* best_idx;           // [S] flat pair index c*n_cand2+d, nullable
    signed char* codes;      // [2][N], nullable
    unsigned char* packed;   // [2][ceil(N/2)], nullable
    unsigned long long* evals;   // executed (element, pair, first code) evaluations (instrumentation), nullable
    float* curve;            // workspace: [gridDim.x][n_cand1*n_cand2] fp32 grid values of the block's current row
    unsigned int* status;
    int rows_per_unit;       // 2 when nibble packing needs an even element count per unit (odd K)
};

// scales of pair (c, d) for a row with max|x| = m: the same binary32 expressions as the 1-D grid
__device__ __forceinline__ void dual_scales(float m, const DualArgs& a, int c, int d, float& a1, float& a2) {
    const float step1 = __fdiv_rn(__fmul_rn(a.hi_frac1, m), (float)a.n_cand1);
    a1 = __fmul_rn((float)(c + 1), step1);
    const float step2 = __fdiv_rn(__fmul_rn(a.hi_frac2, a1), (float)a.n_cand2);
    a2 = __fmul_rn((float)(d + 1), step2);
}

// Full enumeration for one element in the reference arithmetic: lowest t on equal fp32 errors.
__device__ __forceinline__ void dual_codes_of(float x, float a1, float a2, const DualArgs& a, int& t_out, int& q_out) {
    float best = INFINITY;
    int bt = a.lo1, bq = 0;
    for (int t = a.lo1; t <= a.hi1; ++t) {
        const float r = fmaf(-a1, (float)t, x);
        const int q = code_of(r, a2, (float)a.lo2, (float)a.hi2);
        const float e = fmaf(-a2, (float)q, r);
        const float ee = __fmul_rn(e, e);
        if (ee < best) {
            best = ee;
            bt = t;
            bq = q;
        }
    }
    t_out = bt;
    q_out = bq;
}

__global__ void __launch_bounds__(kDualThreads) dual_kernel(const DualArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* xs = reinterpret_cast<float*>(smem_raw);                  // [k]
    const int k = (int)a.K;
    double* scratch = reinterpret_cast<double*>(xs + ((k + 3) & ~3)); // [64]
    int* list = reinterpret_cast<int*>(scratch + 64);                // [kDualListCap]
    int* misc = list + kDualListCap;                                 // [4]: list count, carried codes
    const int tid = threadIdx.x, nthr = blockDim.x;
    const long long n_total = a.S * a.K;
    const long long packed_stride = (n_total + 1) >> 1;
    const long long n_units = (a.S + a.rows_per_unit - 1) / a.rows_per_unit;
    const int dgroups = (a.n_cand2 + kDualDpt - 1) / kDualDpt;
    const int n_slots = a.n_cand1 * dgroups;                         // thread slots: (c, group of DPT d's)
    const float flo2 = (float)a.lo2, fhi2 = (float)a.hi2;
    const float half_range2 = fmaxf(fhi2, -flo2) + 0.5f;
    const int n_levels = a.hi1 - a.lo1 + 1;
    unsigned int st = 0;
    unsigned long long ev = 0ull;

    for (long long unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
        for (int ru = 0; ru < a.rows_per_unit; ++ru) {
            const long long row = unit * a.rows_per_unit + ru;
            if (row >= a.S) break;
            const bool more = (ru + 1 < a.rows_per_unit) && (row + 1 < a.S);
            const long long row_base = row * a.K;
            __syncthreads();
            // ---- stage the row, maxima
            float mx = 0.f;
            bool bad = false;
            for (int i = tid; i < k; i += nthr) {
                const float v = __ldg(a.t + row_base + i);
                xs[i] = v;
                if (fabsf(v) <= FLT_MAX) mx = fmaxf(mx, fabsf(v));
                else bad = true;
            }
            if (bad) st |= 1u;
            float dummy = 0.f;
            block_max2(mx, dummy, scratch);
            const float m = mx;
            float a1_last, a2_last;
            dual_scales(m, a, a.n_cand1 - 1, a.n_cand2 - 1, a1_last, a2_last);
            bool degenerate = !(m > 0.f) || !(a2_last >= FLT_MIN);

            // ---- grid: every thread slot sweeps the row for its alpha1 and DPT alpha2's; values to the workspace
            const int n_pairs_grid = a.n_cand1 * a.n_cand2;
            float* curve = a.curve + (size_t)blockIdx.x * n_pairs_grid;
            if (!degenerate) {
                for (int slot = tid; slot < n_slots; slot += nthr) {
                    // consecutive threads take consecutive alpha1 of one group of alpha2's: the window of first codes
                    // depends on alpha2/alpha1 = (d+1)*hi_frac2/C2 only, so a warp's lanes run the same number of steps
                    const int dg = slot / a.n_cand1, c = slot - dg * a.n_cand1, d0 = dg * kDualDpt;
                    float a1, a2[kDualDpt], inv2[kDualDpt], acc[kDualDpt];
                    double dacc[kDualDpt];
                    bool ok[kDualDpt];
#pragma unroll
                    for (int j = 0; j < kDualDpt; ++j) {
                        dual_scales(m, a, c, min(d0 + j, a.n_cand2 - 1), a1, a2[j]);
                        ok[j] = (d0 + j < a.n_cand2) && a1 >= FLT_MIN && a2[j] >= FLT_MIN;
                        inv2[j] = ok[j] ? __fdiv_rn(1.0f, a2[j]) : 0.f;
                        acc[j] = 0.f;
                        dacc[j] = 0.0;
                    }
                    const float inv1 = a1 >= FLT_MIN ? __fdiv_rn(1.0f, a1) : 0.f;
                    // window of first codes that can win: |t - round(x/alpha1)| <= half_range2*alpha2/alpha1 + 1/2, at least 1
                    const float ratio = a2[kDualDpt - 1] * inv1;         // largest alpha2 of the group
                    const int w = max(1, (int)(half_range2 * fminf(ratio, 16.f) * 1.0001f + 0.501f));
                    const bool full = !(ratio <= 16.f) || 2 * w + 1 >= n_levels;
                    const int n_t = full ? n_levels : 2 * w + 1;
                    ev += (unsigned long long)k * (unsigned long long)n_t * kDualDpt;
                    const float clo2 = kMagic + flo2, chi2 = kMagic + fhi2, flo1 = (float)a.lo1, fhi1 = (float)a.hi1;
                    for (int i = 0; i < k; ++i) {
                        const float x = xs[i];
                        const float t0 = full ? flo1 : rintf(x * inv1) - (float)w;
                        // smallest |error| over the first codes: squaring is monotone, so the square of the smallest
                        // magnitude is the smallest squared error
                        float best[kDualDpt];
#pragma unroll
                        for (int j = 0; j < kDualDpt; ++j) best[j] = INFINITY;
                        // one first code per step: the thread's alpha2's give independent chains, and a window
                        // always holds an odd number of codes
                        float tcur = t0;
                        for (int s = 0; s < n_t; ++s) {
                            const float ta = fminf(fmaxf(tcur, flo1), fhi1);
                            tcur += 1.0f;
                            const float ra = fmaf(-a1, ta, x);
#pragma unroll
                            for (int j = 0; j < kDualDpt; ++j) {
                                float ua = fmaf(ra, inv2[j], kMagic);
                                ua = fminf(fmaxf(ua, clo2), chi2);
                                const float ea = fmaf(-a2[j], ua - kMagic, ra);
                                best[j] = fminf(best[j], fabsf(ea));
                            }
                        }
#pragma unroll
                        for (int j = 0; j < kDualDpt; ++j) acc[j] = fmaf(best[j], best[j], acc[j]);
                        if ((i & 63) == 63) {
#pragma unroll
                            for (int j = 0; j < kDualDpt; ++j) {
                                dacc[j] += (double)acc[j];
                                acc[j] = 0.f;
                            }
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kDualDpt; ++j)
                        if (d0 + j < a.n_cand2)
                            curve[c * a.n_cand2 + d0 + j] = ok[j] ? (float)(dacc[j] + (double)acc[j]) : INFINITY;
                }
            }
            __syncthreads();                            // the block's grid values are visible to the block
            double bv = INFINITY;
            int bi = 0x7fffffff;
            if (!degenerate) {
                for (int p = tid; p < n_pairs_grid; p += nthr) {
                    const float v = curve[p];
                    if (v < bv) {                       // ascending p within a thread: strict < keeps the lowest index
                        bv = v;
                        bi = p;
                    }
                }
            }
            if (tid == 0) misc[0] = 0;
            block_argmin(bv, bi, scratch);
            if (bi == 0x7fffffff || !(bv < INFINITY)) degenerate = true;

            float alpha1 = 0.f, alpha2 = 0.f;
            int best_pair = -1;
            if (!degenerate) {
                // ---- pairs within the fp32 noise band of the minimum: re-score with the full enumeration.
                // The fp32 value squares e = r - alpha2*q with r = fl(x - alpha1*t) ROUNDED to binary32; the
                // winning t leaves |r| <= (max|Z_p2| + 1/2)*alpha2, so r is off by at most 2^-25 of that and a
                // sum of k terms by at most 2*sqrt(k*SSE) * 2^-25 * (max|Z_p2| + 1/2) * alpha2 (Cauchy-Schwarz).
                float a1_top, a2_top;
                dual_scales(m, a, a.n_cand1 - 1, a.n_cand2 - 1, a1_top, a2_top);     // largest alpha2 on the grid
                const double noise = 2.0 * sqrt((double)k * bv) * 2.98e-8 * (double)half_range2 * (double)a2_top;
                const double band = bv * (1.0 + kRescoreBand) + 2.0 * noise;
                for (int p = tid; p < n_pairs_grid; p += nthr) {
                    if ((double)curve[p] <= band) {
                        const int pos = atomicAdd(&misc[0], 1);
                        if (pos < kDualListCap) list[pos] = p;
                    }
                }
                __syncthreads();
                const int n_list = misc[0];
                best_pair = bi;
                if (n_list > 1) {
                    double best_sse = INFINITY;
                    best_pair = 0x7fffffff;
                    auto rescore = [&](int p) {      // full enumeration in the reference arithmetic, fp64 sum
                        float a1, a2;
                        dual_scales(m, a, p / a.n_cand2, p % a.n_cand2, a1, a2);
                        double ss = 0.0;
                        long long zero = 0;
                        for (int i = tid; i < k; i += nthr) {
                            int t, q;
                            dual_codes_of(xs[i], a1, a2, a, t, q);
                            const double d = (double)xs[i] - (double)a1 * (double)t - (double)a2 * (double)q;
                            ss += d * d;
                        }
                        block_sum2(ss, zero, scratch);
                        if (ss < best_sse || (ss == best_sse && p < best_pair)) {
                            best_sse = ss;
                            best_pair = p;
                        }
                    };
                    if (n_list <= kDualListCap) {
                        for (int l = 0; l < n_list; ++l) rescore(list[l]);
                    } else {
                        // more pairs in the band than the list holds: the same re-scoring, one window of
                        // kDualListCap consecutive pairs at a time
                        for (int base = 0; base < n_pairs_grid; base += kDualListCap) {
                            __syncthreads();
                            if (tid == 0) misc[0] = 0;
                            __syncthreads();
                            const int stop = min(base + kDualListCap, n_pairs_grid);
                            for (int p = base + tid; p < stop; p += nthr)
                                if ((double)curve[p] <= band) list[atomicAdd(&misc[0], 1)] = p;
                            __syncthreads();
                            const int n_win = misc[0];
                            for (int l = 0; l < n_win; ++l) rescore(list[l]);
                        }
                    }
                }
                dual_scales(m, a, best_pair / a.n_cand2, best_pair % a.n_cand2, alpha1, alpha2);
            } else {
                st |= 2u;
            }

            // ---- final codes (full enumeration), squared error, emission: one output byte pair per thread
            double ss = 0.0;
            const int o = (int)(row_base & 1);
            const int n_pairs = (k + o + 1) >> 1;
            for (int p = tid; p < n_pairs; p += nthr) {
                const int e0 = 2 * p - o, e1 = e0 + 1;
                int t0c = 0, q0c = 0, t1c = 0, q1c = 0;
                if (e0 >= 0) {
                    const float x = xs[e0];
                    if (!degenerate) dual_codes_of(x, alpha1, alpha2, a, t0c, q0c);
                    const double d = (double)x - (double)alpha1 * (double)t0c - (double)alpha2 * (double)q0c;
                    ss += d * d;
                    if (a.codes) {
                        a.codes[row_base + e0] = (signed char)t0c;
                        a.codes[n_total + row_base + e0] = (signed char)q0c;
                    }
                } else {
                    t0c = misc[1];
                    q0c = misc[2];
                }
                const bool has1 = e1 < k;
                if (has1) {
                    const float x = xs[e1];
                    if (!degenerate) dual_codes_of(x, alpha1, alpha2, a, t1c, q1c);
                    const double d = (double)x - (double)alpha1 * (double)t1c - (double)alpha2 * (double)q1c;
                    ss += d * d;
                    if (a.codes) {
                        a.codes[row_base + e1] = (signed char)t1c;
                        a.codes[n_total + row_base + e1] = (signed char)q1c;
                    }
                }
                if (a.packed) {
                    if (has1 || !more) {
                        const long long b = (row_base + e0) >> 1;
                        a.packed[b] = (unsigned char)((t0c & 0xf) | ((t1c & 0xf) << 4));
                        a.packed[packed_stride + b] = (unsigned char)((q0c & 0xf) | ((q1c & 0xf) << 4));
                    } else {   // last element of the row: its byte is completed by the next row of the unit
                        misc[1] = t0c;
                        misc[2] = q0c;
                    }
                }
            }
            long long zero = 0;
            block_sum2(ss, zero, scratch);
            if (tid == 0) {
                a.alpha[row] = alpha1;
                a.alpha[a.S + row] = alpha2;
                a.sse[row] = (float)ss;
                if (a.best_idx) a.best_idx[row] = best_pair;
            }
        }
    }
    if (st) atomicOr(a.status, st);
    report_evaluations(a.evals, ev);
}

// -------------------------------------------------------------------------------------------------
// The same search from a histogram of the row.
//
// For a pair of scales an element's error is its squared distance to the nearest of the points alpha1*(t + rho*q),
// t in Z_p1, q in Z_p2, rho = alpha2/alpha1, whose order depends on rho only, that is on the index d of alpha2: they are
// sorted once per launch (dual_points_kernel).  With the points sorted outwards from 0, midpoints M_k and gaps g_k,
//     (distance)^2 = x^2 - 2*sum_k g_k*(|x| - M_k)_+      on either side of 0,
// so a pair's error is E - 2*sum_k g_k*R(M_k) with R(y) = sum_i (|x_i| - y)_+ of that side.  R is known exactly at the bin
// edges of a histogram that keeps the number and the sum of the values of each bin; inside a bin with n values it lies
// within n*width*f*(1-f) below the chord, f being the position in the bin.  That gives an estimate of every pair's error and
// a bound of its distance from the truth: pairs whose lower bound is above the smallest upper bound are out.  One or two
// of 1024 pairs are left, and those are re-scored in the reference arithmetic if there is more than one.
// Bound: chains of look-ups, four points of a pair at a time, and in the re-scores and codes instruction issue.  The sweep above takes
// K*(first codes)/4 warp instructions a pair, this whatever the row's length: it is for rows of at least OMSE_DUAL_BOUND_K values,
// sorted point sets of at most kDualPoints and rho <= 1.  512 rows of 4608 values, 4 bits twice, 32 x 32 pairs on one B200: 3.62 ms ->
// 164 us (191 with 16-byte points and bins in binary64, every lane's end tested, five first codes per value), 16 such rows 1636 -> 70
// us, 16 rows of 300 values 57 -> 49.
// -------------------------------------------------------------------------------------------------
constexpr int kDualPoints = 256;
constexpr int kDualSide = 264;         // entries of a side: at most 255 midpoints, then ends (four are read ahead)
constexpr int kDualBins = 1024;        // per side; every value lies below bin kDualBins - 1
constexpr int kDualBoundThreads = 256;

struct DualPoint {                     // one midpoint and its gap, in units of alpha1
    float mid, gap;
};
struct DualPoints {
    const DualPoint* p;                // [n_cand2][2][kDualSide], outwards from 0: positive side, then negative side
};
struct __align__(16) DualBin {
    union {
        struct { unsigned int n, f, pad0, pad1; } h;     // while inserting: values, sum of their fractional parts
        struct { float r, dr, half, pad; } v;            // R at the lower edge, its fall over the bin, half of n
    };
};

__global__ void __launch_bounds__(kDualPoints) dual_points_kernel(DualPoint* out, int n_cand2, float hi_frac2, int lo1, int hi1, int lo2, int hi2) {
    __shared__ double pts[kDualPoints], sorted[kDualPoints];
    const int i = threadIdx.x, d = blockIdx.x, l2 = hi2 - lo2 + 1, n = (hi1 - lo1 + 1) * l2;
    const double rho = (double)(d + 1) * (double)hi_frac2 / (double)n_cand2;
    const double p = (double)(lo1 + i / l2) + rho * (double)(lo2 + i % l2);
    if (i < n) pts[i] = p;
    __syncthreads();
    if (i < n) {
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += pts[j] < p || (pts[j] == p && j < i);
        sorted[rank] = p;
    }
    const int below = __syncthreads_count(i < n && p < 0.0);          // the first zero: t = q = 0 is always a point
    DualPoint* side[2] = {out + (size_t)2 * d * kDualSide, out + (size_t)(2 * d + 1) * kDualSide};
    if (i + 1 < n) {
        const bool neg = i < below;
        const DualPoint e = {(float)(0.5 * (sorted[i] + sorted[i + 1]) * (neg ? -1.0 : 1.0)), (float)(sorted[i + 1] - sorted[i])};
        side[neg][neg ? below - 1 - i : i - below] = e;
    }
    for (int k = n - 1 - below + i; k < kDualSide; k += kDualPoints) side[0][k] = DualPoint{1e9f, 0.f};       // beyond every value
    for (int k = below + i; k < kDualSide; k += kDualPoints) side[1][k] = DualPoint{1e9f, 0.f};
}

// The reference's codes of one element: the first codes that can win (see the window of dual_kernel), lowest first code on
// equal binary32 errors, codes equal to those of the IEEE division.
// Two first codes at a time in packed arithmetic.  Where some first code leaves a rest that does not saturate the second one, only
// those can win (the others err by more than alpha2/2): their range is narrower than the window, 3 codes instead of 5 at alpha2 =
// 0.19*alpha1 on 4 bits twice.
struct DualCodes {
    float a1, a2, inv1, inv2, w, flo1, fhi1, flo2, fhi2, thr, up, down;
    bool every;
    __device__ __forceinline__ void set(float a1_, float a2_, const DualArgs& a, bool every_) {
        a1 = a1_;
        a2 = a2_;
        every = every_;
        inv1 = a1 > 0.f ? __fdiv_rn(1.0f, a1) : 0.f;
        inv2 = a2 > 0.f ? __fdiv_rn(1.0f, a2) : 0.f;
        flo1 = (float)a.lo1;
        fhi1 = (float)a.hi1;
        flo2 = (float)a.lo2;
        fhi2 = (float)a.hi2;
        thr = ambiguity_threshold(flo2, fhi2);
        const float ratio = fminf(a2 * inv1, 16.f);
        w = (float)max(1, (int)((fmaxf(fhi2, -flo2) + 0.5f) * ratio * 1.0001f + 0.501f));
        up = (0.5f - flo2) * ratio + 1e-3f;                  // rests from (lo2 - 1/2)*alpha2 to (hi2 + 1/2)*alpha2, and a margin that
        down = (fhi2 + 0.5f) * ratio + 1e-3f;                // binary32 does not reach
    }
    // codes as M + code
    __device__ __forceinline__ void of(float x, float& t_out, float& q_out) const {
        const float c = x * inv1, near = rintf(c);
        float t0 = fmaxf(ceilf(c - down), flo1), t1 = fminf(floorf(c + up), fhi1);
        // (none, or none for sure: all rests may saturate)
        if (!(fmaxf(ceilf(c - down + 2e-3f), flo1) <= fminf(floorf(c + up - 2e-3f), fhi1)) || !(fabsf(c) < 4096.f)) {
            t0 = fminf(fmaxf(near - w, flo1), fhi1);
            t1 = fminf(fmaxf(near + w, flo1), fhi1);
        }
        if (every) {
            t0 = flo1;
            t1 = fhi1;
        }
        float best = INFINITY, bt = flo1, bq = kMagic;
        const u64 na1 = pack2(-a1, -a1), na2 = pack2(-a2, -a2), i2 = pack2(inv2, inv2), M2 = pack2(kMagic, kMagic), NM2 = pack2(-kMagic, -kMagic),
                  minus = pack2(-1.f, -1.f), x2 = pack2(x, x), z2 = pack2(-0.f, -0.f);
        const float clo = kMagic + flo2, chi = kMagic + fhi2;
        for (float t = t0; t <= t1; t += 2.0f) {
            const u64 r = fma2(na1, pack2(t, t + 1.0f), x2), u = fma2(r, i2, M2);
            float d0, d1, q0, q1, e0, e1;
            unpack2(fma2(r, i2, fma2(u, minus, M2)), d0, d1);
            unpack2(u, q0, q1);
            q0 = fminf(fmaxf(q0, clo), chi);
            q1 = fminf(fmaxf(q1, clo), chi);
            if (!(max3_nan(fabsf(d0), fabsf(d1), 0.f) <= thr)) {
                float r0, r1;
                unpack2(r, r0, r1);
                if (!(fabsf(d0) <= thr)) q0 = kMagic + (float)code_of(r0, a2, flo2, fhi2);
                if (!(fabsf(d1) <= thr)) q1 = kMagic + (float)code_of(r1, a2, flo2, fhi2);
            }
            const u64 e = fma2(na2, add2(pack2(q0, q1), NM2), r);
            unpack2(fma2(e, e, z2), e0, e1);
            if (e0 < best) {
                best = e0;
                bt = t;
                bq = q0;
            }
            if (e1 < best && t + 1.0f <= t1) {
                best = e1;
                bt = t + 1.0f;
                bq = q1;
            }
        }
        t_out = kMagic + bt;
        q_out = bq;
    }
};

// BLOCKS: blocks per SM that the registers are cut for.  Four hide more latency where there are rows for them (512 rows of
// 4608 values 164 us); with up to three rows per SM the wider schedule is faster (16 such rows 70 us).
template <int BLOCKS>
__global__ void __launch_bounds__(kDualBoundThreads, BLOCKS) dual_bound_kernel(const DualArgs a, const DualPoints pts) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DualBin* bins = reinterpret_cast<DualBin*>(smem_raw);            // [2][kDualBins]
    float* xs = reinterpret_cast<float*>(bins + 2 * kDualBins);      // [k]
    __shared__ double scratch[64];
    __shared__ double s_sums[2][kDualBoundThreads / 32];
    __shared__ unsigned int s_part[3][kDualBoundThreads / 32];
    __shared__ int s_list[kDualListCap], s_n;
    __shared__ float s_carry[2];
    const int tid = threadIdx.x, nthr = kDualBoundThreads, lane = tid & 31, warp = tid >> 5, nwarp = kDualBoundThreads / 32;
    const int k = (int)a.K;
    const long long n_total = a.S * a.K, packed_stride = (n_total + 1) >> 1, n_units = (a.S + a.rows_per_unit - 1) / a.rows_per_unit;
    const int n_pairs_grid = a.n_cand1 * a.n_cand2;
    float* curve = a.curve + (size_t)blockIdx.x * n_pairs_grid;      // lower bounds of the row's pairs
    unsigned int st = 0;
    unsigned long long ev = 0ull;
    DualCodes dc;

    for (long long unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
        for (int ru = 0; ru < a.rows_per_unit; ++ru) {
            const long long row = unit * a.rows_per_unit + ru;
            if (row >= a.S) break;
            const bool more = (ru + 1 < a.rows_per_unit) && (row + 1 < a.S);
            const long long row_base = row * a.K;
            __syncthreads();
            // ---- stage the row; maximum over the finite values, sums of x^2 and |x|; bins cleared
            float mx = 0.f, l1 = 0.f;
            double e = 0.0;
            bool bad = false;
            auto look = [&](float v) {
                if (fabsf(v) <= FLT_MAX) mx = fmaxf(mx, fabsf(v));
                else bad = true;
                e = fma((double)v, (double)v, e);
                l1 += fabsf(v);
            };
            const float* src = a.t + row_base;
            if ((k & 3) == 0 && (reinterpret_cast<unsigned long long>(src) & 15ull) == 0) {
                for (int i4 = tid; i4 < (k >> 2); i4 += nthr) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(src) + i4);
                    reinterpret_cast<float4*>(xs)[i4] = v;
                    look(v.x);
                    look(v.y);
                    look(v.z);
                    look(v.w);
                }
            } else {
                for (int i = tid; i < k; i += nthr) {
                    const float v = __ldg(src + i);
                    xs[i] = v;
                    look(v);
                }
            }
            for (int i = tid; i < 2 * kDualBins; i += nthr) reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
            if (bad) st |= 1u;
            const bool any_bad = __syncthreads_or(bad) != 0;
            block_max(mx, scratch);
            const float m = mx;
            float a1_last, a2_last;
            dual_scales(m, a, a.n_cand1 - 1, a.n_cand2 - 1, a1_last, a2_last);
            bool degenerate = any_bad || !(m > 0.f) || !(a2_last >= FLT_MIN);
            // The reference squares errors in binary32.  Below its range squares that round to the same number make it take the
            // lowest of their codes: a window of first codes may not hold it (`every`), and a value's error may be that much above
            // its smallest one (in the margin).  Above its range every square may be infinite: a pair has an upper bound only if
            // its whole error is finite.  What cannot be told apart by the bounds is left to the reference arithmetic.
            const bool every = !(m > 1e-14f && m < 1e18f);
            double bv = INFINITY, inv_es = 0.0;
            int bi = 0x7fffffff;
            if (!degenerate) {                                       // uniform over the block
                // ---- histogram: bin b of a side holds the values with |x|/w in [b, b+1); a power of two keeps 1/w finite
                const float pre = m < 1e-25f ? 18446744073709551616.0f : 1.0f;
                const float w = __fdiv_rn(__fmul_rn(m, pre), (float)(kDualBins - 2)), inv_dn = __fdiv_rn(1.0f, w) * (1.0f - 3.0e-7f);
                const int fbits = lattice_fbits(k);
                const float to_fix = __fdiv_rn((float)(1 << fbits), w);
                for (int i = tid; i < k; i += nthr) {
                    const float x = xs[i] * pre, ax = fabsf(x);
                    const float u = __fmaf_rd(ax, inv_dn, kMagic);
                    DualBin* b = bins + (x < 0.f ? kDualBins : 0) + magic_int(u);
                    atomicAdd(&b->h.n, 1u);
                    atomicAdd(&b->h.f, (unsigned)magic_int(fmaf(fmaf(-(u - kMagic), w, ax), to_fix, kMagic)));
                }
                l1 = warp_allsum(l1);
                e = warp_allsum(e);
                if (lane == 0) {
                    s_sums[0][warp] = e;
                    s_sums[1][warp] = (double)l1;
                }
                __syncthreads();
                // ---- R: suffix scan, half of the warps for each side
                constexpr int run = 2 * kDualBins / kDualBoundThreads;
                DualBin* mine = bins + tid * run;
                ScanPart p = {0u, 0u, 0u};
                unsigned int hn[run], hf[run];
#pragma unroll
                for (int i = run - 1; i >= 0; --i) {
                    hn[i] = mine[i].h.n;
                    hf[i] = mine[i].h.f;
                    p.s += p.n;
                    p.n += hn[i];
                    p.f += hf[i];
                }
                ScanPart q = p;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned int n2 = __shfl_down_sync(0xffffffffu, q.n, o), s2 = __shfl_down_sync(0xffffffffu, q.s, o),
                                       f2 = __shfl_down_sync(0xffffffffu, q.f, o);
                    if (lane + o < 32) {
                        q.s += s2 + (unsigned)(o * run) * n2;
                        q.n += n2;
                        q.f += f2;
                    }
                }
                ScanPart x = scan_exclusive(q);
                if (lane == 0) {
                    s_part[0][warp] = q.n;
                    s_part[1][warp] = q.s;
                    s_part[2][warp] = q.f;
                }
                __syncthreads();
                {
                    ScanPart acc = {0u, 0u, 0u};
                    for (int v = (warp | (nwarp / 2 - 1)); v > warp; --v) {      // the warps behind this one on its side
                        acc.s += s_part[1][v] + 32u * run * acc.n;
                        acc.n += s_part[0][v];
                        acc.f += s_part[2][v];
                    }
                    x.s += acc.s + (unsigned)((31 - lane) * run) * acc.n;
                    x.n += acc.n;
                    x.f += acc.f;
                }
                const double fq = __longlong_as_double((long long)(1023 - fbits) << 52);
                double above = fma((double)x.f, fq, (double)x.s);
#pragma unroll
                for (int i = run - 1; i >= 0; --i) {
                    x.s += x.n;
                    x.n += hn[i];
                    x.f += hf[i];
                    const double r = fma((double)x.f, fq, (double)x.s);
                    mine[i].v.r = (float)r;
                    mine[i].v.dr = (float)(r - above);
                    mine[i].v.half = 0.5f * (float)hn[i];
                    above = r;
                }
                double es = 0.0, ls = 0.0;
#pragma unroll
                for (int v = 0; v < nwarp; ++v) {
                    es += s_sums[0][v];
                    ls += s_sums[1][v];
                }
                __syncthreads();
                // ---- estimate and bounds of every pair.  The margin holds what the fixed point (ls) and binary32 can add, u = 2^-24 each.
                //      Four roundings of a midpoint's position (mid, 1/w, s, f) move its term by 4u of 2*gap*mid per value beyond it, which
                //      sums to the squares of the values' nearest points, at most 1.05*es + 21 errors.  Three of R at the bin's lower edge
                //      and of its fall from there: with r - R at most a bin per value, in all 0.34*es (28,672 values), 2.02u of es.
                //      Five of the term itself, two of `unit`: 7u of unit*acc <= es.  Together 13.3u = 8e-7 of es, and 5e-6 of the error,
                //      which with what goes with the width is inside the factors of those in `off`.
                const float scale_pre = pre;
                const double w_true = (double)w / (double)scale_pre;
                const double margin0 = 1e-6 * es + ls * w_true * fq + 3e-45 * (double)k;
                inv_es = 1.0 / es;
                const float inv_w = __fdiv_rn(1.0f, w);
                // A warp takes 8 neighbouring alpha1 of 4 neighbouring ratios at a time: lanes of similar alpha1 have about as
                // many midpoints below max|x|, a lane keeps its own sums, and the points of a ratio are read by 8 lanes at once.
                // The warps go through all alpha1 of a few ratios before the next ones: L1 holds the points of that many.
                const int n_dq = (a.n_cand2 + 3) >> 2, n_cb = (a.n_cand1 + 7) >> 3, n_task = n_dq * n_cb;
                for (int task = warp; task < n_task; task += nwarp) {
                    // (small alpha1 have the most midpoints: which of them a warp takes changes from ratio to ratio)
                    const int dq = task / n_cb, cb = (task + dq * n_cb / nwarp) % n_cb, d = 4 * dq + (lane >> 3), c = 8 * cb + (lane & 7);
                    const bool valid = d < a.n_cand2 && c < a.n_cand1;
                    const int dv = min(d, a.n_cand2 - 1);
                    float a1, a2;
                    dual_scales(m, a, min(c, a.n_cand1 - 1), dv, a1, a2);
                    const bool ok = a1 >= FLT_MIN && a2 >= FLT_MIN;
                    const float s = (a1 * scale_pre) * inv_w;                // alpha1 in bins
                    double acc = 0.0;
                    float wid = 0.f;
#pragma unroll 1
                    for (int side = 0; side < 2; ++side) {
                        const float4* tab = reinterpret_cast<const float4*>(pts.p + (size_t)(2 * dv + side) * kDualSide);
                        const DualBin* bs = bins + side * kDualBins;
                        constexpr float kEnd = kMagic + (float)(kDualBins - 1);      // R is 0 there: midpoints beyond add nothing
                        float4 next[2] = {__ldg(tab), __ldg(tab + 1)};               // two points each; the next four are on their way
                        for (bool go = true; go;) {
                            const float mid[4] = {next[0].x, next[0].z, next[1].x, next[1].z}, gap[4] = {next[0].y, next[0].w, next[1].y, next[1].w};
                            tab += 2;
                            next[0] = __ldg(tab);
                            next[1] = __ldg(tab + 1);
                            float f[4], u[4], g[4];
                            float4 bin[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                u[j] = fminf(__fmaf_rd(mid[j], s, kMagic), kEnd);
                                f[j] = fminf(fmaf(mid[j], s, -(u[j] - kMagic)), 1.0f);      // (1 beyond the last bin: the square stays finite)
                                bin[j] = *reinterpret_cast<const float4*>(bs + magic_int(u[j]));
                            }
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float h = bin[j].z * fmaf(-f[j], f[j], f[j]);
                                g[j] = gap[j] * (bin[j].x - fmaf(f[j], bin[j].y, h));
                                wid = fmaf(gap[j], h, wid);
                            }
                            acc += (double)((g[0] + g[1]) + (g[2] + g[3]));
                            go = __any_sync(0xffffffffu, u[3] < kEnd);               // midpoints ascend
                        }
                    }
                    if (valid) {
                        const double unit = 2.0 * w_true * w_true * (double)s;
                        const double est = es - unit * acc;
                        const double off = unit * (double)wid * 1.00001 + margin0 + 1e-5 * fabs(est);
                        // (kept as a share of sum x^2, which may lie outside binary32)
                        curve[c * a.n_cand2 + d] = ok ? (float)((est - off) * inv_es * (1.0 - (est > off ? 1e-7 : -1e-7))) : INFINITY;
                        const double up = est + off < 3e38 ? est + off : 1e300;
                        if (ok && (up < bv || (up == bv && c * a.n_cand2 + d < bi))) {
                            bv = up;
                            bi = c * a.n_cand2 + d;
                        }
                    }
                }
                ev += (unsigned long long)k / (unsigned long long)nthr;
            }
            __syncthreads();                                        // the block's bounds are visible to the block
            if (tid == 0) s_n = 0;
            block_argmin(bv, bi, scratch);
            if (bi == 0x7fffffff) degenerate = true;

            float alpha1 = 0.f, alpha2 = 0.f;
            int best_pair = -1;
            if (!degenerate) {
                const float top = (float)fmin(bv * inv_es * (1.0 + 1e-7), (double)FLT_MAX);
                auto rescore_all = [&](int begin, int end) -> int {  // lists the survivors of [begin, end); returns their number
                    __syncthreads();
                    if (tid == 0) s_n = 0;
                    __syncthreads();
                    for (int p = begin + tid; p < end; p += nthr)
                        if (curve[p] <= top) {
                            const int pos = atomicAdd(&s_n, 1);
                            if (pos < kDualListCap) s_list[pos] = p;
                        }
                    __syncthreads();
                    return s_n;
                };
                double best_sse = INFINITY;
                best_pair = 0x7fffffff;
                auto rescore = [&](int p) {                          // the codes of the reference arithmetic, fp64 sum
                    float a1, a2;
                    dual_scales(m, a, p / a.n_cand2, p % a.n_cand2, a1, a2);
                    dc.set(a1, a2, a, every);
                    double ss = 0.0;
                    long long zero = 0;
                    for (int i = tid; i < k; i += nthr) {
                        float t, q;
                        const float v = xs[i];
                        dc.of(v, t, q);
                        const double dd = fma(-(double)a2, magic_double(q), fma(-(double)a1, magic_double(t), (double)v));
                        ss += dd * dd;
                    }
                    block_sum2(ss, zero, scratch);
                    if (tid == 0) ev += (unsigned long long)k;
                    if (ss < best_sse || (ss == best_sse && p < best_pair)) {
                        best_sse = ss;
                        best_pair = p;
                    }
                };
                const int n_list = rescore_all(0, n_pairs_grid);
                if (n_list <= 1) {
                    best_pair = bi;
                } else if (n_list <= kDualListCap) {
                    for (int l = 0; l < n_list; ++l) rescore(s_list[l]);
                } else {                                             // more than the list holds: a window of pairs at a time
                    for (int base = 0; base < n_pairs_grid; base += kDualListCap) {
                        const int n_win = rescore_all(base, min(base + kDualListCap, n_pairs_grid));
                        for (int l = 0; l < n_win; ++l) rescore(s_list[l]);
                    }
                }
                dual_scales(m, a, best_pair / a.n_cand2, best_pair % a.n_cand2, alpha1, alpha2);
            } else {
                st |= 2u;
            }

            // ---- final codes, squared error, emission: one output byte pair per thread
            dc.set(alpha1, alpha2, a, every);
            double ss = 0.0;
            const int o = (int)(row_base & 1);
            const int n_pairs = (k + o + 1) >> 1;
            for (int p = tid; p < n_pairs; p += nthr) {
                const int e0 = 2 * p - o, e1 = e0 + 1;
                float t0c = kMagic, q0c = kMagic, t1c = kMagic, q1c = kMagic;
                if (e0 >= 0) {
                    const float v = xs[e0];
                    if (!degenerate) dc.of(v, t0c, q0c);
                    const double dd = fma(-(double)alpha2, magic_double(q0c), fma(-(double)alpha1, magic_double(t0c), (double)v));
                    ss += dd * dd;
                    if (a.codes) {
                        a.codes[row_base + e0] = (signed char)magic_int(t0c);
                        a.codes[n_total + row_base + e0] = (signed char)magic_int(q0c);
                    }
                } else {
                    t0c = s_carry[0];
                    q0c = s_carry[1];
                }
                const bool has1 = e1 < k;
                if (has1) {
                    const float v = xs[e1];
                    if (!degenerate) dc.of(v, t1c, q1c);
                    const double dd = fma(-(double)alpha2, magic_double(q1c), fma(-(double)alpha1, magic_double(t1c), (double)v));
                    ss += dd * dd;
                    if (a.codes) {
                        a.codes[row_base + e1] = (signed char)magic_int(t1c);
                        a.codes[n_total + row_base + e1] = (signed char)magic_int(q1c);
                    }
                }
                if (a.packed) {
                    if (has1 || !more) {
                        const long long b = (row_base + e0) >> 1;
                        a.packed[b] = (unsigned char)((magic_int(t0c) & 0xf) | ((magic_int(t1c) & 0xf) << 4));
                        a.packed[packed_stride + b] = (unsigned char)((magic_int(q0c) & 0xf) | ((magic_int(q1c) & 0xf) << 4));
                    } else {   // last element of the row: its byte is completed by the next row of the unit
                        s_carry[0] = t0c;
                        s_carry[1] = q0c;
                    }
                }
            }
            long long zero = 0;
            block_sum2(ss, zero, scratch);
            if (tid == 0) {
                a.alpha[row] = alpha1;
                a.alpha[a.S + row] = alpha2;
                a.sse[row] = (float)ss;
                if (a.best_idx) a.best_idx[row] = best_pair;
            }
        }
    }
    if (st) atomicOr(a.status, st);
    report_evaluations(a.evals, ev);
}

}  // namespace omse
