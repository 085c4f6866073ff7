// Kernel-wise MMSE quantization (Sections 3.3, 3.4) and Algorithm 1 (Section 3.5): one thread block
// owns one kernel (row) at a time, staged once from HBM into shared memory; everything that follows
// (max, histogram and error curve, argmin, polish, codes, packing, residual update) reads the on-chip copy.
#pragma once
#include "omse_lattice.cuh"

namespace omse {

// One weight tensor of a launch (Section 3.1: W_l = {W_lk}, row k is kernel W_lk flattened).
struct RowTensor {
    const float* w;          // [S][K]
    long long S, K;
    float* alpha;            // [n_tensors][S]
    float* sse;              // [n_tensors][S]
    int* best_idx;           // [S] (single quantized tensor only), nullable
    signed char* codes;      // [n_tensors][N], nullable
    unsigned char* packed;   // [n_tensors][ceil(N/2)], nullable
    float* delta;            // [S] offset subtracted from each row (Section 3.1 scheme with offset), nullable = no offset
    const float* prior_alpha;   // [S] nullable: scale of an earlier quantized tensor of this row; the row is replaced by its
                                // residual fl(x - alpha*[x/alpha]_Zp) before the search (second tensor of a key layer, Section 3.5)
    const int* gate;         // nullable: the tensor's units are skipped when *gate == 0 (key-layer flag written by an earlier kernel)
    long long unit_begin;    // index of this tensor's first work unit in the launch-wide numbering
    int rows_per_unit;       // block per row: 2 when nibble packing needs an even element count per unit (odd K), else 1;
                             // short rows: what a warp takes, 32 >> lanes at a time (even)
    int lanes;               // short rows: lanes per row (log2)
    int hist_fbits, hist_cshift;    // short rows by a histogram of their warp: see HistShape
};

struct RowArgs {
    const RowTensor* tensors;   // device array, ordered by decreasing K (longest rows are handed out first)
    RowTensor one;              // the tensor itself when n_tensors_in_launch == 1 (tensors == nullptr)
    int n_launch_tensors;
    long long n_units;          // work units in the launch
    unsigned long long* ticket; // [2] next unit to hand out, blocks finished; both return to 0 at kernel end
    int n_cand;
    float hi_frac;
    int refine_iters;
    int n_tensors, n_sweeps;    // Algorithm 1: quantized tensors per row, sweeps
    int lo[4], hi[4];           // grid bounds per quantized tensor (Section 3.1)
    float* sse_history;         // [n_sweeps][n_tensors][S] error after every update of Algorithm 1, nullable (single tensor launches)
    unsigned int* status;
    unsigned long long* evals;  // executed (element, candidate) evaluations, summed over the launch (instrumentation), nullable
    int keep_x0;                // n_sweeps > 1: keep the original row next to the residual
    int max_k4;                 // float4s of the longest row in the launch (shared-memory carve-up)
    int n_bins;                 // bins of |x|/h (see LatticeShape)
    int window;                 // > 0: the bins are taken in windows of this many
    int direct;                 // >= 0: no histogram; lanes per candidate (log2) of lattice_coarse, or kSplitRows for lattice_split
    int packed_counts;          // 16 bits per count (see Counts)
    int smem_bins, smem_bins2;  // words of the bin arrays in shared memory (fine, coarse)
    int solver;                 // 0: grid line search (Section 3.4); 1: uniform scale max|x|/L; 2: alternating from the
                                // uniform scale; 3: golden-section search (the comparison solvers of Section 3.4)
    int solver_iters;           // alternating: least-squares steps; golden: shrink steps
    int n_delta;                // > 0: offsets searched per row (offset scheme of Section 3.1 with delta on a grid); needs keep_x0
    float off_frac;             // offsets span [min, min + off_frac*(max-min))
    float eps;                  // >= 0: Algorithm 1 stops after the first sweep whose relative error decrease is <= eps
    int* sweeps_done;           // [S] sweeps Algorithm 1 ran per row, nullable
    int short_direct;           // short rows: a candidate per lane
    int hist_lb;                // short rows by a histogram: log2 of the bins in a lane's run
    int short_rows4, short_slots, short_codes, short_bytes;   // short rows: shared memory of a warp (float4s of the rows, slots
                                // of the stacks, offset of the codes, size)
    int ext_tensors;            // a tensor of a batched launch has a gate or an earlier tensor's scale
};

// Index of the tensor that a work unit of a batched launch belongs to, found by the lanes of a warp together.
__device__ __forceinline__ int tensor_of_unit(const RowArgs& a, long long unit) {
    int n = 0;
    if (a.tensors)
        for (int t0 = 0; t0 < a.n_launch_tensors; t0 += 32) {
            const int t = t0 + (threadIdx.x & 31);
            n += __popc(__ballot_sync(0xffffffffu, t < a.n_launch_tensors && a.tensors[t].unit_begin <= unit));
        }
    return max(n - 1, 0);
}

// End of a row kernel: status bits and counters; the last block to leave re-arms the ticket pair (no block waits).
__device__ __forceinline__ void rows_done(const RowArgs& a, unsigned int st, unsigned long long ev) {
    if (st) atomicOr(a.status, st);   // any thread that saw a flag reports it
    report_evaluations(a.evals, ev);
    __syncthreads();                  // every warp of the block has taken its last ticket
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned long long done = atomicAdd(a.ticket + 1, 1ull);
        if (done == (unsigned long long)gridDim.x - 1ull) {
            a.ticket[0] = 0ull;
            a.ticket[1] = 0ull;
            __threadfence();
        }
    }
}

}  // namespace omse

#include "omse_rows_short.cuh"

namespace omse {

constexpr int kScratchDoubles = 64;
constexpr int kSplitRows = 31;                   // RowArgs::direct
constexpr int kRowsThreads = 32 * kTeamWarps;    // sets the register budget; blocks have up to 512 threads

struct PhiOut {
    float alpha;
    double sse;       // with PhiCtl::want_sse: squared error at the chosen grid candidate (true division, fp64)
    int idx;
    bool degenerate;
    bool bad;         // a value of the row is not finite
};

// What phi_block does on the row in s.xs besides the default "grid search, then refine_iters polish steps".
struct PhiCtl {
    int solver;       // as RowArgs::solver
    int n_iter;       // as RowArgs::solver_iters
    int start_idx;    // >= 0: skip the search and start from this grid candidate
    int n_refine;     // polish steps
    bool want_sse;    // also return the fp64 error at the chosen candidate (before any polish)
};

// Per-row state of the pass loop of rows_kernel (shared memory; thread 0 writes between barriers).
struct RowMode {
    PhiCtl ctl;             // what the next phi_block call does
    double aff_best;        // offset search: smallest error so far, its offset index and scale index
    int aff_d, aff_c;
    float aff_lo, aff_dstep, aff_dl;   // row minimum, offset step, offset of the current pass
    double e_prev;          // Algorithm 1: error after the previous sweep
    int sweeps_ran;
};

// ||x - alpha*[x/alpha]_Zp||^2 of the row in s.xs in fp64 with true division; every thread gets the sum.
__device__ __forceinline__ double exact_sse_block(const float* xs, int k, float alpha, float flo, float fhi,
                                                   double* scratch) {
    double ss = 0.0;
    long long zero = 0;
    const Coder coder(alpha, __fdiv_rn(1.0f, alpha), flo, fhi);
    const double ad = (double)alpha;
    // four elements per step (the row is zero padded to a multiple of four; a zero has code 0 and error 0)
    const float4* xs4 = reinterpret_cast<const float4*>(xs);
    const int k4 = (k + 3) >> 2;
#pragma unroll 1
    for (int i4 = threadIdx.x; i4 < k4; i4 += blockDim.x) {
        const float4 v = xs4[i4];
        const float x[4] = {v.x, v.y, v.z, v.w};
        float t[4];
        coder.of(v, t);
        double d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = fma(-ad, magic_double(t[e]), (double)x[e]);
#pragma unroll
        for (int e = 0; e < 4; ++e) ss = fma(d[e], d[e], ss);
    }
    block_sum2(ss, zero, scratch);
    return ss;
}

// Least-squares polish of Section 3.4's objective: alpha <- <x,q>/<q,q>, q = [x/alpha]_Zp, at most n times.
__device__ __forceinline__ float polish_block(const float* xs, int k, float alpha, float flo, float fhi, int n,
                                              double* scratch) {
    const float4* xs4 = reinterpret_cast<const float4*>(xs);
    const int k4 = (k + 3) >> 2;
    for (int it = 0; it < n; ++it) {
        double sxq = 0.0;
        u64 qa = 0ull, qb = 0ull;
        const Coder coder(alpha, __fdiv_rn(1.0f, alpha), flo, fhi);
#pragma unroll 1
        for (int i4 = threadIdx.x; i4 < k4; i4 += blockDim.x) {   // four elements per step, kSquareSteps steps at most (see block_threads);
            const float4 v = xs4[i4];                             // the zero padding adds nothing
            const float x[4] = {v.x, v.y, v.z, v.w};
            float t[4];
            coder.of(v, t);
            qa = add_squares(t[0], t[1], qa);
            qb = add_squares(t[2], t[3], qb);
#pragma unroll
            for (int e = 0; e < 4; ++e) sxq = fma((double)x[e], magic_double(t[e]), sxq);
        }
        long long sqq = squares_of(qa, qb);
        block_sum2(sxq, sqq, scratch);
        if (sqq == 0) break;
        const float a_new = (float)(sxq / (double)sqq);
        if (!(a_new >= FLT_MIN) || !(a_new <= FLT_MAX)) break;
        if (a_new == alpha) break;   // fixed point: further steps would repeat it exactly
        alpha = a_new;
    }
    return alpha;
}

// shared-memory carve-up for one block
struct RowSmem {
    float* xs;        // [k4*4] current tensor (row or residual), zero padded to a multiple of 4
    float* x0;        // [k4*4] original row (only when keep_x0)
    LatticeSmem lat;  // histograms and error curve
    double* scratch;  // [kScratchDoubles] reductions
    TeamScratch* ts;
    SplitPoint* stack; // [kSplitSlots] lattice_split
    int* misc;        // [8]: 1..4 nibble carried to the next row, per tensor
};

// max|x| over the finite values of the row (amax: the maximum over all bit patterns, known to every thread).
__device__ __forceinline__ float finite_max_block(const float* xs, int k4, TeamScratch* ts, unsigned int amax) {
    if (amax >= 0x7f800000u) {
        amax = 0u;
        for (int i = threadIdx.x; i < 4 * k4; i += blockDim.x) {
            const unsigned int b = __float_as_uint(xs[i]) & 0x7fffffffu;
            if (b < 0x7f800000u) amax = max(amax, b);
        }
        __syncthreads();
        const BlockTeam team = {(int)threadIdx.x, (int)blockDim.x};
        amax = team_umax(team, amax, ts);
    }
    return __uint_as_float(amax);
}

// The quantization mapping phi of Section 3.4 on the row held in s.xs (k elements, k4 float4s).
template <bool EXT, bool PACKED>
__device__ PhiOut phi_block(const RowArgs& a, const RowSmem& s, int k, int k4, int lo, int hi, unsigned long long& ev,
                             const PhiCtl& ctl) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    const float flo = (float)lo, fhi = (float)hi;
    const float4* xs4 = reinterpret_cast<const float4*>(s.xs);
    const BlockTeam team = {tid, nthr};
    PhiOut out;
    out.alpha = 0.f;
    out.sse = 0.0;
    out.idx = -1;
    out.degenerate = true;
    out.bad = false;

    // ---- max|x| as the largest bit pattern without the sign: values that are not finite come out on top
    unsigned int amax = 0u;
    for (int i4 = tid; i4 < k4; i4 += nthr) {   // the zero padding leaves the maximum alone
        const uint4 v = reinterpret_cast<const uint4*>(s.xs)[i4];
        amax = max(max(max(amax, v.x & 0x7fffffffu), max(v.y & 0x7fffffffu, v.z & 0x7fffffffu)), v.w & 0x7fffffffu);
    }
    if (EXT && (ctl.solver != 0 || ctl.start_idx >= 0)) {
        amax = team_umax(team, amax, s.ts);
        out.bad = amax >= 0x7f800000u;
        if (ctl.start_idx >= 0) {
            const Grid g = grid_of(__uint_as_float(amax), a.hi_frac, a.n_cand);
            const float ac = __fmul_rn((float)(ctl.start_idx + 1), g.step);
            if (amax >= 0x7f800000u || !g.usable || !usable_scale(ac) || ctl.start_idx >= a.n_cand) return out;
            out.degenerate = false;
            out.idx = ctl.start_idx;
            out.alpha = polish_block(s.xs, k, ac, flo, fhi, ctl.n_refine, s.scratch);
            return out;
        }
        // ---- comparison solvers of Section 3.4: another way to the starting scale, then the same polish
        const float m = finite_max_block(s.xs, k4, s.ts, amax);
        float alpha = 0.f;
        if (ctl.solver == 3) {
            // golden-section search on [0, hi_frac*max|x|], scales in binary32, errors in fp64 (uniform over the block)
            const float rho = 0.618034f;
            float lo_a = 0.f, hi_a = __fmul_rn(a.hi_frac, m);
            float t = __fmul_rn(rho, __fsub_rn(hi_a, lo_a));
            float x1 = __fsub_rn(hi_a, t), x2 = __fadd_rn(lo_a, t);
            auto f = [&](float al) -> double {
                return (al >= FLT_MIN && al <= FLT_MAX) ? exact_sse_block(s.xs, k, al, flo, fhi, s.scratch) : (double)INFINITY;
            };
            double f1 = f(x1), f2 = f(x2);
            for (int it = 0; it < ctl.n_iter; ++it) {
                if (f1 <= f2) {          // equal errors keep the smaller scale
                    hi_a = x2;
                    x2 = x1;
                    f2 = f1;
                    t = __fmul_rn(rho, __fsub_rn(hi_a, lo_a));
                    x1 = __fsub_rn(hi_a, t);
                    f1 = f(x1);
                } else {
                    lo_a = x1;
                    x1 = x2;
                    f1 = f2;
                    t = __fmul_rn(rho, __fsub_rn(hi_a, lo_a));
                    x2 = __fadd_rn(lo_a, t);
                    f2 = f(x2);
                }
            }
            alpha = (f1 <= f2) ? x1 : x2;
            if (!(fmin(f1, f2) < (double)INFINITY)) alpha = 0.f;
        } else {
            // no-offset uniform quantizer of Section 3.1: alpha = max|x| / L
            alpha = __fdiv_rn(m, fhi);   // L = 2^(p-1)-1 (signed) or 2^p-1 (unsigned) is the top code of the range
        }
        if (!(alpha >= FLT_MIN) || !(alpha <= FLT_MAX)) return out;
        out.degenerate = false;
        out.idx = 0;
        const int steps = ctl.n_refine + (ctl.solver == 2 ? ctl.n_iter : 0);
        out.alpha = polish_block(s.xs, k, alpha, flo, fhi, steps, s.scratch);
        return out;
    }

    // ---- the error curve; every candidate within its noise band of the minimum is re-scored in fp64 with exact codes
    const LatticeShape shape = {a.n_cand, a.n_bins, a.hi_frac, lo, hi, a.window, a.direct};
    const LatticeResult r = EXT && a.direct == kSplitRows ? lattice_split(team, shape, s.lat.curve, s.stack, xs4, k4, amax, s.ts)
                            : EXT && a.direct >= 0        ? lattice_coarse(team, shape, s.lat.curve, xs4, k4, amax, s.ts)
                            : EXT && a.window > 0         ? lattice_search_wide(team, shape, s.lat, xs4, k, k4, amax, s.ts)
                                                          : lattice_search<PACKED>(team, shape, s.lat, xs4, k, k4, amax, s.ts);
    out.bad = r.bad;
    if (r.degenerate) return out;
    out.degenerate = false;
    if (tid == 0) ev += (unsigned long long)k * (unsigned long long)r.evaluated;
    int best = r.best;
    double best_sse = INFINITY;
    bool other = false;                                     // a candidate beside the minimum lies in the band
    lattice_each(team, r, a.n_cand, [&](int c) { other |= c != r.best && s.lat.curve[c] <= r.band; });
    if (__syncthreads_or(other)) {
        // every warp finds the same candidates in the same (increasing) order
        best = 0x7fffffff;
        for (int c0 = 0; c0 < a.n_cand; c0 += 32) {
            const int cl = c0 + (tid & 31);
            unsigned int mask = __ballot_sync(0xffffffffu, lattice_evaluated(r, cl, a.n_cand) && s.lat.curve[cl] <= r.band);
            while (mask) {
                const int c = c0 + __ffs(mask) - 1;
                mask &= mask - 1;
                const double ss = exact_sse_block(s.xs, k, __fmul_rn((float)(c + 1), r.step), flo, fhi, s.scratch);
                if (tid == 0) ev += (unsigned long long)k;
                if (ss < best_sse) {                        // increasing index: strict < keeps the lowest among equal errors
                    best_sse = ss;
                    best = c;
                }
            }
        }
        if (best == 0x7fffffff) best = r.best;
    }

    // ---- polish: alpha <- <x,q>/<q,q>, q = [x/alpha]_Zp
    const float a_grid = __fmul_rn((float)(best + 1), r.step);
    if (EXT && ctl.want_sse)
        out.sse = best_sse < INFINITY ? best_sse : exact_sse_block(s.xs, k, a_grid, flo, fhi, s.scratch);
    out.alpha = polish_block(s.xs, k, a_grid, flo, fhi, EXT ? ctl.n_refine : a.refine_iters, s.scratch);
    out.idx = best;
    return out;
}

// Final codes at `alpha`, their squared error, and emission as int8 and/or nibbles.
// row_base = flat index of the row's first element in the tensor; n_total = S*K.
__device__ double emit_block(const RowSmem& s, int k, float alpha, float flo, float fhi,
                             signed char* codes, unsigned char* packed, long long row_base,
                             int* carry, bool more_rows_in_unit) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    double ss = 0.0;
    const bool zero = !(alpha > 0.f);
    const float inv = zero ? 0.f : __fdiv_rn(1.0f, alpha), thr = ambiguity_threshold(flo, fhi);
    const Coder coder(alpha, inv, flo, fhi);
    const double ad = (double)alpha;
    const bool aligned = ((reinterpret_cast<unsigned long long>(codes) & 3ull) == 0) &&
                         ((reinterpret_cast<unsigned long long>(packed) & 1ull) == 0);
    if ((k & 3) == 0 && aligned) {
        // aligned fast path: four codes per thread, 32-bit and 16-bit stores
        const float4* xs4 = reinterpret_cast<const float4*>(s.xs);
#pragma unroll 1
        for (int i4 = tid; i4 < (k >> 2); i4 += nthr) {
            const float4 v = xs4[i4];
            const float x[4] = {v.x, v.y, v.z, v.w};
            float t[4] = {kMagic, kMagic, kMagic, kMagic};
            if (!zero) coder.of(v, t);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double d = fma(-ad, magic_double(t[e]), (double)x[e]);
                ss = fma(d, d, ss);
            }
            const unsigned int w = code_bytes(t);
            if (codes) *reinterpret_cast<unsigned int*>(codes + row_base + 4ll * i4) = w;
            if (packed) *reinterpret_cast<unsigned short*>(packed + ((row_base + 4ll * i4) >> 1)) = (unsigned short)byte_nibbles(w);
        }
    } else if (!packed) {
        // codes alone at any offset: a byte per element, four independent ones per step
        for (int i = tid; i < k; i += 4 * nthr) {
            float x[4], t[4] = {kMagic, kMagic, kMagic, kMagic};
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = i + e * nthr < k ? s.xs[i + e * nthr] : 0.f;      // a zero has code 0 and error 0
            if (!zero) coder.of(make_float4(x[0], x[1], x[2], x[3]), t);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double d = fma(-ad, magic_double(t[e]), (double)x[e]);
                ss = fma(d, d, ss);
                if (codes && i + e * nthr < k) codes[row_base + i + e * nthr] = (signed char)magic_int(t[e]);
            }
        }
    } else {
        // general path: one output byte (two flat-consecutive elements) per thread; a byte that
        // straddles two rows is completed by the second row of the unit from the saved nibble
        const int o = (int)(row_base & 1);
        const int n_pairs = (k + o + 1) >> 1;
        for (int p = tid; p < n_pairs; p += nthr) {
            const int e0 = 2 * p - o, e1 = e0 + 1;
            int q0 = 0, q1 = 0;
            if (e0 >= 0) {
                const float x = s.xs[e0];
                q0 = zero ? 0 : exact_code(x, alpha, inv, flo, fhi, thr);
                const double d = fma(-ad, int_double(q0), (double)x);
                ss = fma(d, d, ss);
                if (codes) codes[row_base + e0] = (signed char)q0;
            } else {
                q0 = *carry;
            }
            const bool has1 = e1 < k;
            if (has1) {
                const float x = s.xs[e1];
                q1 = zero ? 0 : exact_code(x, alpha, inv, flo, fhi, thr);
                const double d = fma(-ad, int_double(q1), (double)x);
                ss = fma(d, d, ss);
                if (codes) codes[row_base + e1] = (signed char)q1;
            }
            if (packed) {
                if (has1 || !more_rows_in_unit) {
                    packed[(row_base + e0) >> 1] = (unsigned char)((q0 & 0xf) | ((q1 & 0xf) << 4));
                } else {
                    *carry = q0;   // last element of the row: its byte is written by the next row
                }
            }
        }
    }
    long long zero64 = 0;
    block_sum2(ss, zero64, s.scratch);
    return ss;
}

// EXT = false: the grid search with polish (and Algorithm 1 with a fixed number of sweeps) and nothing else, so that
// the common launches keep their register allocation and code size; EXT = true adds the comparison solvers, the offset
// search, Algorithm 1's loop condition, gated layers, rows that start from an earlier tensor's residual the search without a
// histogram and the one by windows.  PACKED: counts of 16 bits (see Counts).
// 80 registers per thread: 24 warps per SM, in as many blocks as the rows leave shared memory for; the phases of a row are
// separated by barriers, and the blocks of an SM fill each other's gaps.  Against 128 registers (16 warps): 29,127 rows of
// 2304 values 811 -> 697 us, 14,563 of 4608 565 -> 488, 5592 of 12,000 700 -> 434, 2674 of 25,088 539 -> 443.
template <bool EXT, bool PACKED>
__global__ void __launch_bounds__(kRowsThreads) rows_kernel(const RowArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long s_unit;
    __shared__ int s_tensor;
    __shared__ RowMode s_mode;
    __shared__ TeamScratch s_team;
    const int tid = threadIdx.x, nthr = blockDim.x;
    RowSmem s;
    s.xs = reinterpret_cast<float*>(smem_raw);
    s.x0 = s.xs + (a.keep_x0 ? 4 * a.max_k4 : 0);
    const bool windows = EXT && a.window > 0;
    s.lat.f = reinterpret_cast<unsigned int*>(s.x0 + 4 * a.max_k4);
    s.lat.n = s.lat.f + a.smem_bins;
    s.lat.f2 = s.lat.n + (windows ? a.smem_bins : max(Counts<PACKED>::words(a.smem_bins), (a.n_cand + 3) & ~3));
    s.lat.n2 = s.lat.f2 + a.smem_bins2;
    s.lat.curve = reinterpret_cast<float*>(windows ? s.lat.f2 : s.lat.n);
    s.scratch = reinterpret_cast<double*>(windows ? s.lat.f2 + ((a.n_cand + 3) & ~3) : s.lat.n2 + a.smem_bins2);
    s.misc = reinterpret_cast<int*>(s.scratch + kScratchDoubles);
    s.ts = &s_team;
    s.stack = reinterpret_cast<SplitPoint*>(s.misc + 8);
    unsigned int st = 0;
    unsigned long long ev = 0ull;      // evaluations this thread executed

    for (;;) {
        __syncthreads();   // previous unit fully consumed (shared row, s_unit)
        if (tid < 32) {
            long long u = 0;
            if (tid == 0) u = (long long)atomicAdd(a.ticket, 1ull);
            u = __shfl_sync(0xffffffffu, u, 0);
            const int ti = tensor_of_unit(a, u);
            if (tid == 0) {
                s_unit = u;
                s_tensor = ti;
            }
        }
        __syncthreads();
        const long long unit = s_unit;
        if (unit >= a.n_units) break;
        const RowTensor& T = a.tensors ? a.tensors[s_tensor] : a.one;
        if (EXT && T.gate && *T.gate == 0) continue;   // not a key layer: nothing to do for this unit
        const int k = (int)T.K;
        const int k4 = (k + 3) >> 2;
        const long long n_total = T.S * T.K;
        const long long packed_stride = (n_total + 1) >> 1;
        const long long unit_local = unit - T.unit_begin;

        for (int ru = 0; ru < T.rows_per_unit; ++ru) {
            const long long row = unit_local * T.rows_per_unit + ru;
            if (row >= T.S) break;
            const bool more = (ru + 1 < T.rows_per_unit) && (row + 1 < T.S);
            const long long row_base = row * T.K;
            const float* src = T.w + row_base;
            if (ru > 0) __syncthreads();   // previous row of the unit fully consumed
            // ---- stage the row once from HBM, all of it on its way at once (128-bit copies when the row start allows it).
            // Loads through registers keep one or two in flight per thread, which a block that owns an SM alone cannot hide.
            // With the codes four at a time: 4096 rows of 25088 values in 8 bits 694 -> 548 us, the same in two residual
            // tensors 2144 -> 1711 (428 and 1408 with two blocks per SM); ragged lengths also without divisions: 1337 rows of
            // 25087 values 505 -> 300 us, 7281 of 4607 492 -> 300.
            if ((reinterpret_cast<unsigned long long>(src) & 15ull) == 0) {
                for (int i4 = tid; i4 < (k >> 2); i4 += nthr) cp_async16(s.xs + 4 * i4, src + 4 * i4);
                if (tid < (k & 3)) cp_async4(s.xs + (k & ~3) + tid, src + (k & ~3) + tid);
            } else {
                for (int i = tid; i < k; i += nthr) cp_async4(s.xs + i, src + i);
            }
            if (tid < 4 * k4 - k) s.xs[k + tid] = 0.f;
            cp_async_wait();
            if (EXT && T.prior_alpha) {
                // second quantized tensor of a key layer: the row becomes the residual of the first tensor
                __syncthreads();
                const float a1 = T.prior_alpha[row];
                const float flo0 = (float)a.lo[0], fhi0 = (float)a.hi[0];
                if (a1 > 0.f)
                    for (int i = tid; i < k; i += nthr) {
                        const float x = s.xs[i];
                        s.xs[i] = fmaf(-a1, (float)code_of(x, a1, flo0, fhi0), x);
                    }
            }
            if (T.delta && !(EXT && a.n_delta > 0)) {
                // quantization with offset: delta = min of the row, the shifted row fl(x - delta) is what gets searched
                __syncthreads();
                float lo = INFINITY;
                for (int i = tid; i < k; i += nthr) {
                    const float v = s.xs[i];
                    if (fabsf(v) <= FLT_MAX) lo = fminf(lo, v);
                }
                __shared__ float s_min[32];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                if ((tid & 31) == 0) s_min[tid >> 5] = lo;
                __syncthreads();
                float d = INFINITY;
                for (int w = 0; w < ((nthr + 31) >> 5); ++w) d = fminf(d, s_min[w]);
                if (!(d < INFINITY)) d = 0.f;
                for (int i = tid; i < k; i += nthr) s.xs[i] = s.xs[i] - d;
                if (tid == 0) T.delta[row] = d;
            }
            if (a.keep_x0) {
                __syncthreads();
                for (int i = tid; i < 4 * k4; i += nthr) s.x0[i] = s.xs[i];
            }
            __syncthreads();

            // ---- The row goes through phi one or more times; all modes share the one call below.
            //  * default / Algorithm 1 (Section 3.5): pass = (sweep, tensor j); the residual of the other tensors is
            //    quantized; one tensor and one sweep is plain phi.
            //  * offset searched as well (Section 3.1 scheme, a.n_delta > 0): passes 0..n_delta-1 run the line search
            //    on the row shifted by offset d and keep the pair with the smallest error (lowest offset, then lowest
            //    scale index, on equal errors); the last pass polishes and emits at that pair.
            // Everything that steers the passes lives in shared memory (s_mode), not in registers: the search inside
            // phi_block needs the whole register budget.
            const bool affine = EXT && a.n_delta > 0;
            if (affine) {
                float lo = INFINITY, hi = -INFINITY;   // extremes of the finite values of the row
                for (int i = tid; i < k; i += nthr) {
                    const float v = s.x0[i];
                    if (fabsf(v) <= FLT_MAX) {
                        lo = fminf(lo, v);
                        hi = fmaxf(hi, v);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                }
                __shared__ float s_ext[2][32];
                if ((tid & 31) == 0) {
                    s_ext[0][tid >> 5] = lo;
                    s_ext[1][tid >> 5] = hi;
                }
                __syncthreads();
                if (tid == 0) {
                    lo = INFINITY;
                    hi = -INFINITY;
                    for (int w = 0; w < ((nthr + 31) >> 5); ++w) {
                        lo = fminf(lo, s_ext[0][w]);
                        hi = fmaxf(hi, s_ext[1][w]);
                    }
                    if (!(lo <= hi)) lo = hi = 0.f;
                    s_mode.aff_lo = lo;
                    s_mode.aff_dstep = __fdiv_rn(__fmul_rn(a.off_frac, __fsub_rn(hi, lo)), (float)a.n_delta);
                    s_mode.aff_best = INFINITY;
                    s_mode.aff_d = -1;
                    s_mode.aff_c = -1;
                }
            }
            if (EXT && a.eps >= 0.f) {
                // Algorithm 1: error before the first sweep (all tensors zero) is ||T||^2
                double e0 = 0.0;
                long long zero = 0;
                for (int i = tid; i < k; i += nthr) e0 += (double)s.xs[i] * (double)s.xs[i];
                block_sum2(e0, zero, s.scratch);
                if (tid == 0) s_mode.e_prev = e0;
            }
            if (EXT && tid == 0) s_mode.sweeps_ran = 0;
            const int n_pass = affine ? a.n_delta + 1 : a.n_sweeps * a.n_tensors;
            for (int pass = 0; pass < n_pass; ++pass) {
                const int sweep = affine ? 0 : pass / a.n_tensors;
                const int j = affine ? 0 : pass - sweep * a.n_tensors;
                if (EXT) __syncthreads();   // every thread is done with the previous pass's control block
                if (EXT && tid == 0) {
                    PhiCtl c = {a.solver, a.solver_iters, -1, a.refine_iters, false};
                    if (affine) {
                        const bool last = pass == a.n_delta;
                        if (last) {
                            c.start_idx = s_mode.aff_d >= 0 ? s_mode.aff_c : a.n_cand;   // n_cand: no offset had a usable scale
                        } else {
                            c.n_refine = 0;
                            c.want_sse = true;
                        }
                        s_mode.aff_dl = __fadd_rn(s_mode.aff_lo, __fmul_rn((float)(last ? max(s_mode.aff_d, 0) : pass), s_mode.aff_dstep));
                    }
                    s_mode.ctl = c;
                }
                if (EXT) __syncthreads();   // the control block is complete before any thread reads it
                if (affine) {
                    const float dl = s_mode.aff_dl;
                    for (int i = tid; i < 4 * k4; i += nthr) s.xs[i] = i < k ? __fsub_rn(s.x0[i], dl) : 0.f;
                    __syncthreads();
                } else if (a.keep_x0 && pass > 0) {
                    // residual T - sum_{i != j} alpha_i q^i from the original row, increasing i
                    for (int i = tid; i < k; i += nthr) {
                        float v = s.x0[i];
                        for (int i2 = 0; i2 < a.n_tensors; ++i2) {
                            if (i2 == j || (sweep == 0 && i2 > j)) continue;
                            const float ai = T.alpha[(long long)i2 * T.S + row];
                            const float qi = (float)T.codes[(long long)i2 * n_total + row_base + i];
                            v = fmaf(-ai, qi, v);
                        }
                        s.xs[i] = v;
                    }
                    __syncthreads();
                }
                const float flo = (float)a.lo[j], fhi = (float)a.hi[j];
                PhiOut r = phi_block<EXT, PACKED>(a, s, k, k4, a.lo[j], a.hi[j], ev, s_mode.ctl);
                if (affine && pass < a.n_delta) {
                    if (r.bad) st |= 1u;
                    if (tid == 0 && !r.degenerate && r.sse < s_mode.aff_best) {   // increasing offset: strict < keeps the lowest flat index
                        s_mode.aff_best = r.sse;
                        s_mode.aff_d = pass;
                        s_mode.aff_c = r.idx;
                    }
                    continue;      // the barriers of the next pass order these writes before their readers
                }
                if (r.bad) st |= 1u;
                if (r.degenerate) st |= 2u;
                const double sse = emit_block(s, k, r.alpha, flo, fhi,
                                              T.codes ? T.codes + (long long)j * n_total : nullptr,
                                              T.packed ? T.packed + (long long)j * packed_stride : nullptr,
                                              row_base, &s.misc[1 + j], more);
                if (tid == 0) {
                    T.alpha[(long long)j * T.S + row] = r.alpha;
                    T.sse[(long long)j * T.S + row] = (float)sse;
                    if (a.sse_history) a.sse_history[((long long)sweep * a.n_tensors + j) * T.S + row] = (float)sse;
                    if (affine) {
                        if (T.delta) T.delta[row] = s_mode.aff_dl;
                        if (T.best_idx) T.best_idx[row] = r.degenerate ? -1 : s_mode.aff_d * a.n_cand + s_mode.aff_c;
                    } else if (T.best_idx && j == 0) {
                        T.best_idx[row] = r.idx;
                    }
                }
                if (!a.keep_x0 && j + 1 < a.n_tensors) {
                    // first sweep without a kept copy: the residual is updated in place
                    const Coder coder(r.alpha, r.alpha > 0.f ? __fdiv_rn(1.0f, r.alpha) : 0.f, flo, fhi);
                    float4* xw4 = reinterpret_cast<float4*>(s.xs);
                    if (r.alpha > 0.f)
                        for (int i4 = tid; i4 < k4; i4 += nthr) {        // the padding zeros stay
                            const float4 v = xw4[i4];
                            float t[4];
                            coder.of(v, t);
                            xw4[i4] = make_float4(fmaf(-r.alpha, t[0] - kMagic, v.x), fmaf(-r.alpha, t[1] - kMagic, v.y),
                                                  fmaf(-r.alpha, t[2] - kMagic, v.z), fmaf(-r.alpha, t[3] - kMagic, v.w));
                        }
                }
                bool stop = false;
                if (EXT && j == a.n_tensors - 1) {
                    if (tid == 0) s_mode.sweeps_ran = sweep + 1;
                    if (a.eps >= 0.f) {
                        // loop condition of Algorithm 1: go on while the sweep lowered the error by more than eps (relative);
                        // every thread holds the same sse, so the decision is uniform
                        const double e_prev = s_mode.e_prev;
                        stop = !((e_prev - sse) > (double)a.eps * e_prev);
                    }
                }
                __syncthreads();   // alpha / codes of tensor j visible to the block (global + shared); e_prev read by all
                if (EXT && j == a.n_tensors - 1 && a.eps >= 0.f && tid == 0) s_mode.e_prev = sse;
                if (stop) break;
            }
            const int sweeps_ran = EXT ? s_mode.sweeps_ran : a.n_sweeps;
            if (EXT && tid == 0 && !affine) {
                if (a.sweeps_done) a.sweeps_done[row] = sweeps_ran;
                if (a.sse_history)     // sweeps that did not run repeat the last error
                    for (int sweep = sweeps_ran; sweep < a.n_sweeps; ++sweep)
                        for (int j = 0; j < a.n_tensors; ++j)
                            a.sse_history[((long long)sweep * a.n_tensors + j) * T.S + row] = T.sse[(long long)j * T.S + row];
            }
        }
    }
    rows_done(a, st, ev);
}

}  // namespace omse
