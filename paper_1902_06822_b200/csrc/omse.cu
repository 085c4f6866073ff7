// Host side of the C interface declared in include/omse.h: argument checks, launch shapes, context.
// Every step of the method runs in the kernels of omse_rows*.cuh, omse_tensor.cuh and omse_dual.cuh; there is no
// host arithmetic on tensor data and no CPU fallback.
#include "../../include/omse.h"

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "omse_rows.cuh"
#include "omse_tensor.cuh"
#include "omse_dual.cuh"

namespace {

constexpr long long kSmallK = 1280;           // rows up to this length are searched in the registers of a warp or of some of its lanes
                                              // (58,254 rows of 1152 values on 3 bits 684 us against 1078 by blocks),
constexpr long long kJoinK = 1024;            // those beyond this length only in large numbers: see quantize_list
// Rows by a histogram of their warp, from 4 bits on (fewer leave too many candidates open).  Splits, or blocks beyond kJoinK, and
// histogram, 67M Laplace values (Student-t in brackets), 1024 candidates, on 4 bits: 400 values a row 1036 us and 1071 (976 and 1053), 512 888
// and 821 (832 and 795), 640 823 and 728 (776 and 705), 1024 838 and 642 (768 and 616), 1152 1100 and 628, 1600 890 and 639, 2304 705 and 580;
// on 8 bits: 700 1301 and 975 (1087 and 962), 1024 1007 and 781 (822 and 775), 1600 1013 and 704, 2304 786 and 565.  Beyond 2304 values
// the rows leave an SM fewer than twelve warps.
constexpr long long kHistK4 = 400, kHistK8 = 700, kHistMaxK = 2304;
constexpr long long kDualBoundK = 256;        // dual search: rows at least this long go by histogram and bounds (16 rows of 256 values 58 us
                                              // against 100 by the sweep, of 128 values 55 by the sweep, whose time is proportional to the length)
constexpr size_t kPartialBytes = 16u << 20;   // per-block partial sums of the per-tensor search
constexpr size_t kSmSmem = 233472;            // shared memory of an SM, and what a block of the row kernels takes beside the dynamic part:
constexpr size_t kBlockSmem = 1024 + 1232;    // 1 KB for the system, static
constexpr int kMaxSmem = 229376;              // dynamic shared memory per block: the 227 KB opt-in limit of sm_100 less 3 KB for static use

constexpr int kNearValues = 1 << 18;          // (51M values less their minimum, 2048 candidates: some 70,000 next to an edge of a bin)

constexpr int kSides = 2;          // side streams of a context

struct Workspace {
    unsigned int status;
    unsigned int pad_[3];
    unsigned long long ticket[2 + 2 * kSides];      // work-unit dispensers of the row kernels (self-resetting): a pair for launches on
                                    // the context's stream, a pair for each launch that runs beside them on a side stream
    unsigned long long evals;       // executed evaluations since the last omse_read_evaluations
    omse::TensorState tstate;
    double curve[OMSE_MAX_CANDIDATES];
    int list[OMSE_MAX_CANDIDATES];  // candidates of the per-tensor search that are re-scored in fp64
    float near[kNearValues];        // its values next to an edge of a bin
    omse::ResidentExchange exchange;
};

}  // namespace

// What the per-tensor search remembers between calls: launch shapes and attributes that cost more to ask for than a launch.
struct TensorLaunches {
    int occ_pass[3];                                        // blocks per SM of the three pass kernels (0 = not yet asked)
    struct { size_t smem; int occ; } hist[4];               // the histogram kernel's last launch shape, per variant
    bool attr_hist, attr_resident;
};

struct LaunchShape { int kernel, threads; size_t smem; int occ; };

struct omse_ctx {
    int device;
    cudaStream_t stream;
    cudaStream_t side[kSides];         // launches of a batched call run here, beside the last one (fork and join by events)
    cudaEvent_t ev_fork, ev_join[kSides];
    int ticket_pair;                   // which dispenser pair the next row launch uses
    int n_sm;
    Workspace* ws;       // device
    double* partials;    // device, kPartialBytes
    omse::RowTensor* d_tensors;   // device, OMSE_MAX_BATCH descriptors of a batched launch
    // per-context launch bookkeeping (a context is used by one host thread at a time, so no lock)
    bool attr_rows[6], attr_dual[3];   // opt-in shared-memory attribute set, per kernel
    LaunchShape seen[16];                           // blocks per SM of the launch shapes met so far
    int n_seen, next_seen;
    TensorLaunches tensor;                          // the same for the per-tensor kernels
    unsigned long long n_launches;                  // kernels launched since the last omse_read_launches
    unsigned int poll_limit;                        // polls of the one-kernel per-tensor search (omse_set_poll_limit)
    int search_blocks;                              // its blocks at most (omse_set_search_blocks)
};

namespace {

// Makes the context's device current for the duration of a call and puts the caller's device back afterwards.
class DeviceScope {
public:
    explicit DeviceScope(int device) : prev_(-1), ok_(false) {
        if (cudaGetDevice(&prev_) != cudaSuccess) prev_ = -1;
        ok_ = (prev_ == device) || cudaSetDevice(device) == cudaSuccess;
        if (prev_ == device) prev_ = -1;   // nothing to restore
    }
    ~DeviceScope() {
        if (prev_ >= 0) cudaSetDevice(prev_);
    }
    bool ok() const { return ok_; }
private:
    int prev_;
    bool ok_;
};

bool grid_ok(const omse_grid* g) {
    return g && g->n_cand >= 1 && g->n_cand <= OMSE_MAX_CANDIDATES && g->hi_frac > 0.f &&
           g->hi_frac <= 3.0e38f && g->refine_iters >= 0 && g->refine_iters <= 64;
}

void bounds(int bits, int is_signed, int* lo, int* hi) {
    if (is_signed) {
        *lo = -(1 << (bits - 1));
        *hi = (1 << (bits - 1)) - 1;
    } else {
        *lo = 0;
        *hi = (1 << bits) - 1;
    }
}

// Kernels of the row searches, by path (how rows are mapped to threads) and by what a launch needs.
enum RowPath { kPathShort, kPathHist, kPathBlock, kPaths };     // short rows: a warp or some of its lanes per row; a histogram per warp
static_assert(kPaths - 1 <= kSides, "a side stream for every path but the last");

// Blocks per SM of a launch shape, remembered: the query costs more than a small launch.  0: the query failed, or none fits.
int blocks_per_sm(omse_ctx* ctx, int id, const void* kernel, int threads, size_t smem) {
    for (int i = 0; i < ctx->n_seen; ++i)
        if (ctx->seen[i].kernel == id && ctx->seen[i].threads == threads && ctx->seen[i].smem == smem) return ctx->seen[i].occ;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess || occ < 1) return 0;
    ctx->seen[ctx->next_seen] = LaunchShape{id, threads, smem, occ};   // round robin once the table is full
    ctx->next_seen = (ctx->next_seen + 1) % 16;
    if (ctx->n_seen < 16) ++ctx->n_seen;
    return occ;
}
constexpr int kRowKernels = 6;       // ids of launch shapes: the row kernels, then the dual search's

int launch_rows_kernel(omse_ctx* ctx, const omse::RowArgs& a, int path, bool ext, int threads, size_t smem) {
    typedef void (*Kernel)(const omse::RowArgs);
    const Kernel kernels[kRowKernels] = {omse::rows_kernel<false, false>, omse::rows_kernel<true, false>, omse::rows_kernel<false, true>,
                                         omse::rows_short_kernel<omse::kBySplits>, omse::rows_short_kernel<omse::kByLanes>,
                                         omse::rows_short_kernel<omse::kByHistogram>};
    const int id = path == kPathHist ? 5 : path == kPathShort ? (a.short_direct ? 4 : 3) : ext ? 1 : a.packed_counts ? 2 : 0;
    const Kernel kernel = kernels[id];
    if (!ctx->attr_rows[id]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess) return OMSE_ECUDA;
        ctx->attr_rows[id] = true;
    }
    const int occ = blocks_per_sm(ctx, id, (const void*)kernel, threads, smem);
    if (occ == 0) return OMSE_ECUDA;
    long long grid = (long long)ctx->n_sm * occ;
    const long long teams = path != kPathBlock ? (a.n_units + threads / 32 - 1) / (threads / 32) : a.n_units;
    if (grid > teams) grid = teams;
    kernel<<<(unsigned)grid, threads, smem, ctx->stream>>>(a);
    ++ctx->n_launches;
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

// Bins of |x|/h that hold every value of a row: |x|/h <= 2*n_cand/hi_frac up to the rounding of step and h (0: too many
// to address in one piece).
int all_bins(int n_cand, float hi_frac) {
    const double v = 2.0 * (double)n_cand / (double)hi_frac * (1.0 + 1e-6);
    return v >= (double)(1 << 21) ? 0 : v < 1.0 ? 1 : (int)v;
}

// Words of the coarse histogram (the extra negative level of a signed range), over the launch's quantized tensors.
int coarse_words(const omse::RowArgs& a, int n_bins) {
    int words = 0;
    for (int j = 0; j < a.n_tensors; ++j) {
        const int bins = a.lo[j] < 0 ? n_bins / (-2 * a.lo[j] - 1) : 0;
        if (bins > 0) words = std::max(words, omse::lattice_padded(bins, 32));
    }
    return words;
}

// Shared memory of the block path beside the rows themselves.
size_t lattice_bytes(const omse::RowArgs& a, int threads, int n_bins, bool packed) {
    const int words = omse::lattice_padded(n_bins, threads), n = packed ? omse::Counts<true>::words(words) : words;
    return ((size_t)words + (size_t)std::max(n, (a.n_cand + 3) & ~3) + 2 * (size_t)coarse_words(a, n_bins)) * 4;
}

// Threads of a block for rows that leave room for `fit` blocks on an SM: the 24 warps that the registers allow, shared out.
// (At 5592 rows of 12,000 values, three blocks: 8 warps 456 us, 6 493, 12 537; at 3728 of 18,000, two blocks: 12 warps 482 us,
// 8 494, 16 629; at 2396 of 28,000, one block: 16 warps 563, 24 590, 12 609.)  No more than a thread per 8 values.
constexpr int kLeastWarps = 4, kOneWarpK = 160;      // ... and four warps at least; rows of up to kOneWarpK values may have one
static_assert((OMSE_MAX_KERNEL_LEN + 3) / 4 <= omse::kSquareSteps * 32 * kLeastWarps && (kOneWarpK + 3) / 4 <= omse::kSquareSteps * 32,
              "float4s of a row per thread");
int block_threads(int fit, long long max_k) {
    const int warps = std::min(16, std::max(kLeastWarps, 24 / fit));
    return 32 * (int)std::min<long long>(warps, std::max<long long>(kLeastWarps, (max_k / 8 + 31) / 32));
}

// Launch over rows of at most max_k elements on one path: threads per block and shared memory.
int launch_rows(omse_ctx* ctx, omse::RowArgs& a, long long max_k, int path) {
    const int k4 = (int)((max_k + 3) >> 2);
    a.max_k4 = k4;
    a.ticket = ctx->ws->ticket + 2 * ctx->ticket_pair;
    a.status = &ctx->ws->status;
    a.evals = &ctx->ws->evals;
    // the extended kernel only where a launch needs what it adds
    bool ext = a.solver != 0 || a.n_delta > 0 || a.eps >= 0.f || a.sweeps_done != nullptr;
    if (a.tensors == nullptr) ext = ext || a.one.gate || a.one.prior_alpha;
    else ext = ext || a.ext_tensors;
    const int bins = all_bins(a.n_cand, a.hi_frac);
    if (path != kPathBlock)
        return launch_rows_kernel(ctx, a, path, ext, omse::kShortThreads, (size_t)(omse::kShortThreads / 32) * a.short_bytes);
    const size_t fixed = (size_t)(a.keep_x0 ? 2 : 1) * k4 * 16 + omse::kScratchDoubles * 8 + 8 * 4;
    a.direct = -1;
    a.window = 0;
    int threads = 0;
    size_t smem = 0;
    // Rows that are shorter than this evaluate candidates instead of making a histogram.  In a small launch a row's chain of steps
    // counts, in a large one the barriers: 32 threads per row then.  (Two tensors of 4 bits, 1024 candidates, histogram and candidates:
    // 38,836 rows of 27 values 993 us and 326, 16,384 of 64 429 and 203, 10,485 of 100 283 and 161, 7133 of 147 205 and 163; 64
    // rows of 27 22.8 us and 18.5, of 64 22.7 and 18.5, of 100 22.6 and 19.0, of 147 with 200 candidates 20.5 and 21.3.)
    const bool many = a.n_units >= 8ll * ctx->n_sm;
    if (max_k <= (many ? kOneWarpK : 128)) {
        ext = true;
        a.direct = k4 >= 32 ? 2 : k4 >= 16 ? 1 : 0;
        smem = fixed + (size_t)((a.n_cand + 3) & ~3) * 4;
        threads = many ? 32 : max_k <= 36 ? 64 : 128;
    } else if (bins > 0 && (double)bins * (double)max_k < 2147483648.0) {
        // blocks of this launch that an SM holds, by shared memory and by the rows there are
        const long long per_sm = std::max(1ll, (a.n_units + ctx->n_sm - 1) / ctx->n_sm);
        auto fits = [&](bool packed) {
            return std::max(1ll, std::min(per_sm, (long long)(kSmSmem / (fixed + lattice_bytes(a, 128, bins, packed) + kBlockSmem))));
        };
        a.packed_counts = !ext && fits(false) == 1 && fits(true) > 1;
        threads = block_threads((int)fits(a.packed_counts), max_k);
        a.n_bins = bins;
        a.smem_bins = omse::lattice_padded(bins, threads);
        a.smem_bins2 = coarse_words(a, bins);
        smem = fixed + lattice_bytes(a, threads, bins, a.packed_counts);
    }
    if (smem == 0 || smem > (size_t)kMaxSmem) {
        // The bins do not fit at once: windows of them, up to the last threshold that any candidate has, where the row leaves room
        // for one block in any case and the windows are few; evaluations otherwise.  A window costs about what five evaluations do at
        // 25,088 values, of which a search takes 45 (4 bits) to 110 (8 bits).  4096 candidates, 4 and 8 bits, windows and
        // evaluations: 80 rows of 25,088, grid to a quarter of max|x| 165 us and 172, 178 and 296, to a tenth 297 and 192, 361 and 396,
        // to a hundredth 189 and 64, 3546 and 472; 434 rows of 4608 values 220 and 137, 264 and 231; 366 and 160, 488 and 327; 545
        // and 49, 7568 and 255.
        ext = true;
        a.packed_counts = 0;
        a.smem_bins = a.smem_bins2 = 0;
        int top = 1, sides = 1;
        for (int j = 0; j < a.n_tensors; ++j) {
            top = std::max(top, std::max(a.hi[j], -a.lo[j]));
            if (a.lo[j] < 0) sides = 2;
        }
        a.n_bins = std::max(1, (int)std::min(2.0 * (double)a.n_cand / (double)a.hi_frac * (1.0 + 1e-6), (double)(2 * top - 1) * (double)a.n_cand));
        threads = block_threads((int)std::max(1ll, (long long)(kSmSmem / (fixed + (size_t)a.n_cand * 4 + kBlockSmem))), max_k);
        const size_t curve = (size_t)((a.n_cand + 3) & ~3) * 4;
        for (a.window = 16384; a.window >= 4096; a.window >>= 1) {
            a.smem_bins = omse::lattice_padded(a.window, threads);
            smem = fixed + 2 * (size_t)a.smem_bins * 4 + curve;
            if (smem <= (size_t)kMaxSmem) break;
        }
        const int n_win = (a.n_bins + a.window - 1) / a.window;
        if (max_k < 12288 || a.window < 4096 || n_win * sides > (top < 64 ? 8 : 20)) {
            a.direct = omse::kSplitRows;
            a.window = a.smem_bins = 0;
            smem = fixed + curve + omse::kSplitSlots * sizeof(omse::SplitPoint);
        }
    }
    return launch_rows_kernel(ctx, a, path, ext, threads, smem);
}

void fill_tensor(omse::RowTensor& t, const float* w, int64_t S, int64_t K, float* alpha, float* sse, int32_t* idx,
                 int8_t* codes, uint8_t* packed) {
    t.w = w;
    t.S = S;
    t.K = K;
    t.alpha = alpha;
    t.sse = sse;
    t.best_idx = idx;
    t.codes = reinterpret_cast<signed char*>(codes);
    t.packed = packed;
    t.delta = nullptr;
    t.prior_alpha = nullptr;
    t.gate = nullptr;
    t.unit_begin = 0;
    t.rows_per_unit = (packed && (K & 1)) ? 2 : 1;
    t.lanes = 5;
    t.hist_fbits = t.hist_cshift = 0;
}

// The context's side streams and events, those that exist.
void release_launches(omse_ctx* ctx) {
    if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
    for (int i = 0; i < kSides; ++i) {
        if (ctx->ev_join[i]) cudaEventDestroy(ctx->ev_join[i]);
        if (ctx->side[i]) cudaStreamDestroy(ctx->side[i]);
    }
}

bool misaligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3) != 0; }

// ---- per-tensor search: the launches shared by omse_activation_scale* and the allocation-free entry point
struct TensorEnv {
    int n_sm;
    cudaStream_t stream;
    TensorLaunches* seen;
    unsigned long long* launches;   // launch counter of the caller
};

template <int MODE>
int pass_grid(const TensorEnv& env, long long n) {
    int& occ = env.seen->occ_pass[MODE];
    if (occ == 0 && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, omse::tensor_pass_kernel<MODE>, 256, 0) != cudaSuccess || occ < 1))
        occ = 4;
    long long grid = (n + 1023) / 1024;            // at least one float4 per thread
    if (grid > (long long)env.n_sm * occ) grid = (long long)env.n_sm * occ;   // one wave: every block is resident
    return grid < 1 ? 1 : (int)grid;
}

constexpr int kHistWindow = 8192;    // bins that the blocks of a histogram launch keep in shared memory
constexpr int kHistBlocks = 1024;    // its blocks at most (room for their sums)
constexpr int kScanChunks = 512;     // chunks of a window of many bins at most

int launch_hist(const TensorEnv& env, const omse::TensorArgs& a, bool full, int* n_blocks) {
    typedef void (*Kernel)(const omse::TensorArgs);
    const Kernel kernels[4] = {omse::tensor_hist_kernel<false, false>, omse::tensor_hist_kernel<false, true>,
                               omse::tensor_hist_kernel<true, false>, omse::tensor_hist_kernel<true, true>};
    const size_t smem = (size_t)a.shared_win * 20 + 8 * omse::kHotWords + (size_t)a.n_bins2 * 12;
    if (!env.seen->attr_hist) {
        for (const auto k : kernels)
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem - 4096) != cudaSuccess) return OMSE_ECUDA;   // (static: 4.6 KB)
        env.seen->attr_hist = true;
    }
    const int id = (full ? 2 : 0) + (a.lo < 0 ? 1 : 0);
    const Kernel kernel = kernels[id];
    auto& seen = env.seen->hist[id];
    if (seen.occ == 0 || seen.smem != smem) {
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, omse::kHistThreads, smem) != cudaSuccess || occ < 1) return OMSE_ECUDA;
        seen.occ = occ;
        seen.smem = smem;
    }
    long long grid = (a.n + omse::kHistChunk - 1) / omse::kHistChunk;
    if (grid > (long long)env.n_sm * seen.occ) grid = (long long)env.n_sm * seen.occ;
    if (grid > kHistBlocks) grid = kHistBlocks;
    *n_blocks = (int)grid;
    kernel<<<(unsigned)grid, omse::kHistThreads, smem, env.stream>>>(a);
    ++*env.launches;
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

// Bins of the per-tensor search: up to max|x| or, for a grid that ends far below it, up to the last threshold.
void tensor_bins(omse::TensorArgs& a) {
    const double all = 2.0 * (double)a.n_cand / (double)a.hi_frac * (1.0 + 1e-6);
    const double last = (double)(2 * a.hi - 1) * (double)a.n_cand;
    a.clipped = all > last ? 1 : 0;
    a.n_bins = std::max(1, (int)std::min(all, last));
    a.n_bins2 = 0;
    if (a.lo < 0) {
        const double all2 = all / (double)(-2 * a.lo - 1);
        a.n_bins2 = (int)std::min(all2, (double)a.n_cand);
    }
}

// Everything after the state has been cleared: maxima, histogram, scan, levels (once per window of bins), argmin, re-score,
// polish, final error.  `a` carries the buffers (a.partials: workspace of a.partial_doubles); the rest is filled here.
int enqueue_tensor_search(const TensorEnv& env, omse::TensorArgs& a, int refine_iters) {
    cudaStream_t s = env.stream;
    const long long n = a.n;
    tensor_bins(a);
    a.refine_iters = refine_iters;
    // the workspace until the passes take it over: the blocks' sums, <x,q> and <q,q>, then the histogram and N and P.  The blocks keep
    // up to kHistWindow bins in shared memory, and one block scans them; up to twice as many are two such windows, each with a
    // look at the tensor.  More bins (a grid that ends far below max|x|) are one window too where the workspace holds
    // them, N and P in the place of the histogram: the first ones, where most values of a heavy-tailed tensor lie, stay in
    // shared memory, the others are global.  51,380,224 values, windows of 8192 and this: post-ReLU, 1024 candidates to a tenth
    // of max|x| 973 us and 490, to a hundredth on 8 bits 6.0 ms and 0.51; uniform, 2048 candidates to a quarter (16,384 bins) 1.03
    // ms and 1.45, to a twentieth 3.24 and 2.0.
    double* at = a.partials;
    a.block_sums = at;
    a.levels = (at += omse::kBlockSums * kHistBlocks);
    a.chunks = (at += 2 * a.n_cand);
    at += 3 * kScanChunks;
    const bool few = a.n_bins <= 2 * kHistWindow;
    const long long room = a.partials + a.partial_doubles - at - 2ll * a.n_bins2;
    const int win = (int)std::min<long long>((a.n_bins + 3) & ~3, few ? kHistWindow : std::min<long long>(room / 2, (long long)kScanChunks * omse::kScanChunk) & ~3ll);
    const int n_win = (a.n_bins + win - 1) / win;
    a.win = win;
    a.shared_win = std::min(win, kHistWindow);
    const int hist_words = 2 * win + 2 * a.n_bins2;
    a.hist = reinterpret_cast<unsigned long long*>(at);
    a.above = few ? at + hist_words : at;
    if ((few ? 2 : 1) * (long long)hist_words > room + 2ll * a.n_bins2) return OMSE_ELIMIT;
    long long absmax_grid = (n + 1023) / 1024;
    if (absmax_grid > (long long)env.n_sm * 8) absmax_grid = (long long)env.n_sm * 8;
    if (absmax_grid < 1) absmax_grid = 1;
    if (n > 0) {
        omse::tensor_absmax_kernel<<<(unsigned)absmax_grid, 256, 0, s>>>(a.x, n, a.st, a.status, a.hist, hist_words);
        ++*env.launches;
        if (a.delta_out) {
            omse::tensor_offset_kernel<<<1, 32, 0, s>>>(a.st);
            ++*env.launches;
        }
        const bool full = a.n_bins <= kHistWindow && !a.clipped;      // every value in a bin, every bin in shared memory
        for (int w = n_win - 1; w >= 0; --w) {             // from the top down
            a.win_base = w * win;
            a.first_window = w == n_win - 1 ? 1 : 0;
            a.which = w & 1;
            if (!a.first_window && cudaMemsetAsync(a.hist, 0, 2 * (size_t)win * sizeof(double), s) != cudaSuccess) return OMSE_ECUDA;
            const int rc = launch_hist(env, a, full, &a.n_blocks);
            if (rc != OMSE_OK) return rc;
            if (few) {
                omse::tensor_scan_kernel<<<1, omse::kScanThreads, 0, s>>>(a);
            } else {
                a.n_chunks = (win + omse::kScanChunk - 1) / omse::kScanChunk;
                omse::tensor_chunks_kernel<<<(unsigned)(a.n_chunks + (a.first_window ? 1 : 0)), omse::kScanThreads, 0, s>>>(a);
                omse::tensor_chunk_scan_kernel<<<(unsigned)a.n_chunks, omse::kScanThreads, 0, s>>>(a);
                ++*env.launches;
            }
            ++*env.launches;
            if (!few || a.n_cand > omse::kLevelsHere) {
                omse::tensor_levels_kernel<<<(unsigned)((8 * a.n_cand + 255) / 256), 256, 0, s>>>(a);
                ++*env.launches;
            }
        }
    }
    omse::tensor_finish_kernel<<<1, 1024, 0, s>>>(a);
    omse::tensor_pass_kernel<0><<<(unsigned)pass_grid<0>(env, n), 256, 0, s>>>(a);
    const int g1 = pass_grid<1>(env, n);
    for (int it = 0; it < refine_iters; ++it) {
        a.first_pass = it == 0 ? 1 : 0;
        omse::tensor_pass_kernel<1><<<(unsigned)g1, 256, 0, s>>>(a);
    }
    omse::tensor_pass_kernel<2><<<(unsigned)pass_grid<2>(env, n), 256, 0, s>>>(a);
    *env.launches += 3 + (unsigned long long)refine_iters;   // argmin, re-score, polish steps, final
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

// The search in one kernel, for tensors that fit in the shared memory of all SMs together.  Returns OMSE_ELIMIT, with
// nothing enqueued, when this one does not, or when fewer SMs are there than the device has (a context or a stream limited to some
// of them, other users of a shared GPU): the launch is then refused, since the blocks would wait for ones that cannot run.
int enqueue_resident_search(const TensorEnv& env, omse::TensorArgs a, omse::ResidentExchange* ex, int max_blocks, unsigned int poll_limit,
                            int refine_iters) {
    if (a.n < 1 || a.n_cand > omse::kResidentCands) return OMSE_ELIMIT;
    tensor_bins(a);
    if (a.clipped || a.n_bins > omse::kResidentBins) return OMSE_ELIMIT;
    a.win = (a.n_bins + 3) & ~3;
    const size_t fixed = (size_t)(a.win + a.n_bins2) * 16 + (size_t)a.n_cand * 12 + 16;
    const long long n4 = (a.n + 3) >> 2, fit4 = (long long)((kMaxSmem - fixed) / 16);
    const long long blocks = std::min((long long)max_blocks, (n4 + omse::kResidentThreads - 1) / omse::kResidentThreads);
    if ((n4 + blocks - 1) / blocks > fit4 || (long long)a.n_cand * blocks > a.partial_doubles) return OMSE_ELIMIT;
    omse::ResidentArgs r;
    r.ex = ex;
    r.slice4 = (int)((n4 + blocks - 1) / blocks);
    r.rescore = a.partials;
    r.spin_limit = poll_limit;
    if (!env.seen->attr_resident) {
        if (cudaFuncSetAttribute(omse::tensor_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess)
            return OMSE_ECUDA;
        env.seen->attr_resident = true;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(omse::kResidentThreads);
    cfg.dynamicSmemBytes = fixed + (size_t)r.slice4 * 16;
    cfg.stream = env.stream;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof(attr));
    attr.id = cudaLaunchAttributeCooperative;       // every block runs: they wait for one another
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, omse::tensor_resident_kernel, (const omse::TensorArgs)a, (const omse::ResidentArgs)r, refine_iters);
    if (e != cudaSuccess) {
        cudaGetLastError();                         // not left for the next check of this thread
        return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported ? OMSE_ELIMIT : OMSE_ECUDA;
    }
    ++*env.launches;
    return OMSE_OK;
}

}  // namespace

namespace {

// How the scale of each row is found, for launches that do not use the default grid search with polish.
struct ListMode {
    int solver = 0, solver_iters = 0;   // comparison solvers of Section 3.4 (RowArgs::solver)
    int n_delta = 0;                    // offsets searched per row (0: none)
    float off_frac = 0.f;
};

// Launch for a list of weight tensors (bounds already set by the caller).
int quantize_list(omse_ctx* ctx, std::vector<omse::RowTensor>& list, int bits, int is_signed, const omse_grid* grid,
                  const ListMode& mode = ListMode()) {
    if (list.empty()) return OMSE_OK;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse::RowArgs a;
    memset(&a, 0, sizeof(a));
    a.n_cand = grid->n_cand;
    a.hi_frac = grid->hi_frac;
    a.refine_iters = grid->refine_iters;
    a.n_tensors = 1;
    a.n_sweeps = 1;
    bounds(bits, is_signed, &a.lo[0], &a.hi[0]);
    a.solver = mode.solver;
    a.solver_iters = mode.solver_iters;
    a.n_delta = mode.n_delta;
    a.off_frac = mode.off_frac;
    a.eps = -1.f;
    a.keep_x0 = mode.n_delta > 0 ? 1 : 0;   // every offset is applied to the original row
    // Which path a tensor's rows take.  Few rows keep a GPU of warps idle, and a block per row is sooner done, unless the
    // rows are so short that its barriers cost more (1200 rows of 288 values 22 us against 33 by blocks, 512 rows 20.5 and
    // 19.6; 512 rows of 147 values 26 and 27, of 27 values 16 and 24).  Short rows in small numbers go a candidate per lane,
    // whose chain is short, large numbers by splits, which evaluate less (6000 rows of 27 values 23 us against 31, 10,000
    // 40 and 33; 2400 rows of 288 values 29 and 33, 10,000 75 and 70; 1200 rows of 576 values 34 and 31); 8 bits, whose
    // best scale lies where the splits have furthest to go, change over later (10,000 rows of 27 values 41 and 52).
    // Rows of 1025 to 1280 values take a warp long, and few of them hold up a launch of short rows (1500 rows of 64 values and 20 of 1152, 4
    // bits, 256 candidates 43 us, 19 with those by blocks): they go by splits from 12 per SM on (3 bits, 256 candidates, 1500 rows of 1280
    // values 33 by blocks and 32, outliers 33 and 37; 1024 candidates, 1776 rows of 1152 46 and 40, 2400 of 1280 57 and 49), or from two per SM
    // beside 32 shorter rows per SM, which take as long anyway (10,000 rows of 64 values and 300 of 1152, 8 bits, 256 candidates 44 and 36).
    const bool plain = mode.solver == 0 && mode.n_delta == 0;   // the block path implements everything else
    long long short_rows = 0, short_elements = 0, short_warps = 0, mid_rows = 0, long_rows = 0, mid_elements = 0;
    bool longer = false;
    for (const auto& t : list) {
        if (t.K > kHistMaxK) {
            longer = true;
        } else if (t.K > kSmallK) {
            long_rows += t.S;
        } else if (t.K > kJoinK) {
            mid_rows += t.S;
            mid_elements += t.S * t.K;
        } else {
            short_rows += t.S;
            short_elements += t.S * t.K;
            short_warps += (t.S << omse::short_lanes(t.K)) / 32;
        }
    }
    // (Rows that go by a histogram below are counted here too: they fill the GPU beside the others.  Not counting them, 2000 rows of 64 values
    // and 8000 of 576 take 69 us instead of 90, but 10,000 of 64 and 2000 of 1152 on 8 bits 58 instead of 49.)
    const long long hist_rows = short_rows + mid_rows + long_rows;
    const bool join = mid_rows >= 12ll * ctx->n_sm || (short_rows >= 32ll * ctx->n_sm && mid_rows >= 2ll * ctx->n_sm);
    if (join) {
        short_rows += mid_rows;
        short_elements += mid_elements;
        short_warps += mid_rows;
    }
    const long long short_k = short_rows < 8ll * ctx->n_sm ? 160 : join ? kSmallK : kJoinK;
    a.short_direct = short_rows < (a.hi[0] > 63 ? 96ll : 48ll) * ctx->n_sm && short_elements < 5120ll * ctx->n_sm;
    int spread = 0;                                             // more lanes per row where the warps do not fill the GPU
    while (spread < 5 && (short_warps << (spread + 1)) <= 16ll * ctx->n_sm) ++spread;
    std::vector<int> path_of(list.size(), kPathBlock);
    // Rows by a histogram of their warp.
    a.n_bins = all_bins(a.n_cand, a.hi_frac);
    a.hist_lb = 4;
    while (a.hist_lb < 6 && (32 << a.hist_lb) < a.n_bins) ++a.hist_lb;
    const int hist_words = 32 << a.hist_lb;
    // (the largest |x|/h, rounded up to a fraction, lies in a bin)
    const bool hist_fits = plain && a.hi[0] >= 7 && a.n_bins > 0 &&
                           2.0 * a.n_cand / (double)a.hi_frac * (1.0 + 4e-7) + 1.0 / 64 < (double)hist_words + 1.0;
    // A row takes a warp 15 to 30 us, a block a third of that: with fewer than seven rows per SM blocks are sooner done (1036 rows of 1024
    // values on 4 bits, 1024 candidates 33 us by blocks and 24, of 2304 42 and 40; 592 of 2304 28 and 37), and down to four only where they have
    // many candidates to look at and not many levels (592 of 576 values on 4 bits 21 and 19, of 768 23 and 22, 256 candidates and 448 values 15 and
    // 17; on 8 bits 592 of 768 21 and 25).  Rows of more than 1280 values beside longer ones, whose blocks are on the SMs anyway, from 16 per
    // SM on (256 candidates, 512 rows of 4608 and 1200 of 2304 values 53 by blocks and 65, 2700 of 2048 79 and 69).  And beside rows of other
    // paths the launch has to be worth its cost.  Less than 2M values: rows of up to 1024 values, the others by blocks (8192 rows of 128 values
    // and 1200 of 576 49 and 54 with a launch for those, 3600 of 576 61 and 69; 512 of 4608 and 1200 of 1152 on 8 bits 58 and 63), where
    // they are a quarter of all values (100 rows of 25,088 and 1200 of 1000 74 and 49, 4000 of 128 and 300 of 720 45 and 30) and the list is
    // short (a call with 54 tensors takes the host 130 us, a launch more some 6).  Launches that fill the GPU many times over are bound by
    // issue, not by chains, and the splits of up to 447 values are the cheaper ones there (150,000 rows of 400, 1024 candidates 916 and 941,
    // Student-t 861 and 920; 24,000 rows 166 and 154), on 5 bits with few candidates up to 639 (256 candidates, 576 values 910 and 923, 830 and 917).
    long long hist_from = a.hi[0] > 15 ? kHistK8 : kHistK4, hist_to = kHistMaxK, hist_elements = 0, other_elements = 0;
    if (hist_rows >= 256ll * ctx->n_sm) hist_from = std::max<long long>(hist_from, a.hi[0] > 7 && a.n_cand < 512 ? 640 : 448);
    if (longer && long_rows < 16ll * ctx->n_sm) hist_to = kSmallK;
    if (hist_rows < 7ll * ctx->n_sm) hist_to = a.hi[0] > 15 || a.n_cand < 512 ? 0 : 800;
    if (!hist_fits || hist_rows < 4ll * ctx->n_sm) hist_to = 0;
    auto by_hist = [&](const omse::RowTensor& t) { return t.K >= hist_from && t.K <= hist_to; };
    auto share = [&]() {
        hist_elements = other_elements = 0;
        for (const auto& t : list) (by_hist(t) ? hist_elements : other_elements) += t.S * t.K;
    };
    share();
    if (other_elements > 0 && hist_elements < 1 << 21) {
        hist_from = std::max(hist_from, kHistK8);
        hist_to = std::min(hist_to, kJoinK);
        share();
        if (3 * hist_elements < other_elements || list.size() > 32) hist_to = 0;
    }
    // One launch per row path present in the list: each launch then runs the kernel instantiation that holds only its path.
    // Longest rows first inside a launch: the dispenser hands out work in decreasing size and the tail is short.
    std::stable_sort(list.begin(), list.end(), [](const omse::RowTensor& x, const omse::RowTensor& y) { return x.K > y.K; });
    bool present[kPaths] = {};
    for (size_t i = 0; i < list.size(); ++i) {
        omse::RowTensor& t = list[i];
        if (by_hist(t)) {
            // count and fractions of all values in one word, bin and fraction in 23 bits
            int count = 1, frac = 1;
            while ((1ll << count) <= t.K) ++count;
            while (frac < 12 && (t.K << (frac + 1)) <= (1ll << (32 - count)) && ((long long)hist_words << (frac + 1)) <= (1ll << 23)) ++frac;
            path_of[i] = kPathHist;
            t.hist_fbits = frac;
            t.hist_cshift = 32 - count;
        } else if (plain && t.K <= short_k) {
            path_of[i] = kPathShort;
            t.lanes = a.short_direct ? 5 : omse::short_lanes(t.K);
            for (int s = 0; s < spread && t.lanes < 5 && (4ll << t.lanes) < t.K; ++s) ++t.lanes;
        }
        if (path_of[i] != kPathBlock) {
            // several steps of a warp per unit, so that the dispenser is not the limit, where every warp of the GPU still
            // gets a few units; an even number of rows, for the packed nibbles
            const long long groups = 32 >> t.lanes, many = t.S / (groups * 128 * ctx->n_sm);
            t.rows_per_unit = (int)std::max((long long)t.rows_per_unit, groups * (many >= 2 ? std::min(many, 16ll) & ~1ll : 1));
        }
        present[path_of[i]] = true;
    }
    // The tensors of each path, one after the other; one copy for all descriptors.
    std::vector<omse::RowTensor> sorted;
    int first_of[kPaths + 1] = {}, last = 0;
    for (int path = 0; path < kPaths; ++path) {
        long long units = 0;
        for (size_t i = 0; i < list.size(); ++i) {
            if (path_of[i] != path) continue;
            list[i].unit_begin = units;
            units += (list[i].S + list[i].rows_per_unit - 1) / list[i].rows_per_unit;
            sorted.push_back(list[i]);
        }
        first_of[path + 1] = (int)sorted.size();
        if (present[path]) last = path;
    }
    if (sorted.size() > 1 && cudaMemcpyAsync(ctx->d_tensors, sorted.data(), sizeof(omse::RowTensor) * sorted.size(), cudaMemcpyHostToDevice,
                                             ctx->stream) != cudaSuccess)
        return OMSE_ECUDA;
    // With rows of several paths in the list, the launches of the shorter rows go first, on side streams (forked from and joined to
    // the context's stream by events, with work dispensers of their own), and the longest rows' launch runs beside them: the blocks
    // of the next one fill the SMs as the blocks of the first run out of work, so only one tail is left.  The launches touch
    // different tensors.
    bool forked[kSides] = {};
    int rc_all = OMSE_OK;
    for (int path = 0; path <= last && rc_all == OMSE_OK; ++path) {
        if (!present[path]) continue;
        const omse::RowTensor* sub = sorted.data() + first_of[path];
        a.n_launch_tensors = first_of[path + 1] - first_of[path];
        a.ext_tensors = 0;
        int rows4 = 0, groups_most = 0, codes_most = 0;
        long long sub_max_k = 0;
        for (int i = 0; i < a.n_launch_tensors; ++i) {
            const omse::RowTensor& t = sub[i];
            const int groups = 32 >> t.lanes;
            a.ext_tensors |= (t.gate || t.prior_alpha) ? 1 : 0;
            sub_max_k = std::max(sub_max_k, t.K);
            if (path == kPathBlock) continue;
            rows4 = std::max(rows4, groups * omse::short_stride4((int)((t.K + 3) >> 2), t.lanes));
            groups_most = std::max(groups_most, groups);
            codes_most = std::max(codes_most, (int)(groups * t.K));
        }
        const omse::RowTensor& end = sub[a.n_launch_tensors - 1];
        a.n_units = end.unit_begin + (end.S + end.rows_per_unit - 1) / end.rows_per_unit;
        if (path != kPathBlock) {
            const int by_lanes = (omse::kMaxCoarse + omse::kHullValues) / 2;
            a.short_rows4 = rows4;
            a.short_slots = path == kPathHist ? std::max((hist_words + omse::kMaxCoarse) / 2, by_lanes)      // (rows of extreme values go by lanes)
                            : a.short_direct  ? by_lanes : groups_most * omse::short_slots(a.n_cand);
            a.short_codes = a.short_rows4 * 16;    // the codes come where the search's stack has been
            a.short_bytes = (a.short_codes + std::max(a.short_slots * 8 + omse::kShortClose * groups_most * 2, codes_most + 16) + 15) & ~15;
        }
        a.tensors = a.n_launch_tensors > 1 ? ctx->d_tensors + first_of[path] : nullptr;
        a.one = sub[0];
        const bool on_side = path != last;
        cudaStream_t own = ctx->stream;
        if (on_side) {
            if (cudaEventRecord(ctx->ev_fork, own) != cudaSuccess || cudaStreamWaitEvent(ctx->side[path], ctx->ev_fork, 0) != cudaSuccess) {
                rc_all = OMSE_ECUDA;
                break;
            }
            forked[path] = true;
            ctx->stream = ctx->side[path];
            ctx->ticket_pair = 1 + path;
        }
        rc_all = launch_rows(ctx, a, sub_max_k, path);
        if (on_side) {
            ctx->stream = own;
            ctx->ticket_pair = 0;
        }
    }
    for (int i = 0; i < kSides; ++i)   // a side stream always rejoins, also after an error
        if (forked[i] && (cudaEventRecord(ctx->ev_join[i], ctx->side[i]) != cudaSuccess ||
                          cudaStreamWaitEvent(ctx->stream, ctx->ev_join[i], 0) != cudaSuccess))
            rc_all = rc_all == OMSE_OK ? OMSE_ECUDA : rc_all;
    return rc_all;
}

}  // namespace

static int activation_impl(omse_ctx* ctx, const float* d_x, int64_t n, int bits, int is_signed, const omse_grid* grid,
                           float* d_alpha, float* d_delta, float* d_sse, int32_t* d_best_idx, double* d_sse_curve);

extern "C" {

const char* omse_status_string(int status) {
    switch (status) {
        case OMSE_OK: return "ok";
        case OMSE_EINVAL: return "invalid argument";
        case OMSE_ECUDA: return "CUDA runtime or launch failure";
        case OMSE_ENOMEM: return "out of device memory";
        case OMSE_ELIMIT: return "size beyond the fixed scratch of the allocation-free entry point";
        default: return "unknown status";
    }
}

int omse_create(omse_ctx** out, int device, void* cuda_stream) {
    if (!out) return OMSE_EINVAL;
    *out = nullptr;
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device < 0 || device >= n_dev) return OMSE_ECUDA;
    DeviceScope dev(device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse_ctx* c = new (std::nothrow) omse_ctx;
    if (!c) return OMSE_ENOMEM;
    memset(c, 0, sizeof(*c));
    c->device = device;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    c->ws = nullptr;
    c->partials = nullptr;
    c->d_tensors = nullptr;
    c->poll_limit = omse::kSpinLimit;
    if (cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
        delete c;
        return OMSE_ECUDA;
    }
    c->search_blocks = std::min(c->n_sm, omse::kResidentBlocks);
    if (cudaMalloc(&c->ws, sizeof(Workspace)) != cudaSuccess || cudaMalloc(&c->partials, kPartialBytes) != cudaSuccess ||
        cudaMalloc(&c->d_tensors, sizeof(omse::RowTensor) * OMSE_MAX_BATCH) != cudaSuccess) {
        cudaFree(c->ws);
        cudaFree(c->partials);
        delete c;
        cudaGetLastError();
        return OMSE_ENOMEM;
    }
    bool ok = cudaMemsetAsync(c->ws, 0, sizeof(Workspace), c->stream) == cudaSuccess &&
              cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; i < kSides && ok; ++i)
        ok = cudaStreamCreateWithFlags(&c->side[i], cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&c->ev_join[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        release_launches(c);
        cudaFree(c->ws);
        cudaFree(c->partials);
        cudaFree(c->d_tensors);
        delete c;
        cudaGetLastError();
        return OMSE_ECUDA;
    }
    *out = c;
    return OMSE_OK;
}

int omse_destroy(omse_ctx* ctx) {
    if (!ctx) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    for (cudaStream_t s : ctx->side) cudaStreamSynchronize(s);
    release_launches(ctx);
    cudaFree(ctx->ws);
    cudaFree(ctx->partials);
    cudaFree(ctx->d_tensors);
    delete ctx;
    return OMSE_OK;
}

int omse_set_stream(omse_ctx* ctx, void* cuda_stream) {
    if (!ctx) return OMSE_EINVAL;
    ctx->stream = static_cast<cudaStream_t>(cuda_stream);
    return OMSE_OK;
}

size_t omse_workspace_bytes(int64_t n_kernels, int64_t kernel_len, int32_t n_cand, int32_t n_tensors) {
    // Rows are searched on chip, so the workspace does not grow with the problem: status and dispenser words, the
    // per-tensor search state and curve, per-block partial sums, descriptors of a batched launch.
    if (n_kernels < 0 || kernel_len < 1 || n_cand < 1 || n_cand > OMSE_MAX_CANDIDATES || n_tensors < 1 ||
        n_tensors > OMSE_MAX_TENSORS)
        return 0;
    return sizeof(Workspace) + kPartialBytes + sizeof(omse::RowTensor) * OMSE_MAX_BATCH;
}

int omse_last_device_status(omse_ctx* ctx, uint32_t* host_out) {
    if (!ctx || !host_out) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    if (cudaMemcpyAsync(host_out, &ctx->ws->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess)
        return OMSE_ECUDA;
    if (cudaMemsetAsync(&ctx->ws->status, 0, sizeof(uint32_t), ctx->stream) != cudaSuccess) return OMSE_ECUDA;
    return cudaStreamSynchronize(ctx->stream) == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

int omse_read_launches(omse_ctx* ctx, uint64_t* host_out) {
    if (!ctx || !host_out) return OMSE_EINVAL;
    *host_out = ctx->n_launches;
    ctx->n_launches = 0;
    return OMSE_OK;
}

int omse_set_search_blocks(omse_ctx* ctx, int blocks) {
    if (!ctx || blocks < 1 || blocks > omse::kResidentBlocks) return OMSE_EINVAL;
    ctx->search_blocks = blocks;
    return OMSE_OK;
}

int omse_set_poll_limit(omse_ctx* ctx, uint32_t polls) {
    if (!ctx) return OMSE_EINVAL;
    ctx->poll_limit = polls;
    return OMSE_OK;
}

int omse_read_evaluations(omse_ctx* ctx, uint64_t* host_out) {
    if (!ctx || !host_out) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    unsigned long long v = 0;
    if (cudaMemcpyAsync(&v, &ctx->ws->evals, sizeof(v), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess) return OMSE_ECUDA;
    if (cudaMemsetAsync(&ctx->ws->evals, 0, sizeof(v), ctx->stream) != cudaSuccess) return OMSE_ECUDA;
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) return OMSE_ECUDA;
    *host_out = v;
    return OMSE_OK;
}

int omse_measure_fp32_peak(omse_ctx* ctx, int target_ms, double* host_out) {
    if (!ctx || !host_out || target_ms < 1 || target_ms > 5000) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    const int blocks = ctx->n_sm * 4, threads = 256;
    float* out = reinterpret_cast<float*>(ctx->partials);        // blocks*threads floats, far below the 16 MB held
    // iterations for about target_ms at 128 lane operations per clock and SM at 2 GHz
    const double lane_ops_per_iter = (double)blocks * threads * omse::kPeakChains * 2.0;
    long long iters = (long long)((double)target_ms * 1e-3 * (double)ctx->n_sm * 128.0 * 2.0e9 / lane_ops_per_iter);
    if (iters < 1024) iters = 1024;
    if (iters > 0x7fffffff) iters = 0x7fffffff;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return OMSE_ECUDA;
    }
    omse::fma_peak_kernel<<<blocks, threads, 0, ctx->stream>>>(out, 4096, 1.0f);      // warm-up
    cudaEventRecord(e0, ctx->stream);
    omse::fma_peak_kernel<<<blocks, threads, 0, ctx->stream>>>(out, (int)iters, 1.0f);
    cudaEventRecord(e1, ctx->stream);
    float ms = 0.f;
    const bool ok = cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess &&
                    cudaGetLastError() == cudaSuccess && ms > 0.f;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (!ok) return OMSE_ECUDA;
    *host_out = lane_ops_per_iter * (double)iters / ((double)ms * 1e-3);
    return OMSE_OK;
}

int omse_quantize_weights(omse_ctx* ctx, const float* d_w, int64_t n_kernels, int64_t kernel_len, int bits,
                          int is_signed, const omse_grid* grid, float* d_alpha, float* d_sse,
                          int32_t* d_best_idx, int8_t* d_codes, uint8_t* d_packed) {
    omse_weight_tensor t;
    t.d_w = d_w;
    t.n_kernels = n_kernels;
    t.kernel_len = kernel_len;
    t.d_alpha = d_alpha;
    t.d_sse = d_sse;
    t.d_best_idx = d_best_idx;
    t.d_codes = d_codes;
    t.d_packed = d_packed;
    return omse_quantize_weights_batched(ctx, &t, 1, bits, is_signed, grid);
}

int omse_quantize_weights_batched(omse_ctx* ctx, const omse_weight_tensor* tensors, int n_tensors, int bits,
                                  int is_signed, const omse_grid* grid) {
    if (!ctx || !grid_ok(grid) || bits < 2 || bits > 8 || n_tensors < 0 || n_tensors > OMSE_MAX_BATCH ||
        (n_tensors > 0 && !tensors))
        return OMSE_EINVAL;
    std::vector<omse::RowTensor> list;
    list.reserve((size_t)n_tensors);
    for (int i = 0; i < n_tensors; ++i) {
        const omse_weight_tensor& u = tensors[i];
        if (u.n_kernels < 0 || u.kernel_len < 1 || u.kernel_len > OMSE_MAX_KERNEL_LEN || u.n_kernels > (int64_t)1 << 40)
            return OMSE_EINVAL;
        if (u.d_packed && bits > 4) return OMSE_EINVAL;
        if (u.n_kernels == 0) continue;
        if (!u.d_w || !u.d_alpha || !u.d_sse) return OMSE_EINVAL;
        if (misaligned4(u.d_w) || misaligned4(u.d_alpha) || misaligned4(u.d_sse) || misaligned4(u.d_best_idx))
            return OMSE_EINVAL;
        omse::RowTensor t;
        fill_tensor(t, u.d_w, u.n_kernels, u.kernel_len, u.d_alpha, u.d_sse, u.d_best_idx, u.d_codes, u.d_packed);
        list.push_back(t);
    }
    return quantize_list(ctx, list, bits, is_signed, grid);
}

int omse_quantize_weights_offset(omse_ctx* ctx, const float* d_w, int64_t n_kernels, int64_t kernel_len, int bits,
                                 const omse_grid* grid, float* d_alpha, float* d_delta, float* d_sse,
                                 int32_t* d_best_idx, int8_t* d_codes, uint8_t* d_packed) {
    if (!ctx || !grid_ok(grid) || bits < 2 || bits > 8 || n_kernels < 0 || kernel_len < 1 ||
        kernel_len > OMSE_MAX_KERNEL_LEN || n_kernels > (int64_t)1 << 40 || (d_packed && bits > 4))
        return OMSE_EINVAL;
    if (n_kernels == 0) return OMSE_OK;
    if (!d_w || !d_alpha || !d_sse || !d_delta) return OMSE_EINVAL;
    if (misaligned4(d_w) || misaligned4(d_alpha) || misaligned4(d_sse) || misaligned4(d_best_idx) || misaligned4(d_delta))
        return OMSE_EINVAL;
    std::vector<omse::RowTensor> list(1);
    fill_tensor(list[0], d_w, n_kernels, kernel_len, d_alpha, d_sse, d_best_idx, d_codes, d_packed);
    list[0].delta = d_delta;
    return quantize_list(ctx, list, bits, /*is_signed=*/0, grid);
}

int omse_residual_quantize(omse_ctx* ctx, const float* d_t, int64_t n_kernels, int64_t kernel_len, const int* bits,
                           int is_signed, const omse_grid* grid, int n_tensors, int n_sweeps, float* d_alpha,
                           float* d_sse, int8_t* d_codes, uint8_t* d_packed) {
    int flags[OMSE_MAX_TENSORS];
    for (int j = 0; j < OMSE_MAX_TENSORS; ++j) flags[j] = is_signed;
    return omse_alg1_quantize(ctx, d_t, n_kernels, kernel_len, bits, flags, grid, n_tensors, n_sweeps, d_alpha, d_sse,
                              nullptr, d_codes, d_packed);
}

static int alg1_impl(omse_ctx* ctx, const float* d_t, int64_t n_kernels, int64_t kernel_len, const int* bits,
                     const int* is_signed, const omse_grid* grid, int n_tensors, int n_sweeps, float eps, float* d_alpha,
                     float* d_sse, float* d_sse_history, int32_t* d_sweeps_done, int8_t* d_codes, uint8_t* d_packed) {
    if (!ctx || !grid_ok(grid) || !bits || !is_signed || n_tensors < 1 || n_tensors > OMSE_MAX_TENSORS || n_sweeps < 1 ||
        n_sweeps > 64 || n_kernels < 0 || kernel_len < 1 || kernel_len > OMSE_MAX_KERNEL_LEN ||
        n_kernels > (int64_t)1 << 40)
        return OMSE_EINVAL;
    for (int j = 0; j < n_tensors; ++j) {
        if (bits[j] < 2 || bits[j] > 8) return OMSE_EINVAL;
        if (d_packed && bits[j] > 4) return OMSE_EINVAL;
    }
    if (n_sweeps > 1 && (!d_codes || kernel_len > OMSE_MAX_KERNEL_LEN_MULTISWEEP)) return OMSE_EINVAL;
    if (n_kernels == 0) return OMSE_OK;
    if (!d_t || !d_alpha || !d_sse) return OMSE_EINVAL;
    if (misaligned4(d_t) || misaligned4(d_alpha) || misaligned4(d_sse) || misaligned4(d_sse_history) ||
        misaligned4(d_sweeps_done))
        return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse::RowArgs a;
    memset(&a, 0, sizeof(a));
    fill_tensor(a.one, d_t, n_kernels, kernel_len, d_alpha, d_sse, nullptr, d_codes, d_packed);
    a.tensors = nullptr;
    a.n_launch_tensors = 1;
    a.n_units = (n_kernels + a.one.rows_per_unit - 1) / a.one.rows_per_unit;
    a.n_cand = grid->n_cand;
    a.hi_frac = grid->hi_frac;
    a.refine_iters = grid->refine_iters;
    a.n_tensors = n_tensors;
    a.n_sweeps = n_sweeps;
    for (int j = 0; j < n_tensors; ++j) bounds(bits[j], is_signed[j], &a.lo[j], &a.hi[j]);
    a.keep_x0 = n_sweeps > 1 ? 1 : 0;
    a.sse_history = d_sse_history;
    a.eps = eps;
    a.sweeps_done = d_sweeps_done;
    return launch_rows(ctx, a, kernel_len, kPathBlock);   // Algorithm 1 always takes the block-per-row path
}

int omse_alg1_quantize(omse_ctx* ctx, const float* d_t, int64_t n_kernels, int64_t kernel_len, const int* bits,
                       const int* is_signed, const omse_grid* grid, int n_tensors, int n_sweeps, float* d_alpha,
                       float* d_sse, float* d_sse_history, int8_t* d_codes, uint8_t* d_packed) {
    return alg1_impl(ctx, d_t, n_kernels, kernel_len, bits, is_signed, grid, n_tensors, n_sweeps, -1.f, d_alpha, d_sse,
                     d_sse_history, nullptr, d_codes, d_packed);
}

int omse_alg1_quantize_converge(omse_ctx* ctx, const float* d_t, int64_t n_kernels, int64_t kernel_len, const int* bits,
                                const int* is_signed, const omse_grid* grid, int n_tensors, int max_sweeps, float eps,
                                float* d_alpha, float* d_sse, float* d_sse_history, int32_t* d_sweeps_done,
                                int8_t* d_codes, uint8_t* d_packed) {
    if (!(eps >= 0.f)) return OMSE_EINVAL;
    return alg1_impl(ctx, d_t, n_kernels, kernel_len, bits, is_signed, grid, n_tensors, max_sweeps, eps, d_alpha, d_sse,
                     d_sse_history, d_sweeps_done, d_codes, d_packed);
}

int omse_quantize_weights_solver(omse_ctx* ctx, const float* d_w, int64_t n_kernels, int64_t kernel_len, int bits,
                                 int is_signed, int solver, int n_iter, const omse_grid* grid, float* d_alpha,
                                 float* d_sse, int32_t* d_best_idx, int8_t* d_codes, uint8_t* d_packed) {
    if (solver == OMSE_SOLVER_GRID)
        return omse_quantize_weights(ctx, d_w, n_kernels, kernel_len, bits, is_signed, grid, d_alpha, d_sse, d_best_idx,
                                     d_codes, d_packed);
    if (!ctx || !grid_ok(grid) || bits < 2 || bits > 8 || n_kernels < 0 || kernel_len < 1 ||
        kernel_len > OMSE_MAX_KERNEL_LEN || n_kernels > (int64_t)1 << 40 || (d_packed && bits > 4) ||
        solver < OMSE_SOLVER_UNIFORM || solver > OMSE_SOLVER_GOLDEN || n_iter < 0 || n_iter > 1024)
        return OMSE_EINVAL;
    if (n_kernels == 0) return OMSE_OK;
    if (!d_w || !d_alpha || !d_sse) return OMSE_EINVAL;
    if (misaligned4(d_w) || misaligned4(d_alpha) || misaligned4(d_sse) || misaligned4(d_best_idx)) return OMSE_EINVAL;
    std::vector<omse::RowTensor> list(1);
    fill_tensor(list[0], d_w, n_kernels, kernel_len, d_alpha, d_sse, d_best_idx, d_codes, d_packed);
    ListMode mode;
    mode.solver = solver;
    mode.solver_iters = n_iter;
    return quantize_list(ctx, list, bits, is_signed, grid, mode);
}

int omse_quantize_weights_affine(omse_ctx* ctx, const float* d_w, int64_t n_kernels, int64_t kernel_len, int bits,
                                 const omse_grid* grid, const omse_offset_grid* offsets, float* d_alpha, float* d_delta,
                                 float* d_sse, int32_t* d_best_idx, int8_t* d_codes, uint8_t* d_packed) {
    if (!ctx || !grid_ok(grid) || !offsets || offsets->n_delta < 1 || offsets->n_delta > OMSE_MAX_OFFSETS ||
        !(offsets->off_frac >= 0.f) || !(offsets->off_frac <= 1.f) || bits < 2 || bits > 8 || n_kernels < 0 ||
        kernel_len < 1 || kernel_len > OMSE_MAX_KERNEL_LEN_MULTISWEEP || n_kernels > (int64_t)1 << 40 ||
        (d_packed && bits > 4) || (int64_t)offsets->n_delta * grid->n_cand > 0x7fffffff)
        return OMSE_EINVAL;
    if (n_kernels == 0) return OMSE_OK;
    if (!d_w || !d_alpha || !d_sse || !d_delta) return OMSE_EINVAL;
    if (misaligned4(d_w) || misaligned4(d_alpha) || misaligned4(d_sse) || misaligned4(d_best_idx) || misaligned4(d_delta))
        return OMSE_EINVAL;
    std::vector<omse::RowTensor> list(1);
    fill_tensor(list[0], d_w, n_kernels, kernel_len, d_alpha, d_sse, d_best_idx, d_codes, d_packed);
    list[0].delta = d_delta;
    ListMode mode;
    mode.n_delta = offsets->n_delta;
    mode.off_frac = offsets->off_frac;
    return quantize_list(ctx, list, bits, /*is_signed=*/0, grid, mode);
}

int omse_quantize_key_layers(omse_ctx* ctx, const omse_key_layer* layers, int n_layers, int bits, int is_signed,
                             const omse_grid* grid, float tau, double* d_mse, int32_t* d_is_key, double* d_cr) {
    if (!ctx || !grid_ok(grid) || bits < 2 || bits > 8 || n_layers < 0 || n_layers > OMSE_MAX_BATCH ||
        (n_layers > 0 && (!layers || !d_mse || !d_is_key)) || !(tau >= 0.f))
        return OMSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_mse) & 7) || (reinterpret_cast<uintptr_t>(d_cr) & 7) || misaligned4(d_is_key))
        return OMSE_EINVAL;
    std::vector<omse_weight_tensor> first((size_t)n_layers);
    std::vector<omse_layer_error> errs((size_t)n_layers);
    for (int l = 0; l < n_layers; ++l) {
        const omse_key_layer& L = layers[l];
        if (L.first.n_kernels < 1 || L.first.kernel_len < 1 || L.first.kernel_len > OMSE_MAX_KERNEL_LEN ||
            !L.d_alpha2 || !L.d_sse2 || misaligned4(L.d_alpha2) || misaligned4(L.d_sse2) || (L.d_packed2 && bits > 4))
            return OMSE_EINVAL;
        first[l] = L.first;
        errs[l].d_sse = L.first.d_sse;
        errs[l].n_kernels = L.first.n_kernels;
        errs[l].kernel_len = L.first.kernel_len;
    }
    if (n_layers == 0) return OMSE_OK;
    // 1. every layer with one quantized tensor; 2. MSE per layer against tau
    int rc = omse_quantize_weights_batched(ctx, first.data(), n_layers, bits, is_signed, grid);
    if (rc != OMSE_OK) return rc;
    rc = omse_select_key_layers(ctx, errs.data(), n_layers, tau, d_mse, d_is_key);
    if (rc != OMSE_OK) return rc;
    // 3. one launch over all layers for the second tensor: blocks skip the layers whose flag is 0, so the host
    //    never reads the flags; each row's residual is rebuilt on chip from the first scale
    std::vector<omse::RowTensor> list((size_t)n_layers);
    for (int l = 0; l < n_layers; ++l) {
        const omse_key_layer& L = layers[l];
        fill_tensor(list[l], L.first.d_w, L.first.n_kernels, L.first.kernel_len, L.d_alpha2, L.d_sse2, nullptr,
                    L.d_codes2, L.d_packed2);
        list[l].prior_alpha = L.first.d_alpha;
        list[l].gate = d_is_key + l;
    }
    rc = quantize_list(ctx, list, bits, is_signed, grid);
    if (rc != OMSE_OK) return rc;
    // 4. compression ratio of the result (one or two quantized tensors per layer)
    if (d_cr) {
        DeviceScope dev(ctx->device);
        if (!dev.ok()) return OMSE_ECUDA;
        std::vector<omse::LayerError> shape((size_t)n_layers);
        for (int l = 0; l < n_layers; ++l) {
            shape[l].sse = nullptr;
            shape[l].n_kernels = layers[l].first.n_kernels;
            shape[l].kernel_len = layers[l].first.kernel_len;
        }
        omse::LayerError* d_layers = reinterpret_cast<omse::LayerError*>(ctx->d_tensors);
        if (cudaMemcpyAsync(d_layers, shape.data(), sizeof(omse::LayerError) * shape.size(), cudaMemcpyHostToDevice,
                            ctx->stream) != cudaSuccess)
            return OMSE_ECUDA;
        omse::compression_ratio_kernel<<<1, 32, 0, ctx->stream>>>(d_layers, n_layers, bits, d_is_key, d_cr);
        ++ctx->n_launches;
        if (cudaGetLastError() != cudaSuccess) return OMSE_ECUDA;
    }
    return OMSE_OK;
}

int omse_dual_quantize(omse_ctx* ctx, const float* d_t, int64_t n_kernels, int64_t kernel_len, int bits1, int bits2,
                       int is_signed, const omse_dual_grid* grid, float* d_alpha, float* d_sse, int32_t* d_best_idx,
                       int8_t* d_codes, uint8_t* d_packed) {
    if (!ctx || !grid || grid->n_cand1 < 1 || grid->n_cand2 < 1 || grid->n_cand1 > OMSE_DUAL_MAX_CANDIDATES ||
        grid->n_cand2 > OMSE_DUAL_MAX_CANDIDATES || !(grid->hi_frac1 > 0.f) || !(grid->hi_frac2 > 0.f) ||
        !(grid->hi_frac1 <= 3.0e38f) || !(grid->hi_frac2 <= 3.0e38f) || bits1 < 2 || bits1 > 8 || bits2 < 2 ||
        bits2 > 8 || n_kernels < 0 || kernel_len < 1 || kernel_len > OMSE_MAX_KERNEL_LEN || n_kernels > (int64_t)1 << 40)
        return OMSE_EINVAL;
    if (d_packed && (bits1 > 4 || bits2 > 4)) return OMSE_EINVAL;
    if (n_kernels == 0) return OMSE_OK;
    if (!d_t || !d_alpha || !d_sse) return OMSE_EINVAL;
    if (misaligned4(d_t) || misaligned4(d_alpha) || misaligned4(d_sse) || misaligned4(d_best_idx)) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse::DualArgs a;
    memset(&a, 0, sizeof(a));
    a.t = d_t;
    a.S = n_kernels;
    a.K = kernel_len;
    a.n_cand1 = grid->n_cand1;
    a.n_cand2 = grid->n_cand2;
    a.hi_frac1 = grid->hi_frac1;
    a.hi_frac2 = grid->hi_frac2;
    bounds(bits1, is_signed, &a.lo1, &a.hi1);
    bounds(bits2, is_signed, &a.lo2, &a.hi2);
    a.alpha = d_alpha;
    a.sse = d_sse;
    a.best_idx = d_best_idx;
    a.codes = reinterpret_cast<signed char*>(d_codes);
    a.packed = d_packed;
    a.status = &ctx->ws->status;
    a.rows_per_unit = (d_packed && (kernel_len & 1)) ? 2 : 1;
    // Which of the two kernels: see dual_bound_kernel.  Where alpha1 comes near the last place of max|x| (2^-23 of it) binary32 cannot
    // tell neighbouring first codes apart and the reference takes the lowest one, which only the full enumeration finds.
    const bool bound = kernel_len >= kDualBoundK && bits1 + bits2 <= 8 && grid->hi_frac2 <= 1.0f &&
                       (double)grid->hi_frac1 * 1048576.0 >= (double)grid->n_cand1;
    const long long n_units = (n_kernels + a.rows_per_unit - 1) / a.rows_per_unit;
    const bool few = n_units <= 3ll * ctx->n_sm;
    const int id = !bound ? 0 : few ? 1 : 2;
    const void* kernel = !bound ? (const void*)omse::dual_kernel
                         : few ? (const void*)omse::dual_bound_kernel<3> : (const void*)omse::dual_bound_kernel<4>;
    const int threads = bound ? omse::kDualBoundThreads : omse::kDualThreads;
    const size_t row_bytes = (size_t)((kernel_len + 3) & ~3ll) * 4;
    const size_t smem = bound ? 2 * omse::kDualBins * sizeof(omse::DualBin) + row_bytes : row_bytes + 64 * 8 + omse::kDualListCap * 4 + 4 * 4;
    if (!ctx->attr_dual[id]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess) return OMSE_ECUDA;
        ctx->attr_dual[id] = true;
    }
    const int occ = blocks_per_sm(ctx, kRowKernels + id, kernel, threads, smem);
    if (occ == 0) return OMSE_ECUDA;
    long long blocks = (long long)ctx->n_sm * occ;
    if (blocks > n_units) blocks = n_units;
    // the context workspace holds the sorted points of every alpha2, then each block's grid values of its current row
    const size_t point_bytes = bound ? (size_t)grid->n_cand2 * 2 * omse::kDualSide * sizeof(omse::DualPoint) : 0;
    const long long cap = (long long)((kPartialBytes - point_bytes) / ((size_t)grid->n_cand1 * grid->n_cand2 * 4));
    if (blocks > cap) blocks = cap;
    if (blocks < 1) return OMSE_EINVAL;
    a.curve = reinterpret_cast<float*>(reinterpret_cast<char*>(ctx->partials) + point_bytes);
    a.evals = &ctx->ws->evals;
    if (bound) {
        omse::DualPoint* points = reinterpret_cast<omse::DualPoint*>(ctx->partials);
        omse::dual_points_kernel<<<(unsigned)grid->n_cand2, omse::kDualPoints, 0, ctx->stream>>>(points, grid->n_cand2, grid->hi_frac2, a.lo1,
                                                                                                 a.hi1, a.lo2, a.hi2);
        const omse::DualPoints pts = {points};
        if (few) omse::dual_bound_kernel<3><<<(unsigned)blocks, threads, smem, ctx->stream>>>(a, pts);
        else omse::dual_bound_kernel<4><<<(unsigned)blocks, threads, smem, ctx->stream>>>(a, pts);
        ctx->n_launches += 2;
    } else {
        omse::dual_kernel<<<(unsigned)blocks, threads, smem, ctx->stream>>>(a);
        ++ctx->n_launches;
    }
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

int omse_select_key_layers(omse_ctx* ctx, const omse_layer_error* layers, int n_layers, float tau, double* d_mse,
                           int32_t* d_is_key) {
    if (!ctx || n_layers < 0 || n_layers > OMSE_MAX_BATCH || (n_layers > 0 && (!layers || !d_mse)) || !(tau >= 0.f))
        return OMSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_mse) & 7) || misaligned4(d_is_key)) return OMSE_EINVAL;
    static_assert(sizeof(omse::LayerError) <= sizeof(omse::RowTensor), "descriptor buffer too small");
    std::vector<omse::LayerError> list((size_t)n_layers);
    for (int i = 0; i < n_layers; ++i) {
        if (!layers[i].d_sse || layers[i].n_kernels < 1 || layers[i].kernel_len < 1 || misaligned4(layers[i].d_sse))
            return OMSE_EINVAL;
        list[i].sse = layers[i].d_sse;
        list[i].n_kernels = layers[i].n_kernels;
        list[i].kernel_len = layers[i].kernel_len;
    }
    if (n_layers == 0) return OMSE_OK;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse::LayerError* d_layers = reinterpret_cast<omse::LayerError*>(ctx->d_tensors);
    if (cudaMemcpyAsync(d_layers, list.data(), sizeof(omse::LayerError) * list.size(), cudaMemcpyHostToDevice,
                        ctx->stream) != cudaSuccess)
        return OMSE_ECUDA;
    omse::layer_mse_kernel<<<(unsigned)n_layers, 256, 0, ctx->stream>>>(d_layers, tau, d_mse, d_is_key);
    ++ctx->n_launches;
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

double omse_compression_ratio(const int64_t* n_kernels, const int64_t* kernel_len, const int* bits, const int* n_tensors,
                              int n_layers) {
    if (!n_kernels || !kernel_len || !bits || !n_tensors || n_layers < 1) return -1.0;
    double q = 0.0, f = 0.0;
    for (int l = 0; l < n_layers; ++l) {
        if (n_kernels[l] < 0 || kernel_len[l] < 1 || bits[l] < 1 || n_tensors[l] < 1) return -1.0;
        const double n = (double)n_kernels[l] * (double)kernel_len[l];
        q += (double)n_tensors[l] * (n * (double)bits[l] + 32.0 * (double)n_kernels[l]);
        f += 32.0 * n;
    }
    return f > 0.0 ? q / f : -1.0;
}

int omse_activation_scale(omse_ctx* ctx, const float* d_x, int64_t n, int bits, int is_signed, const omse_grid* grid,
                          float* d_alpha, float* d_sse, int32_t* d_best_idx, double* d_sse_curve) {
    return activation_impl(ctx, d_x, n, bits, is_signed, grid, d_alpha, nullptr, d_sse, d_best_idx, d_sse_curve);
}

int omse_activation_scale_offset(omse_ctx* ctx, const float* d_x, int64_t n, int bits, const omse_grid* grid,
                                 float* d_alpha, float* d_delta, float* d_sse, int32_t* d_best_idx,
                                 double* d_sse_curve) {
    if (!d_delta || misaligned4(d_delta)) return OMSE_EINVAL;
    return activation_impl(ctx, d_x, n, bits, /*is_signed=*/0, grid, d_alpha, d_delta, d_sse, d_best_idx, d_sse_curve);
}

}  // extern "C"

static int activation_impl(omse_ctx* ctx, const float* d_x, int64_t n, int bits, int is_signed, const omse_grid* grid,
                           float* d_alpha, float* d_delta, float* d_sse, int32_t* d_best_idx, double* d_sse_curve) {
    if (!ctx || !grid_ok(grid) || bits < 2 || bits > 8 || n < 0 || !d_alpha || !d_sse) return OMSE_EINVAL;
    if (n > 0 && !d_x) return OMSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_x) & 15) || (reinterpret_cast<uintptr_t>(d_alpha) & 3) ||
        (reinterpret_cast<uintptr_t>(d_sse) & 3) || (reinterpret_cast<uintptr_t>(d_best_idx) & 3) ||
        (reinterpret_cast<uintptr_t>(d_sse_curve) & 7))
        return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    omse::TensorArgs a;
    memset(&a, 0, sizeof(a));
    a.x = d_x;
    a.n = n;
    a.n_cand = grid->n_cand;
    a.hi_frac = grid->hi_frac;
    bounds(bits, is_signed, &a.lo, &a.hi);
    a.st = &ctx->ws->tstate;
    a.partials = ctx->partials;
    a.partial_doubles = (long long)(kPartialBytes / 8);
    a.list = ctx->ws->list;
    a.near = ctx->ws->near;
    a.near_cap = kNearValues;
    a.curve = ctx->ws->curve;
    a.curve_out = d_sse_curve;
    a.alpha_out = d_alpha;
    a.sse_out = d_sse;
    a.idx_out = d_best_idx;
    a.delta_out = d_delta;
    a.evals = &ctx->ws->evals;
    a.status = &ctx->ws->status;
    const TensorEnv env = {ctx->n_sm, ctx->stream, &ctx->tensor, &ctx->n_launches};
    const int rc = enqueue_resident_search(env, a, &ctx->ws->exchange, ctx->search_blocks, ctx->poll_limit, grid->refine_iters);
    if (rc != OMSE_ELIMIT) return rc;
    omse::tensor_init_kernel<<<1, 32, 0, ctx->stream>>>(a.st);
    ++ctx->n_launches;
    return enqueue_tensor_search(env, a, grid->refine_iters);
}

extern "C" {

int omse_pack_int4(omse_ctx* ctx, const int8_t* d_codes, int64_t n, int is_signed, uint8_t* d_packed) {
    (void)is_signed;
    if (!ctx || n < 0) return OMSE_EINVAL;
    if (n == 0) return OMSE_OK;
    if (!d_codes || !d_packed) return OMSE_EINVAL;
    DeviceScope dev(ctx->device);
    if (!dev.ok()) return OMSE_ECUDA;
    long long grid = (n / 16 + 255) / 256;
    if (grid > (long long)ctx->n_sm * 16) grid = (long long)ctx->n_sm * 16;
    if (grid < 1) grid = 1;
    omse::pack_int4_kernel<<<(unsigned)grid, 256, 0, ctx->stream>>>(reinterpret_cast<const signed char*>(d_codes), n, d_packed);
    ++ctx->n_launches;
    return cudaGetLastError() == cudaSuccess ? OMSE_OK : OMSE_ECUDA;
}

}  // extern "C"

// -------------------------------------------------------------------------------------------------
// Allocation-free per-tensor search (omse_activation_scale_static).  The scratch that
// omse_activation_scale takes from the context workspace lives here in a fixed device array; every
// GPU that loads the library holds OMSE_STATIC_SCRATCH_BYTES of it until the process exits.
// -------------------------------------------------------------------------------------------------
namespace {

constexpr size_t kStaticPartialDoubles = 1u << 19;   // 4 MiB of per-block partial sums
constexpr int kStaticNear = 1024;                    // values next to an edge of a bin; more, and the polish starts with a look at the tensor

struct StaticScratch {
    unsigned int status;
    unsigned int pad_[3];
    omse::TensorState tstate;
    double curve[OMSE_STATIC_MAX_CANDIDATES];
    int list[OMSE_STATIC_MAX_CANDIDATES];
    float near[kStaticNear];
    double partials[kStaticPartialDoubles];
};
static_assert(sizeof(StaticScratch) <= OMSE_STATIC_SCRATCH_BYTES, "static scratch larger than documented");

// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_static_scratch[OMSE_STATIC_SCRATCH_BYTES];

struct StaticDevice {
    StaticScratch* ptr;   // device address of g_static_scratch on this device
    int n_sm;
    bool ready;
    TensorLaunches tensor;
};
StaticDevice g_static_dev[64];
std::mutex g_static_mutex;

// Everything that must start from zero: the array keeps the previous call's contents.
__global__ void static_begin_kernel(StaticScratch* s) {
    if (threadIdx.x == 0) {
        s->status = 0u;
        omse::tensor_state_init(&s->tstate);
    }
}

}  // namespace

extern "C" int omse_activation_scale_static(int device, void* cuda_stream, const float* d_x, int64_t n, int bits,
                                            int is_signed, const omse_grid* grid, float* d_alpha, float* d_sse,
                                            int32_t* d_best_idx, double* d_sse_curve, uint32_t* d_status) {
    if (!grid_ok(grid) || bits < 2 || bits > 8 || n < 0 || !d_alpha || !d_sse || device < 0 || device >= 64)
        return OMSE_EINVAL;
    if (grid->n_cand > OMSE_STATIC_MAX_CANDIDATES) return OMSE_ELIMIT;
    if (n > 0 && !d_x) return OMSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_x) & 15) || (reinterpret_cast<uintptr_t>(d_alpha) & 3) ||
        (reinterpret_cast<uintptr_t>(d_sse) & 3) || (reinterpret_cast<uintptr_t>(d_best_idx) & 3) ||
        (reinterpret_cast<uintptr_t>(d_sse_curve) & 7) || (reinterpret_cast<uintptr_t>(d_status) & 3))
        return OMSE_EINVAL;
    DeviceScope dev(device);
    if (!dev.ok()) return OMSE_ECUDA;
    StaticDevice& sd = g_static_dev[device];
    {
        // once per device, with that device current: the device address of the array
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!sd.ready) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return OMSE_ECUDA;
            if (cudaDeviceGetAttribute(&sd.n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return OMSE_ECUDA;
            sd.ptr = static_cast<StaticScratch*>(p);
            sd.ready = true;
        }
    }
    StaticScratch* sc = sd.ptr;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    omse::TensorArgs a;
    memset(&a, 0, sizeof(a));
    a.x = d_x;
    a.n = n;
    a.n_cand = grid->n_cand;
    a.hi_frac = grid->hi_frac;
    bounds(bits, is_signed, &a.lo, &a.hi);
    a.st = &sc->tstate;
    a.partials = sc->partials;
    a.partial_doubles = (long long)kStaticPartialDoubles;
    a.list = sc->list;
    a.near = sc->near;
    a.near_cap = kStaticNear;
    a.curve = sc->curve;
    a.curve_out = d_sse_curve;
    a.alpha_out = d_alpha;
    a.sse_out = d_sse;
    a.idx_out = d_best_idx;
    a.status = &sc->status;
    a.status_out = d_status;

    static_begin_kernel<<<1, 32, 0, s>>>(sc);
    unsigned long long not_counted = 0;
    const TensorEnv env = {sd.n_sm, s, &sd.tensor, &not_counted};
    return enqueue_tensor_search(env, a, grid->refine_iters);
}

