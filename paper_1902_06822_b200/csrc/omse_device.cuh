// Device-side building blocks of the MMSE scale search for sm_100a.
//
// Section 3.4 of the paper reduces the constrained MSE problem to a one-dimensional search over the
// scale alpha, the codes being [T_i/alpha]_Zp.  Where the squared error at a scale is evaluated value by value (short rows),
// the inner loop is pure FP32 arithmetic,
//     t = x*inv_alpha + M       (M = 1.5*2^23: the add rounds to the nearest integer, ties to even)
//     t = min(max(t, M+lo), M+hi)            only for candidates that can saturate on this tensor
//     q = t - M ;  e = x - alpha*q ;  acc += e*e
// written with Blackwell's packed fma.rn.f32x2 / add.rn.f32x2 on two elements at a time.  inv_alpha is within 2 ulp of
// 1/alpha: a code can differ from the divided one only where both neighbours give the same error to ~1e-7, and the winners
// are re-scored with true division afterwards.
#pragma once
#include <cfloat>
#include <cstdint>
#include <cuda_runtime.h>

namespace omse {

typedef unsigned long long u64;

constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23
constexpr int kFlushEvery4 = 32;        // float4 loads between folds of fp32 partial sums
constexpr double kRescoreBand = 4e-6;   // candidates within this relative band of the fp32 minimum are re-scored

__device__ __forceinline__ u64 pack2(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// [x/alpha]_Zp exactly as Section 3.1 writes it: IEEE division, round to nearest even, saturate.
__device__ __forceinline__ int code_of(float x, float alpha, float flo, float fhi) {
    float r = rintf(__fdiv_rn(x, alpha));
    r = fminf(fmaxf(r, flo), fhi);
    return (int)r;
}

// [x/alpha]_Zp without a division on the common path.  t = fl(x*inv + M) rounds the exact product to the nearest
// integer (ties to even); with inv = fl(1/alpha) the product is within 2^-24 relative of x/alpha, and so is the IEEE
// quotient, so both round to the same integer unless the product lies within (|integer| + 1) * 2^-21 of a
// half-integer.  Integers beyond the range by more than one saturate either way, so the test only has to hold for
// |integer| <= range + 1: amb_thr = 1/2 - (range + 2) * 2^-21 serves every element; `ambiguous` reports a product
// closer to a half-integer than that (or too large to be rounded by the addition), and the caller then takes the
// division.  Returns M + code (the code sits in the low mantissa bits).
__device__ __forceinline__ float magic_code(float x, float inv, float clo, float chi, float amb_thr, bool& ambiguous) {
    const float t = fmaf(x, inv, kMagic);
    const float rq = t - kMagic;
    const float delta = fmaf(x, inv, -rq);
    ambiguous = !(fabsf(delta) <= amb_thr);
    return fminf(fmaxf(t, clo), chi);
}

// integer held by M + q as an int, and as a double without a conversion instruction
__device__ __forceinline__ int magic_int(float tc) { return __float_as_int(tc) - 0x4B400000; }
__device__ __forceinline__ double int_double(int q) {
    return __hiloint2double(0x43380000 + (q >> 31), q) - 6755399441055744.0;   // (1.5*2^52 + q) - 1.5*2^52, exact
}

// The code of x at scale alpha (inv = fl(1/alpha)) as an int, equal to code_of(x, alpha, flo, fhi) bit for bit.
__device__ __forceinline__ int exact_code(float x, float alpha, float inv, float flo, float fhi, float amb_thr) {
    bool amb;
    const float tc = magic_code(x, inv, kMagic + flo, kMagic + fhi, amb_thr, amb);
    return amb ? code_of(x, alpha, flo, fhi) : magic_int(tc);   // rare: the division decides
}
__device__ __forceinline__ float ambiguity_threshold(float flo, float fhi) {
    return 0.5f - (fmaxf(fhi, -flo) + 2.0f) * 4.76837158203125e-7f;
}
// Four codes at once: one branch for the rare division instead of four.
__device__ __forceinline__ void exact_codes4(const float (&x)[4], float alpha, float inv, float flo, float fhi, float amb_thr,
                                             int (&q)[4]) {
    bool amb[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) q[e] = magic_int(magic_code(x[e], inv, kMagic + flo, kMagic + fhi, amb_thr, amb[e]));
    if (amb[0] || amb[1] || amb[2] || amb[3]) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (amb[e]) q[e] = code_of(x[e], alpha, flo, fhi);
    }
}
// M + q (q an integer above -2^22) as a double that holds q: the bits are the low word of a double in [2^52, 2^53).
__device__ __forceinline__ double magic_double(float tc) {
    return __hiloint2double(0x43300000, __float_as_int(tc)) - (4503599627370496.0 + 1262485504.0);   // 2^52 + the bits of M, exact
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {     // NaN if one of them is
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// The codes of four values at a scale, as M + code: those of code_of, by the argument at magic_code, with one branch for the rare
// divisions; in packed arithmetic and with one test (a pass over rows in shared memory, 24 warps per SM: 5.9 clocks per 32 values
// with exact_codes4, 4.8 so; in the rolled loops over a few values per lane that short rows have, it costs 1 % more than it saves).
struct Coder {
    u64 inv2;
    float alpha, flo, fhi, thr;
    __device__ __forceinline__ Coder(float alpha_, float inv, float flo_, float fhi_)
        : inv2(pack2(inv, inv)), alpha(alpha_), flo(flo_), fhi(fhi_), thr(ambiguity_threshold(flo_, fhi_)) {}
    __device__ __forceinline__ void of(const float4& v, float (&t)[4]) const {
        const u64 M2 = pack2(kMagic, kMagic), minus = pack2(-1.0f, -1.0f), xa = pack2(v.x, v.y), xb = pack2(v.z, v.w);
        const u64 ta = fma2(xa, inv2, M2), tb = fma2(xb, inv2, M2);
        float d0, d1, d2, d3;
        unpack2(fma2(xa, inv2, fma2(ta, minus, M2)), d0, d1);              // the product less the integer that it was rounded to
        unpack2(fma2(xb, inv2, fma2(tb, minus, M2)), d2, d3);
        unpack2(ta, t[0], t[1]);
        unpack2(tb, t[2], t[3]);
        const float clo = kMagic + flo, chi = kMagic + fhi;
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] = fminf(fmaxf(t[e], clo), chi);
        if (!(max3_nan(max3_nan(fabsf(d0), fabsf(d1), fabsf(d2)), fabsf(d3), 0.f) <= thr)) {
            const float x[4] = {v.x, v.y, v.z, v.w}, d[4] = {d0, d1, d2, d3};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (!(fabsf(d[e]) <= thr)) t[e] = kMagic + (float)code_of(x[e], alpha, flo, fhi);
        }
    }
};
// sums of q*q over pairs of codes M + q, in binary32: exact below 2^24, so for 258 pairs of squares of up to 255^2
constexpr int kSquareSteps = 258;
static_assert(kSquareSteps * 255 * 255 < 1 << 24, "sums of squared codes stay exact in binary32");
__device__ __forceinline__ u64 add_squares(float t0, float t1, u64 acc) {
    const u64 q = add2(pack2(t0, t1), pack2(-kMagic, -kMagic));
    return fma2(q, q, acc);
}
__device__ __forceinline__ long long squares_of(u64 a, u64 b) {
    float v[4];
    unpack2(a, v[0], v[1]);
    unpack2(b, v[2], v[3]);
    return (long long)(int)v[0] + (int)v[1] + (int)v[2] + (int)v[3];
}
// four codes M + q as bytes; bytes as nibbles
__device__ __forceinline__ unsigned int code_bytes(const float (&t)[4]) {
    const unsigned int a = __byte_perm(__float_as_uint(t[0]), __float_as_uint(t[1]), 0x0040),
                       b = __byte_perm(__float_as_uint(t[2]), __float_as_uint(t[3]), 0x0040);
    return __byte_perm(a, b, 0x5410);
}
__device__ __forceinline__ unsigned int byte_nibbles(unsigned int v) {
    const unsigned int w = (v & 0x0f0f0f0fu) | ((v >> 4) & 0x00f000f0u);       // bytes 0 and 2 hold two codes each
    return __byte_perm(w, 0u, 0x4420);
}
// Asynchronous copies of 16 and of 4 bytes from global to shared memory; the caller waits for them (cp_async_wait).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned int)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned int)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// Block-wide reductions (fixed order: lanes by shuffle tree, warps in index order) so that results
// do not depend on scheduling.  `scratch` holds at least 2*32 doubles.  All threads get the result.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// smallest power of two that is not below n (n <= 32): groups of so many lanes each hold one item per warp of the block
__device__ __forceinline__ int group_lanes(int n) { return n <= 1 ? 1 : 1 << (32 - __clz(n - 1)); }

// sums a double and a 64-bit integer over the block (at most 1024 threads).  The warps' sums are added by every warp for
// itself, by a shuffle tree again: a loop over 32 of them is a chain of as many dependent additions.
__device__ __forceinline__ void block_sum2(double& d, long long& q, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
    d = warp_sum(d);
    q = warp_sum(q);
    long long* qs = reinterpret_cast<long long*>(scratch + 32);
    __syncthreads();
    if (lane == 0) {
        scratch[warp] = d;
        qs[warp] = q;
    }
    __syncthreads();
    const int l = lane & (group_lanes(nwarp) - 1);
    d = l < nwarp ? scratch[l] : 0.0;
    q = l < nwarp ? qs[l] : 0ll;
    for (int o = 1; o < nwarp; o <<= 1) {          // (all lanes end with the same bits: a + b == b + a)
        d += __shfl_xor_sync(0xffffffffu, d, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
}

__device__ __forceinline__ void block_max(float& a, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_down_sync(0xffffffffu, a, o));
    float* fs = reinterpret_cast<float*>(scratch);
    __syncthreads();
    if (lane == 0) fs[warp] = a;
    __syncthreads();
    a = fs[0];
    for (int w = 1; w < nwarp; ++w) a = fmaxf(a, fs[w]);
}

__device__ __forceinline__ void block_max2(float& a, float& b, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = fmaxf(a, __shfl_down_sync(0xffffffffu, a, o));
        b = fmaxf(b, __shfl_down_sync(0xffffffffu, b, o));
    }
    float* fs = reinterpret_cast<float*>(scratch);
    __syncthreads();
    if (lane == 0) {
        fs[warp] = a;
        fs[32 + warp] = b;
    }
    __syncthreads();
    float ta = 0.f, tb = 0.f;
    for (int w = 0; w < nwarp; ++w) {
        ta = fmaxf(ta, fs[w]);
        tb = fmaxf(tb, fs[32 + w]);
    }
    a = ta;
    b = tb;
}

// lexicographic minimum of (value, index) over the block
__device__ __forceinline__ void block_argmin(double& v, int& idx, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_down_sync(0xffffffffu, v, o);
        const int oi = __shfl_down_sync(0xffffffffu, idx, o);
        if (ov < v || (ov == v && oi < idx)) {
            v = ov;
            idx = oi;
        }
    }
    int* is = reinterpret_cast<int*>(scratch + 32);
    __syncthreads();
    if (lane == 0) {
        scratch[warp] = v;
        is[warp] = idx;
    }
    __syncthreads();
    const int l = lane & (group_lanes(nwarp) - 1);
    double bv = l < nwarp ? scratch[l] : INFINITY;
    int bi = l < nwarp ? is[l] : 0x7fffffff;
    for (int o = 1; o < nwarp; o <<= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov < bv || (ov == bv && oi < bi)) {
            bv = ov;
            bi = oi;
        }
    }
    v = bv;
    idx = bi;
}

// The same for values that are not negative (Inf among them): they order like their bit patterns, and a reduction instruction for each
// half of them and one for the index replaces five exchanges of a double and an index.
__device__ __forceinline__ void warp_argmin_error(double& v, int& idx) {
    const unsigned int hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned int least = __reduce_min_sync(0xffffffffu, hi), low = __reduce_min_sync(0xffffffffu, hi == least ? lo : 0xffffffffu);
    idx = __reduce_min_sync(0xffffffffu, hi == least && lo == low ? idx : 0x7fffffff);
    v = __hiloint2double((int)least, (int)low);
}
__device__ __forceinline__ void block_argmin_error(double& v, int& idx, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
    int* is = reinterpret_cast<int*>(scratch + 32);
    warp_argmin_error(v, idx);
    __syncthreads();
    if (lane == 0) {
        scratch[warp] = v;
        is[warp] = idx;
    }
    __syncthreads();
    v = lane < nwarp ? scratch[lane] : INFINITY;
    idx = lane < nwarp ? is[lane] : 0x7fffffff;
    warp_argmin_error(v, idx);
}

// Adds this thread's count of executed (element, candidate) evaluations to a global counter: one atomic per warp.
__device__ __forceinline__ void report_evaluations(unsigned long long* counter, unsigned long long mine) {
    if (!counter) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(counter, mine);
}

// Register-only loop of independent packed multiply-adds: measures the FP32 lane-operation rate of the FMA pipe,
// the roof the candidate sweep is compared with.  Every thread runs kPeakChains chains of fma.rn.f32x2.
constexpr int kPeakChains = 8;
__global__ void __launch_bounds__(256) fma_peak_kernel(float* __restrict__ out, int iters, float seed) {
    u64 v[kPeakChains];
#pragma unroll
    for (int s = 0; s < kPeakChains; ++s) v[s] = pack2(seed + 1e-3f * (float)(threadIdx.x + s), seed - 1e-3f * (float)s);
    const u64 m = pack2(0.9999999f, 1.0000001f), c = pack2(1e-7f, -1e-7f);
#pragma unroll 16   // long straight-line stretches: with a short body the loop bookkeeping costs ~8 % of the rate
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int s = 0; s < kPeakChains; ++s) v[s] = fma2(v[s], m, c);
    }
    float r = 0.f;
#pragma unroll
    for (int s = 0; s < kPeakChains; ++s) {
        float a, b;
        unpack2(v[s], a, b);
        r += a + b;
    }
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = r;
}

}  // namespace omse
