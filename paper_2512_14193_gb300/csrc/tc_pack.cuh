// Operand packs of the tensor-core products (gemm_tc.cu): a row of K entries is, per 32 of them, 32 FP16 hi parts
// and their 32 lo parts, of the entries times a power of two of the row.
#pragma once
#include "common.cuh"

#include <cuda_fp16.h>

// 2^e, e clamped to the normal range
__device__ __forceinline__ float tc_pow2(int e) { return __int_as_float((min(max(e, -126), 127) + 127) << 23); }

// The scale 2^(15 - ex) of a row whose largest |Re| or |Im| is mx < 2^ex.  Zero and non-finite rows take ex = 0
// (infinities and NaN stay what they are); ex stops at -111, so that the scale and its inverse are normal numbers
// (a row below 2^-112 still keeps its 22 bits down to FP32's own limit).
struct TcRowScale {
    float f;
    int ex;
    __device__ __forceinline__ explicit TcRowScale(float mx) {
        ex = 0;
        if (mx > 0.f && mx < __int_as_float(0x7f800000)) ex = max((__float_as_int(mx) >> 23) - 126, -111);
        f = tc_pow2(15 - ex);
    }
    __device__ __forceinline__ float operator()(float v) const { return v * f; }
};
// 2^e for any e, as exact factors f g (one may not reach)
struct TcExpScale {
    float f, g;
    __device__ __forceinline__ explicit TcExpScale(int e) : f(tc_pow2(e >> 1)), g(tc_pow2(e - (e >> 1))) {}
    __device__ __forceinline__ float operator()(float v) const { return v * f * g; }
};

__device__ __forceinline__ long tc_pos(long k) { return (k >> 5) * 64 + (k & 31); }  // hi part of entry k; lo: + 32

// entry v (scaled) as hi and lo
__device__ __forceinline__ void tc_split(float v, __half& hi, __half& lo) {
    hi = __float2half_rn(v);
    lo = __float2half_rn(v - __half2float(hi));
}

// One row of K entries get(k) (zeros up to the next multiple of 32) by a CTA of TC_PACK_THREADS threads, and its
// exponent e: the entries are the packed numbers times 2^e.  Two passes over the entries: the maximum, the pack.
constexpr int TC_PACK_THREADS = 256;
template <class G>
__device__ __forceinline__ void tc_pack_column(const G& get, int K, __half* __restrict__ Pr, __half* __restrict__ Pi,
                                               int* __restrict__ e) {
    __shared__ float part[TC_PACK_THREADS / 32];
    const int t = threadIdx.x;
    float mx = 0.f;
#pragma unroll 8
    for (int k = t; k < K; k += TC_PACK_THREADS) {
        const float2 v = get(k);
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((t & 31) == 0) part[t >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < TC_PACK_THREADS / 32; ++w) mx = fmaxf(mx, part[w]);
    const TcRowScale sc(mx);
    if (t == 0) *e = sc.ex - 15;
    const int kp = (K + 31) & ~31;
#pragma unroll 4
    for (int k = 2 * t; k < kp; k += 2 * TC_PACK_THREADS) {  // a pair of entries, 4-byte stores
        const float2 z = make_float2(0.f, 0.f), a = k < K ? get(k) : z, b = k + 1 < K ? get(k + 1) : z;
        __half2 hr, lr, hi, li;
        tc_split(sc(a.x), hr.x, lr.x);
        tc_split(sc(b.x), hr.y, lr.y);
        tc_split(sc(a.y), hi.x, li.x);
        tc_split(sc(b.y), hi.y, li.y);
        const long o = tc_pos(k);
        *reinterpret_cast<__half2*>(Pr + o) = hr;
        *reinterpret_cast<__half2*>(Pr + o + 32) = lr;
        *reinterpret_cast<__half2*>(Pi + o) = hi;
        *reinterpret_cast<__half2*>(Pi + o + 32) = li;
    }
}
