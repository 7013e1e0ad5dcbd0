// What the fp32 SIMT kernels (nystra_generic.cuh, exact_generic.cu) share:
// packed-FMA register tiles of A B^T and the staging of token rows.
#pragma once

#include "common.cuh"

namespace nystra {
namespace simt {

constexpr size_t kSmemLimit = 232448;  // opt-in dynamic shared memory per CTA

// Opts `kern` in to kSmemLimit once per device; `cache` is a zero-initialised
// static of the launcher that keeps the device's number of SMs, returned in *sms.
template <typename K>
cudaError_t opt_in_smem(K kern, std::atomic<int> (&cache)[kMaxDevices], int* sms = nullptr) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        cache[dev].store(n, std::memory_order_relaxed);
    }
    if (sms) *sms = n;
    return cudaSuccess;
}

// ---- A B^T register tiles ----
using f32x2 = unsigned long long;
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum2(f32x2 x) {
    return __uint_as_float((unsigned)x) + __uint_as_float((unsigned)(x >> 32));
}

// acc[i][j] += a_i . b_j over 4 kg values, a_i = a + i * as, b_j = b + j * bs.
template <int TI, int TJ, int KU = 1>
__device__ __forceinline__ void tile_nt(const float* a, int as, const float* b, int bs, int kg, f32x2 (&acc)[TI][TJ]) {
#pragma unroll KU
    for (int k = 0; k < kg; ++k) {
        ulonglong2 x[TI], y[TJ];
#pragma unroll
        for (int i = 0; i < TI; ++i) x[i] = *reinterpret_cast<const ulonglong2*>(a + i * as);
#pragma unroll
        for (int j = 0; j < TJ; ++j) y[j] = *reinterpret_cast<const ulonglong2*>(b + j * bs);
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TJ; ++j) fma2(acc[i][j], x[i].x, y[j].x);
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TJ; ++j) fma2(acc[i][j], x[i].y, y[j].y);
        a += 4;
        b += 4;
    }
}

// ---- token rows in and out ----
// Columns c, c + 1 (c even) of a row at p.  Rows of an even d start at an even
// element of a 16-byte aligned tensor, so a pair is aligned; an odd d takes
// single elements (the second one, at c1, is c itself in the last column).
template <typename T, bool EVEN>
__device__ __forceinline__ float2 ld_pair(const T* p, int c1) {
    if constexpr (!EVEN) return make_float2(ldg_f32(p), ldg_f32(p + c1));
    else if constexpr (sizeof(T) == 4) return __ldg(reinterpret_cast<const float2*>(p));
    else {
        const unsigned x = __ldg(reinterpret_cast<const unsigned*>(p));
        const T* h = reinterpret_cast<const T*>(&x);
        return make_float2(to_f32(h[0]), to_f32(h[1]));
    }
}
template <typename T>
__device__ __forceinline__ void st_pair(T* p, int c, int d, float x, float y) {
    if ((d & 1) != 0) {
        p[c] = from_f32<T>(x);
        if (c + 1 < d) p[c + 1] = from_f32<T>(y);
    } else if constexpr (sizeof(T) == 4)
        *reinterpret_cast<float2*>(p + c) = make_float2(x, y);
    else {
        unsigned u;
        T* h = reinterpret_cast<T*>(&u);
        h[0] = from_f32<T>(x);
        h[1] = from_f32<T>(y);
        *reinterpret_cast<unsigned*>(p + c) = u;
    }
}

// Rows 0 .. 4 tg - 1 of a chunk, 2^pl lanes per row, one pair of columns each:
// put(row, column, values), zeros beyond the nt tokens and the d columns up to
// `cols`.  Addresses beyond the chunk are moved into it (and the values
// dropped), so the loads of a batch are in flight together.
template <typename T, bool EVEN, typename Put>
__device__ __forceinline__ void load_rows_as(const T* __restrict__ src, int nt, int tg, int d, int cols, int pl,
                                             Put put) {
    const int c = 2 * (threadIdx.x & ((1 << pl) - 1)), step = blockDim.x >> pl, r00 = threadIdx.x >> pl;
    if (c >= cols) return;
    constexpr int U = 8;
    const T* p = src + (c < d ? c : 0);
    const int c1 = c + 1 < d ? 1 : 0;
    for (int r0 = r00; r0 < 4 * tg; r0 += U * step) {
        float2 x[U];
#pragma unroll
        for (int k = 0; k < U; ++k) x[k] = ld_pair<T, EVEN>(p + min(r0 + k * step, nt - 1) * d, c1);
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int r = r0 + k * step;
            const bool in = r < nt;
            if (r < 4 * tg) put(r, c, make_float2(in && c < d ? x[k].x : 0.f, in && c + 1 < d ? x[k].y : 0.f));
        }
    }
}
template <typename T, typename Put>
__device__ __forceinline__ void load_rows(const T* __restrict__ src, int nt, int tg, int d, int cols, int pl, Put put) {
    if ((d & 1) == 0) load_rows_as<T, true>(src, nt, tg, d, cols, pl, put);
    else load_rows_as<T, false>(src, nt, tg, d, cols, pl, put);
}

}  // namespace simt
}  // namespace nystra
