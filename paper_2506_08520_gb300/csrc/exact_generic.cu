// Generic exact window attention, Eq. (1): O = softmax(Q K^T / sqrt(d_h)) V,
// for any N <= 1024 and d_h <= 64, fp32 arithmetic with expf.
//
// One CTA (256 threads) per block of 64 query rows of a (window, head) unit (16
// rows and keys in windows of up to 16 tokens).
// Keys and values are staged in chunks of 64 tokens; a thread computes a 4 x 4
// tile of the chunk's scores and keeps it in registers through the row maximum
// (shuffles over the 16 lanes of a row) and the exponentials, P is stored once,
// and P V accumulates in 4 x 4 register tiles across the chunks, rescaled as
// the running maxima grow: the online form of the row softmax, which equals
// the max-shifted Eq. (2) up to rounding.  Products as in nystra_generic.cuh:
// packed FMAs on rows contiguous along the contraction (V transposed), row
// strides of an odd number of 16-byte granules.
//
// What bounds it: instruction issue (about a third of them packed FMAs).
// Measured against one thread per query row with the scores in shared memory:
// 600 units of 32x32 windows, d_h = 30, fp32 11.4 -> 3.5 ms; 3000 units of 12x12,
// bf16 1.9 -> 0.65 ms; 108 units of 10x10, d_h = 33, fp32 203 -> 27 us.
#include "simt.cuh"

namespace nystra {
namespace {

using namespace simt;

constexpr int kThreads = 256;
constexpr int kG = 16;  // score tiles per row and column: 16 x 16 threads

// TI: rows and columns of a thread's score tile, 4, or 1 for windows of up to 16
// tokens, most of whose 64 rows and keys would be padding (1000 units, d_h = 16: 4
// tokens 23.6 -> 12.0 us, with a thread per query row 20.3; 16 tokens 23.5 -> 12.1, 62).
// DS: row stride of d_h columns; c4: groups of four columns (at most kG, so that
// every thread has at most one tile of O).
template <int DS, int TI>
struct Shape {
    static constexpr int kRows = kG * TI;   // query rows per CTA, keys per chunk
    static constexpr int kNS = kRows + 4;   // row stride of anything with key columns
    static_assert(kG * kG == kThreads && (kNS / 4) % 2 == 1, "one score tile per thread");
    int c4;
    __host__ __device__ explicit Shape(int d) : c4((d + 3) / 4) {}
    __host__ __device__ size_t bytes() const {
        // Q rows | K rows or V^T | P | row factors
        const int kv = kRows * DS > 4 * c4 * kNS ? kRows * DS : 4 * c4 * kNS;
        return sizeof(float) * (size_t)(kRows * DS + kv + kRows * kNS + kRows);
    }
};

template <int DS, int TI, typename T>
__device__ __forceinline__ void run(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                    T* __restrict__ out, long long n_units, int N, int d, float scale, float* sm) {
    constexpr int kRows = Shape<DS, TI>::kRows, kNS = Shape<DS, TI>::kNS;
    const Shape<DS, TI> G(d);
    const int tid = threadIdx.x, c4 = G.c4, pl = 4 * c4 <= 16 ? 3 : (4 * c4 <= 32 ? 4 : 5);
    float* Qs = sm;                                                           // kRows rows
    float* KV = Qs + kRows * DS;                                              // K rows, then V^T
    float* P = KV + (kRows * DS > 4 * c4 * kNS ? kRows * DS : 4 * c4 * kNS);  // [row][key]
    float* fac = P + kRows * kNS;                                             // rescale factors, then 1 / denominators
    const int j0 = tid % kG, t0 = tid / kG;  // score tile: keys j0 + kG j, rows t0 + kG i
    // O tile: columns oc + c4 j (oc < c4), rows t0 + kG i; narrow heads leave
    // lanes over, which take a half or a quarter of the keys each
    const int wd = c4 <= 4 ? 4 : (c4 <= 8 ? 8 : kG), oc = j0 % wd, g0 = (j0 / wd) * wd;
    const int blocks = (N + kRows - 1) / kRows;

    for (long long w = blockIdx.x; w < n_units * blocks; w += gridDim.x) {
        const long long u = w / blocks;
        const int r0 = (int)(w - u * blocks) * kRows, nr = min(kRows, N - r0);
        const size_t base = (size_t)u * N * d;
        load_rows<T>(q + base + (size_t)r0 * d, nr, kRows / 4, d, 4 * c4, pl,
                     [&](int r, int c, float2 x) { *reinterpret_cast<float2*>(Qs + r * DS + c) = x; });
        float run_max[TI], den[TI], o[TI][4];
#pragma unroll
        for (int i = 0; i < TI; ++i) {
            run_max[i] = -INFINITY;
            den[i] = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) o[i][j] = 0.f;
        }
        for (int k0 = 0; k0 < N; k0 += kRows) {
            const int nt = min(kRows, N - k0);
            load_rows<T>(k + base + (size_t)k0 * d, nt, kRows / 4, d, 4 * c4, pl,
                         [&](int r, int c, float2 x) { *reinterpret_cast<float2*>(KV + r * DS + c) = x; });
            __syncthreads();
            f32x2 sacc[TI][TI];
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < TI; ++j) sacc[i][j] = 0ull;
            tile_nt<TI, TI>(Qs + t0 * DS, kG * DS, KV + j0 * DS, kG * DS, c4, sacc);
            float s[TI][TI];
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                float mx = run_max[i];
#pragma unroll
                for (int j = 0; j < TI; ++j) {
                    s[i][j] = j0 + kG * j < nt ? scale * sum2(sacc[i][j]) : -INFINITY;
                    mx = fmaxf(mx, s[i][j]);
                }
#pragma unroll
                for (int x = kG / 2; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
                const float f = run_max[i] == -INFINITY ? 0.f : expf(run_max[i] - mx);
                run_max[i] = mx;
                den[i] *= f;
#pragma unroll
                for (int j = 0; j < TI; ++j) {
                    const float p = j0 + kG * j < nt ? expf(s[i][j] - mx) : 0.f;
                    den[i] += p;
                    P[(t0 + kG * i) * kNS + j0 + kG * j] = p;
                }
                if (j0 == 0) fac[t0 + kG * i] = f;
            }
            __syncthreads();  // K has been read: V takes its place
            load_rows<T>(v + base + (size_t)k0 * d, nt, kRows / 4, d, 4 * c4, pl, [&](int r, int c, float2 x) {
                KV[c * kNS + r] = x.x;
                KV[(c + 1) * kNS + r] = x.y;
            });
            __syncthreads();
            if (oc < c4 && (TI == 4 || g0 == 0)) {  // (TI = 1: the 16 keys are one split)
                f32x2 acc[TI][4];
#pragma unroll
                for (int i = 0; i < TI; ++i) {
                    const float f = fac[t0 + kG * i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = __float_as_uint(o[i][j] * f);  // (o f, 0)
                }
                tile_nt<TI, 4>(P + t0 * kNS + 4 * g0, kG * kNS, KV + oc * kNS + 4 * g0, c4 * kNS,
                               TI == 4 ? wd : kRows / 4, acc);
#pragma unroll
                for (int i = 0; i < TI; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) o[i][j] = sum2(acc[i][j]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < TI; ++i) {
#pragma unroll
            for (int x = kG / 2; x > 0; x >>= 1) den[i] += __shfl_xor_sync(0xffffffffu, den[i], x);
            if (j0 == 0) fac[t0 + kG * i] = 1.f / den[i];
        }
        __syncthreads();
        for (int x = wd; x < kG; x <<= 1)  // the splits' sums
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) o[i][j] += __shfl_xor_sync(0xffffffffu, o[i][j], x);
        if (oc < c4 && g0 == 0) {  // O over the Q rows, then out in row order
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    Qs[(t0 + kG * i) * DS + oc + c4 * j] = o[i][j] * fac[t0 + kG * i];
        }
        __syncthreads();
        {
            const int c = 2 * (tid & ((1 << pl) - 1));
            if (c < d)
                for (int r = tid >> pl; r < nr; r += kThreads >> pl)
                    st_pair<T>(out + base + (size_t)(r0 + r) * d, c, d, Qs[r * DS + c], Qs[r * DS + c + 1]);
        }
        __syncthreads();
    }
}

template <int DS, int TI>
__global__ void __launch_bounds__(kThreads, 2)
exact_generic_kernel(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d,
                     int dtype, float scale) {
    extern __shared__ __align__(16) float sm[];
    if (dtype == 0)
        run<DS, TI, float>((const float*)q, (const float*)k, (const float*)v, (float*)out, n_units, N, d, scale, sm);
    else if (dtype == 1)
        run<DS, TI, __nv_bfloat16>((const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                               (__nv_bfloat16*)out, n_units, N, d, scale, sm);
    else
        run<DS, TI, __half>((const __half*)q, (const __half*)k, (const __half*)v, (__half*)out, n_units, N, d, scale, sm);
}

template <int DS, int TI>
cudaError_t launch_ds(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d,
                      int dtype, cudaStream_t stream) {
    static std::atomic<int> s_ready[kMaxDevices];
    auto kern = exact_generic_kernel<DS, TI>;
    if (cudaError_t e = opt_in_smem(kern, s_ready); e != cudaSuccess) return e;
    constexpr int kRows = Shape<DS, TI>::kRows;
    const long long want = n_units * ((N + kRows - 1) / kRows);
    const long long grid = want < (1LL << 30) ? want : (1LL << 30);
    kern<<<(unsigned)grid, kThreads, Shape<DS, TI>(d).bytes(), stream>>>(q, k, v, out, n_units, N, d, dtype,
                                                                      1.0f / sqrtf((float)d));
    return cudaGetLastError();
}

template <int DS>
cudaError_t launch_n(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d,
                     int dtype, cudaStream_t stream) {
    if (N <= kG) return launch_ds<DS, 1>(q, k, v, out, n_units, N, d, dtype, stream);
    return launch_ds<DS, 4>(q, k, v, out, n_units, N, d, dtype, stream);
}

}  // namespace
}  // namespace nystra

namespace nystra_host {
// Row strides: d_h columns padded to whole granules, an odd number of them.
cudaError_t launch_exact_generic(const void* q, const void* k, const void* v, void* out, long long n_units, int N,
                                 int d, int dtype, cudaStream_t stream) {
    using namespace nystra;
    if (d <= 20) return launch_n<20>(q, k, v, out, n_units, N, d, dtype, stream);
    if (d <= 36) return launch_n<36>(q, k, v, out, n_units, N, d, dtype, stream);
    return launch_n<68>(q, k, v, out, n_units, N, d, dtype, stream);
}
}  // namespace nystra_host
