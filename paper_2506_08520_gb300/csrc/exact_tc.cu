// Tensor-core exact window attention, Eq. 1: O = softmax(Q K^T / sqrt(d_h)) V,
// even d_h <= 32; 16-bit I/O for windows of N = 64, 256 or 1024 tokens, fp32
// I/O (split bf16 operands, three MMAs per product) for N = 64 and 256.
//
// A group of WPU = N/64 warps processes one (window, head) unit.  Its K and V
// are laid out in shared memory in rows of 40 16-bit values (fp32: a hi and a
// lo plane), padded with zeros and, in V, a ones column, so that every B
// fragment comes from ldmatrix without bank conflicts (rows of 60 bytes, as
// they lie in HBM, take a 4-byte load and, for V, an 8x8 transpose per
// register, with two-way conflicts).  Warp r computes output rows 64r .. 64r +
// 63, 32 at a time so that a fragment serves two 16-row tiles, streaming the
// keys in chunks of 64 with the online (running-max) softmax: S = Q K_c^T
// (mma.sync, fp32 accumulate), P = exp(S - m) in registers fed directly as the
// A operand of P [V_c | 1], whose last column accumulates the row sums of the
// same rounded P.  P is rounded to 16 bits relative to the maximum so far, so
// the chunk length is part of the result (32 keys at a time move it by 1.4e-3
// in bf16, at the same distance of 2.1e-3 from float64).  Scores are scaled by
// log2(e)/sqrt(d_h) so each exponential is half a packed FMA and one ex2.  This
// is the computation PnP-Nystra replaces; it is the in-library comparator.
//
// What bounds it: at 32x32 windows the tensor pipe, 61% busy (32 MMAs and 32
// ex2 per warp for 32 rows and 32 keys); at 16x16 windows (53%) also laying out
// K and V, at 8x8 windows HBM.  The next unit's rows are brought to L2 meanwhile.
// Measured (d_h = 30, bf16) against fragments loaded from 60-byte rows by one
// 16-row tile: 5520 units of 32x32 windows 3.34 -> 2.02 ms, 6144 of 16x16
// 271 -> 176 us, 86400 of 8x8 269 -> 224 us; fp32, 2000 units of 16x16: 502 ->
// 163 us.
#include "common.cuh"
#include "ptx.cuh"

#include <type_traits>

namespace nystra {
namespace {

constexpr size_t kSmemLimit = 232448;
constexpr int kRow = 40;  // 16-bit values per staged row: 80 bytes, an odd number of granules

template <typename T>
struct ExactOp {  // 16-bit I/O: one plane
    using E = T;
    static constexpr int NP = 1;
    // per SM: the scores of 32 rows and 64 keys take twelve warps' registers
    // (160 of up to 168; 128 of sixteen warps spill up to 156 bytes: 6144 units of
    // 16x16 windows 201 us, d_h = 32 240, against 179 and 192); the sixteen warps
    // of a 32x32 window have 128, and at 8x8 windows with d_h read at run time
    // sixteen (124 registers) are faster, laying out K and V being most of the work
    // (40000 units, d_h = 24, 103 against 117 us; d_h = 30, compiled in, 267 against 220
    // with twelve for 86400 units)
    static constexpr int warps(int wpu, int dc) { return wpu == 16 || (wpu == 1 && dc == 0) ? 16 : 12; }
};
template <>
struct ExactOp<float> {
    using E = __nv_bfloat16;
    static constexpr int NP = 2;
    static constexpr int warps(int, int) { return 8; }
};

template <typename T, int WPU, int DC>
struct ExactLayout {
    static constexpr int N = 64 * WPU;
    static constexpr size_t PLANE = (size_t)N * kRow * 2;
    static constexpr size_t GROUP = 2 * ExactOp<T>::NP * PLANE;  // K, then V
    static constexpr int by_smem = (int)(kSmemLimit / GROUP);
    static constexpr int by_warps = ExactOp<T>::warps(WPU, DC) / WPU;
    static constexpr int GROUPS = by_smem < by_warps ? by_smem : by_warps;
    static_assert(GROUPS >= 1, "does not fit");
};

// Two elements at p as an operand register (fp32: a split pair).
__device__ __forceinline__ uint32_t ld_global2(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const unsigned*>(p)); }
__device__ __forceinline__ uint32_t ld_global2(const __half* p) { return __ldg(reinterpret_cast<const unsigned*>(p)); }
__device__ __forceinline__ RegPair ld_global2(const float* p) {
    const float2 x = __ldg(reinterpret_cast<const float2*>(p));
    return Opnd<float>::pk(x.x, x.y);
}
// Four elements at p, and their operand registers 0 and 1.
__device__ __forceinline__ uint2 ld_global4(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint2*>(p)); }
__device__ __forceinline__ uint2 ld_global4(const __half* p) { return __ldg(reinterpret_cast<const uint2*>(p)); }
__device__ __forceinline__ float4 ld_global4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ uint32_t word(uint2 x, int i) { return i ? x.y : x.x; }
__device__ __forceinline__ RegPair word(float4 x, int i) { return i ? Opnd<float>::pk(x.z, x.w) : Opnd<float>::pk(x.x, x.y); }
__device__ __forceinline__ void st_plane(unsigned char* p, size_t, uint32_t x) { *reinterpret_cast<uint32_t*>(p) = x; }
__device__ __forceinline__ void st_plane(unsigned char* p, size_t plane, RegPair x) {
    *reinterpret_cast<uint32_t*>(p) = x.hi;
    *reinterpret_cast<uint32_t*>(p + plane) = x.lo;
}

// ldmatrix x4 (TR: transposed) as operand registers.
template <bool TR>
__device__ __forceinline__ void ld_frag(uint32_t (&r)[4], const unsigned char* p, size_t) {
    if (TR) ldsm_x4_t(r, p);
    else ldsm_x4(r, p);
}
template <bool TR>
__device__ __forceinline__ void ld_frag(RegPair (&r)[4], const unsigned char* p, size_t plane) {
    uint32_t h[4], l[4];
    ld_frag<TR>(h, p, 0);
    ld_frag<TR>(l, p + plane, 0);
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = {h[i], l[i]};
}

template <typename T, int NCOL, int WPU, int DC>
__global__ void __launch_bounds__(ExactLayout<T, WPU, DC>::GROUPS * WPU * 32, 1)
exact_tc_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ out,
                long long n_units, int d_in, float sl2) {
    using Lay = ExactLayout<T, WPU, DC>;
    using O = Opnd<T>;
    using R = typename O::Reg;
    constexpr int N = Lay::N, NTO = NCOL / 8;
    const int groups = blockDim.x / (WPU * 32);
    constexpr size_t PL = Lay::PLANE;
    const int d = DC ? DC : d_in, h = d >> 1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp / WPU, r = warp - grp * WPU, id = r * 32 + lane;
    const int g = lane >> 2, t = lane & 3;
    unsigned char* Ks = smem_raw + (size_t)grp * Lay::GROUP;
    unsigned char* Vs = Ks + ExactOp<T>::NP * PL;
    auto gsync = [&]() {
        if constexpr (WPU == 1) __syncwarp();
        else named_barrier(1 + grp, WPU * 32);
    };
    // columns d .. 31: zeros, in V a ones column first (d = 32 has it as a constant
    // fragment); the columns from 32 on are never read
    for (int row = id; row < N; row += WPU * 32)
        for (int c = h; c < 16; ++c) {
            st_plane(Ks + (row * kRow + 2 * c) * 2, PL, O::zero());
            st_plane(Vs + (row * kRow + 2 * c) * 2, PL, c == h ? O::one() : O::zero());
        }
    // fragment addresses: rows 8 (lane / 8) .. of an ldmatrix x4
    const unsigned char* kf = Ks + ((lane & 7) * kRow + 8 * (lane >> 3)) * 2;                              // 8 keys x 32
    const unsigned char* vf = Vs + (((lane & 7) + 8 * ((lane >> 3) & 1)) * kRow + 8 * (lane >> 4)) * 2;  // 16 keys x 16
    R one0;  // B fragment of the ones column at d = 32: column 0 (lanes g = 0) is 1
    if constexpr (NCOL > 32) one0 = g == 0 ? O::pk(1.f, 1.f) : O::zero();
    // i / h for i < 2^14 and 2 <= h <= 16 (2^32 / h rounded up errs by less than i h / 2^32 < 1 / h)
    const uint32_t magic = DC ? 0u : 0xffffffffu / (uint32_t)h + 1u;
    auto row_of = [&](int i) { return DC ? i / h : h == 1 ? i : (int)__umulhi((uint32_t)i, magic); };
    const int jd = d >> 3, src = (lane & ~3) | ((d & 7) >> 1);

    for (long long u = (long long)blockIdx.x * groups + grp; u < n_units; u += (long long)gridDim.x * groups) {
        const size_t base = (size_t)u * N * d;
        const long long un = u + (long long)gridDim.x * groups;
        if (id == 0 && un < n_units) {  // the next unit's rows on their way to L2
            const size_t nb = (size_t)un * N * d;
            const uint32_t bytes = (uint32_t)(N * d * sizeof(T));
            bulk_prefetch_l2(k + nb, bytes);
            bulk_prefetch_l2(v + nb, bytes);
            bulk_prefetch_l2(q + nb, bytes);
        }
        gsync();  // every warp is done with the previous unit's K and V
        // four elements (two words) a load, U loads in flight; word i of the unit
        // belongs to row i / h, 20 words long here
        auto stage = [&](auto batch) {
            constexpr int U = decltype(batch)::value;
            const T* ku = k + base;
            const T* vu = v + base;
            const int n = N * h / 2;
            for (int i0 = id; i0 < n; i0 += U * WPU * 32) {
                decltype(ld_global4(ku)) x[U], y[U];
#pragma unroll
                for (int e = 0; e < U; ++e) {
                    const int i = min(i0 + e * WPU * 32, n - 1);
                    x[e] = ld_global4(ku + 4 * i);
                    y[e] = ld_global4(vu + 4 * i);
                }
#pragma unroll
                for (int e = 0; e < U; ++e) {
                    const int i = 2 * min(i0 + e * WPU * 32, n - 1);  // the last words may be written twice
                    const int a0 = 4 * i + row_of(i) * (2 * kRow - 4 * h), a1 = 4 * (i + 1) + row_of(i + 1) * (2 * kRow - 4 * h);
                    st_plane(Ks + a0, PL, word(x[e], 0));
                    st_plane(Ks + a1, PL, word(x[e], 1));
                    st_plane(Vs + a0, PL, word(y[e], 0));
                    st_plane(Vs + a1, PL, word(y[e], 1));
                }
            }
        };
        // One warp makes h such loads per tensor and lane: all in one go where d_h is
        // compiled in (86400 units, d_h = 30, 245 -> 222 us), else in batches with little
        // over, as lanes beyond the end repeat its last words (40000 units, four at a
        // time, eight, twelve: d_h = 24, 121, 108 and 103 us; 28, 134, 118 and 126).
        // Four warps: eight at a time (6144 units, 178 -> 173 us), fp32 four (2000 units,
        // 163 us, eight 180).
        if constexpr (WPU > 1) stage(std::integral_constant<int, WPU == 4 && sizeof(T) == 2 ? 8 : 4>());
        else if constexpr (DC != 0) stage(std::integral_constant<int, 16>());
        else if (h > 8 && h <= 12) stage(std::integral_constant<int, 12>());
        else stage(std::integral_constant<int, 8>());
        gsync();
#pragma unroll 1
        for (int blk = 0; blk < 2; ++blk) {
            const T* q0 = q + base + (size_t)(64 * r + 32 * blk + g) * d;
            R aq[2][2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int c = 16 * kk + 8 * (e >> 1) + 2 * t;
                        aq[mt][kk][e] = c < d ? ld_global2(q0 + (16 * mt + 8 * (e & 1)) * d + c) : O::zero();
                    }
            float o[2][NTO][4], run[2][2];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                run[mt][0] = run[mt][1] = -INFINITY;
#pragma unroll
                for (int j = 0; j < NTO; ++j) o[mt][j][0] = o[mt][j][1] = o[mt][j][2] = o[mt][j][3] = 0.f;
            }
            // two chunks in a loop body where registers allow (5520 units of 32x32 windows
            // 2.09 -> 2.02 ms; fp32 would spill: 163 -> 184 us)
            constexpr int CU = ExactOp<T>::NP == 1 ? 2 : 1;
#pragma unroll CU
            for (int c = 0; c < N; c += 64) {
                float s[2][8][4];
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    R b[4];
                    ld_frag<false>(b, kf + (c + 8 * nt) * kRow * 2, PL);
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) {
                        O::mmaz(s[mt][nt], aq[mt][0], b[0], b[1]);
                        O::mma(s[mt][nt], aq[mt][1], b[2], b[3]);
                    }
                }
                // running maxima; the accumulators are rescaled
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float m = fmaxf(s[mt][0][2 * e], s[mt][0][2 * e + 1]);
#pragma unroll
                        for (int nt = 1; nt < 8; ++nt) m = fmaxf(m, fmaxf(s[mt][nt][2 * e], s[mt][nt][2 * e + 1]));
                        m = fmaxf(run[mt][e], quad_max(m) * sl2);
                        const float f = ex2(run[mt][e] - m);
                        run[mt][e] = m;
#pragma unroll
                        for (int j = 0; j < NTO; ++j) mul_x2(o[mt][j][2 * e], o[mt][j][2 * e + 1], f);
                    }
#pragma unroll
                for (int kt = 0; kt < 4; ++kt) {
                    R a[2][4];
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float* x = s[mt][2 * kt + (e >> 1)] + 2 * (e & 1);
                            const float m = -run[mt][e & 1];
                            float p0, p1;
                            fma_x2(p0, p1, x[0], x[1], sl2, sl2, m, m);
                            a[mt][e] = O::pk(ex2(p0), ex2(p1));
                        }
#pragma unroll
                    for (int j = 0; j < 4; j += 2) {
                        R b[4];
                        ld_frag<true>(b, vf + ((c + 16 * kt) * kRow + 8 * j) * 2, PL);
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt) {
                            O::mma(o[mt][j], a[mt], b[0], b[1]);
                            O::mma(o[mt][j + 1], a[mt], b[2], b[3]);
                        }
                    }
                    if constexpr (NCOL > 32) {
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt) O::mma(o[mt][4], a[mt], one0, one0);
                    }
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float d0 = 0.f, d1 = 0.f;
#pragma unroll
                for (int j = 0; j < NTO; ++j)
                    if (j == jd) {
                        d0 = o[mt][j][0];
                        d1 = o[mt][j][2];
                    }
                const float i0 = __fdividef(1.f, __shfl_sync(0xffffffffu, d0, src));
                const float i1 = __fdividef(1.f, __shfl_sync(0xffffffffu, d1, src));
                T* o0 = out + base + (size_t)(64 * r + 32 * blk + 16 * mt + g) * d;
                T* o1 = o0 + 8 * d;
#pragma unroll
                for (int j = 0; j < NTO; ++j) {
                    const int c = 8 * j + 2 * t;
                    if (c < d) {
                        O::st2(o0 + c, o[mt][j][0] * i0, o[mt][j][1] * i0);
                        O::st2(o1 + c, o[mt][j][2] * i1, o[mt][j][3] * i1);
                    }
                }
            }
        }
    }
}

template <typename T, int NCOL, int WPU, int DC>
cudaError_t launch_dc(const void* q, const void* k, const void* v, void* out, long long n_units, int d,
                      cudaStream_t stream) {
    using Lay = ExactLayout<T, WPU, DC>;
    constexpr int kThreads = Lay::GROUPS * WPU * 32;
    auto kern = exact_tc_kernel<T, NCOL, WPU, DC>;
    const size_t smem = (size_t)Lay::GROUPS * Lay::GROUP;
    static std::atomic<int> s_blocks[kMaxDevices];  // persistent grid size per device
    int blocks = 0;
    if (cudaError_t e = persistent_grid(kern, kThreads, smem, s_blocks, &blocks); e != cudaSuccess) return e;
    // the fewest groups per CTA that still reach the minimal number of rounds: few
    // units spread over the SMs (384 units of 8x8 windows, d_h = 30, 7.2 -> 3.9 us; 6 of
    // 16x16 13.6 -> 6.6) and more of them share an SM no longer than needed
    const long long rounds = (n_units + blocks * Lay::GROUPS - 1) / (blocks * Lay::GROUPS);
    const long long groups = (n_units + blocks * rounds - 1) / (blocks * rounds);
    const long long want = (n_units + groups - 1) / groups;
    const long long grid = want < blocks ? want : blocks;
    const float sl2 = 1.4426950408889634f / sqrtf((float)d);
    kern<<<(unsigned)grid, (unsigned)(groups * WPU * 32), (size_t)groups * Lay::GROUP, stream>>>(
        (const T*)q, (const T*)k, (const T*)v, (T*)out, n_units, d, sl2);
    return cudaGetLastError();
}

// The common head widths get kernels with d_h as a compile-time constant.
template <typename T, int WPU>
cudaError_t launch_n(const void* q, const void* k, const void* v, void* out, long long n_units, int d,
                     cudaStream_t stream) {
    if (d == 32) return launch_dc<T, 40, WPU, 32>(q, k, v, out, n_units, d, stream);
    if (d == 30) return launch_dc<T, 32, WPU, 30>(q, k, v, out, n_units, d, stream);
    return launch_dc<T, 32, WPU, 0>(q, k, v, out, n_units, d, stream);
}

template <typename T>
cudaError_t launch_t(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d,
                     cudaStream_t stream) {
    switch (N) {
        case 64: return launch_n<T, 1>(q, k, v, out, n_units, d, stream);
        case 256: return launch_n<T, 4>(q, k, v, out, n_units, d, stream);
        default:
            if constexpr (sizeof(T) == 4) return cudaErrorInvalidValue;  // not offered (see supports)
            else return launch_n<T, 16>(q, k, v, out, n_units, d, stream);
    }
}

}  // namespace
}  // namespace nystra

namespace nystra_host {
bool exact_tc_supports(int N, int d, int dtype) {
    const bool shape = d >= 2 && d <= 32 && d % 2 == 0;
    if (dtype == 0) return shape && (N == 64 || N == 256);
    return (dtype == 1 || dtype == 2) && (N == 64 || N == 256 || N == 1024) && shape;
}

cudaError_t launch_exact_tc(const void* q, const void* k, const void* v, void* out, long long n_units, int N,
                            int d, int dtype, cudaStream_t stream) {
    if (dtype == 0) return nystra::launch_t<float>(q, k, v, out, n_units, N, d, stream);
    if (dtype == 1) return nystra::launch_t<__nv_bfloat16>(q, k, v, out, n_units, N, d, stream);
    return nystra::launch_t<__half>(q, k, v, out, n_units, N, d, stream);
}
}  // namespace nystra_host
