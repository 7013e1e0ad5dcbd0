// Wide-landmark PnP-Nystra kernel: m = 64 at 8x8 and 16x16 windows (N = 64,
// 256 tokens), even d_h <= 32, 16-bit I/O, segment landmarks.  Included by the N =
// 64 and 256 translation units after nystra_tc.cuh, whose per-phase device
// functions it reuses.
//
// With so many landmarks the m x m core dominates a unit, so a unit's group is
// the core's CW = m/16 warps, and they share the token side too, by landmarks:
//   stage    Q, K, V of the unit by three bulk copies on two mbarriers;
//   front    landmark means, every warp a share; [sync]; warp c: S_U of its 16
//            landmarks against all tokens, its rows of W in registers (no partial
//            W, no combine);
//   core     sc_core; its scratch overlays K and V, W Qbar, Y^T one of its
//            matrices; [sync]
//   output   every warp a share of the 16-token tiles: S_L, G_L^n from the
//            resident Q, O in place over Q; [sync]; one bulk store.
// Nothing of the next unit is copied while a unit runs: its K and V would cost
// a group per SM, and the SM's other groups fill the wait.  Three groups of
// four warps run per SM (73 KB each at N = 256), against two groups with 108 KB
// and two token warps each on the grouped kernel.
// What bounds it: dependent MMAs and the tensor pipe (63% busy at 16x16 windows,
// 0.40 instructions issued per cycle, LSU data pipe 66%).
// Measured (bf16): 4096 units of 16x16 windows, d_h = 32: 0.92 -> 0.45 ms; 8640
// units of 8x8 windows, d_h = 30: 1.44 -> 0.72 ms.
//
// Every wait on an mbarrier is bounded; the warps of a group share its
// barriers, and a wait that gives up is agreed on at the next one.
#pragma once

#include "nystra_tc.cuh"

namespace nystra {
namespace tc {

template <typename T, int M, int NCOL, int N>
struct WideLayout {
    using Sc = ScScratch<M>;
    static constexpr int CW = Sc::CW;
    static constexpr int DS = (NCOL == 32) ? 30 : 32;
    static constexpr size_t ROWS = (size_t)N * DS * 2;
    static constexpr size_t G_Q = 0;
    static constexpr size_t G_KV = ROWS;  // K, V; the core's two matrices
    static constexpr size_t KV = ((2 * ROWS > 2 * Sc::MAT ? 2 * ROWS : 2 * Sc::MAT) + 15) / 16 * 16;
    static constexpr size_t G_QV = G_KV + KV;  // Qbar; W
    static constexpr size_t WMAT = (size_t)M * (NCOL + 4) * 4;
    static constexpr size_t QV = LmS<T>::bytes(M) > WMAT ? LmS<T>::bytes(M) : WMAT;
    static constexpr size_t G_KBAR = G_QV + QV;
    static constexpr size_t G_AUX = G_KBAR + LmS<T>::bytes(M);
    static constexpr size_t G_BAR = G_AUX + Sc::AUX;  // Q and K rows; V rows
    static constexpr size_t GROUP = ((G_BAR + 16 + 127) / 128) * 128;
    static constexpr int by_smem = (int)(kSmemLimit / GROUP);
    static constexpr int by_regs = 12 / CW;  // 12 warps of up to 168 registers
    static constexpr int GROUPS = by_smem < by_regs ? by_smem : by_regs;
    static_assert(ROWS % 16 == 0 && QV % 16 == 0 && LmS<T>::bytes(M) % 16 == 0, "16-byte alignment");
    static_assert(GROUPS >= 1, "does not fit");
};

// Landmark means of X (N rows of d) into xbar, thread id of n: fp32 sums of L
// 16-bit values times 1/L (a power of two), stored as DSt does (in slot order
// for RS = kSlots).
template <typename T, int M, int N, int RS>
__device__ __forceinline__ void wide_landmarks(const T* X, T* xbar, int d, int id, int n) {
    constexpr int L = N / M, LS = LmS<T>::LS, LO = LmS<T>::LO;
    for (int i = id; i < M * 16; i += n) {
        const int j = i >> 4, c = 2 * (i & 15);
        float a = 0.f, b = 0.f;
        if (c < d) {
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const uint32_t x = *reinterpret_cast<const uint32_t*>(X + (j * L + l) * d + c);
                const float2 f = Mma16<T>::unpack(x);
                a += f.x;
                b += f.y;
            }
        }
        const int p = RS == kSlots ? 4 * (c & 6) + 2 * (c >> 3) : c;
        DSt<T>::put(xbar + j * LS + p, LO, a * (1.f / L));
        DSt<T>::put(xbar + j * LS + p + 1, LO, b * (1.f / L));
    }
}

// B operand registers of rows r0 .. r0 + 7 (the columns of B) at k = 16 kk, kk
// = 0, 1, of a DSt matrix with row stride `rs` halves: ldmatrix, no conflicts
// as the strides are odd multiples of 16 bytes.
template <typename T>
__device__ __forceinline__ void wide_b_k32(const T* x, int rs, int lo, int lane, typename Opnd<T>::DReg (&b)[2][2]) {
    const T* p = x + (lane & 7) * rs + 8 * (lane >> 3);
    uint32_t h[4];
    ldsm_x4(h, p);
    if constexpr (sizeof(typename Opnd<T>::DReg) == 8) {
        uint32_t l[4];
        ldsm_x4(l, p + lo);
        b[0][0] = {h[0], l[0]}; b[0][1] = {h[1], l[1]};
        b[1][0] = {h[2], l[2]}; b[1][1] = {h[3], l[3]};
    } else {
        b[0][0] = h[0]; b[0][1] = h[1];
        b[1][0] = h[2]; b[1][1] = h[3];
    }
}

// One 16-token tile of the output: rows q0 (row g) and q0 + mrow (row g + 8)
// of the resident Q, overwritten by O.
template <typename T, int M, int NCOL, int RS>
__device__ __forceinline__ void wide_output_tile(T* q0, const T* kbar, const T* yT, int d, int t, int lane, float sl2) {
    using O = Opnd<T>;
    using R = typename O::Reg;
    using D = typename O::DReg;
    constexpr int NTL = M / 8, KT = M / 16, NTO = NCOL / 8, LS = LmS<T>::LS, LO = LmS<T>::LO, YS = YtS<T, M>::YS,
                  YLO = YtS<T, M>::LO;
    R a[2][4];
    q_afrag<T, RS>(q0, d, t, a);
    float sl[NTL][4];
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int j = 0; j < NTL; ++j) {
        D b[2][2];
        wide_b_k32<T>(kbar + 8 * j * LS, LS, LO, lane, b);
        O::mmaz(sl[j], a[0], b[0][0], b[0][1]);
        O::mma(sl[j], a[1], b[1][0], b[1][1]);
    }
#pragma unroll
    for (int j = 0; j < NTL; ++j) {
        mx0 = fmaxf(mx0, fmaxf(sl[j][0], sl[j][1]));
        mx1 = fmaxf(mx1, fmaxf(sl[j][2], sl[j][3]));
    }
    mx0 = quad_max(mx0) * sl2;
    mx1 = quad_max(mx1) * sl2;
    auto e0 = [&](float x) { return ex2(fmaf(x, sl2, -mx0)); };
    auto e1 = [&](float x) { return ex2(fmaf(x, sl2, -mx1)); };
    float o[NTO][4];
#pragma unroll
    for (int j = 0; j < NTO; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
#pragma unroll
    for (int kp = 0; kp < KT; kp += 2) {  // G_L^n of 32 landmarks, straight from the scores
        D f[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int kk = kp + h;
            f[h][0] = O::dpk(e0(sl[2 * kk][0]), e0(sl[2 * kk][1]));
            f[h][1] = O::dpk(e1(sl[2 * kk][2]), e1(sl[2 * kk][3]));
            f[h][2] = O::dpk(e0(sl[2 * kk + 1][0]), e0(sl[2 * kk + 1][1]));
            f[h][3] = O::dpk(e1(sl[2 * kk + 1][2]), e1(sl[2 * kk + 1][3]));
        }
#pragma unroll
        for (int j = 0; j < NTO; ++j) {
            D b[2][2];
            wide_b_k32<T>(yT + 8 * j * YS + 16 * kp, YS, YLO, lane, b);
            O::mma(o[j], f[0], b[0][0], b[0][1]);
            O::mma(o[j], f[1], b[1][0], b[1][1]);
        }
    }
    const int jd = d >> 3, src = (lane & ~3) | ((d & 7) >> 1);
    float d0 = 0.f, d1 = 0.f;
#pragma unroll
    for (int j = 0; j < NTO; ++j)
        if (j == jd) {
            d0 = o[j][0];
            d1 = o[j][2];
        }
    const float i0 = __fdividef(1.f, __shfl_sync(0xffffffffu, d0, src));
    const float i1 = __fdividef(1.f, __shfl_sync(0xffffffffu, d1, src));
    store_orows<T, NTO, RS>(q0, d, t, o, i0, i1);
}

template <typename T, int M, int NCOL, int N, int DC>
__global__ void __launch_bounds__(WideLayout<T, M, NCOL, N>::GROUPS * WideLayout<T, M, NCOL, N>::CW * 32, 1)
nystra_wide_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ out,
                   long long n_units, int d_in, int iters, float sl2, unsigned int* fault, int active) {
    using Lay = WideLayout<T, M, NCOL, N>;
    using Sc = typename Lay::Sc;
    constexpr int CW = Lay::CW, NTO = NCOL / 8;
    const int d = DC ? DC : d_in;
    constexpr int RS = row_order<T>(DC);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp / CW, c = warp - grp * CW;
    const int g = lane >> 2, t = lane & 3;
    unsigned char* gb = smem_raw + (size_t)grp * Lay::GROUP;
    const int td = N * d;  // elements per tensor of a unit
    T* Qs = reinterpret_cast<T*>(gb + Lay::G_Q);
    T* Ks = reinterpret_cast<T*>(gb + Lay::G_KV);
    T* Vs = Ks + td;
    T* qbar = reinterpret_cast<T*>(gb + Lay::G_QV);
    T* kbar = reinterpret_cast<T*>(gb + Lay::G_KBAR);
    uint64_t* barQK = reinterpret_cast<uint64_t*>(gb + Lay::G_BAR);
    uint64_t* barV = barQK + 1;
    const uint32_t bytes = (uint32_t)(td * sizeof(T));
    const int bar = 1 + grp;  // named barrier of the group
    auto gsync = [&]() { named_barrier(bar, CW * 32); };

    // Only the first `active` groups of a CTA take units (see launch_wide_dc).
    const long long stride = (long long)gridDim.x * active;
    long long u = grp < active ? (long long)blockIdx.x * active + grp : n_units;
    const bool leader = c == 0 && lane == 0;
    auto issue_kv = [&](long long unit) {
        const size_t off = (size_t)unit * td;
        bulk_g2s(Ks, k + off, bytes, barQK);
        mbar_arrive_expect_tx(barV, bytes);
        bulk_g2s(Vs, v + off, bytes, barV);
    };
    auto issue_q = [&](long long unit) { bulk_g2s(Qs, q + (size_t)unit * td, bytes, barQK); };

    if (leader) {
        mbar_init(barQK, 1);
        mbar_init(barV, 1);
        fence_mbar_init();
    }
    gsync();
    bool pend = u < n_units;  // copies issued and not yet seen complete
    if (pend && leader) {
        mbar_arrive_expect_tx(barQK, 2u * bytes);
        issue_q(u);
        issue_kv(u);
    }
    uint32_t phase = 0;
    bool failed = false;  // a bounded wait of this warp gave up (warp-uniform)
    auto wait = [&](uint64_t* b) {
        if (failed) return;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(b, phase, kWaitNs))) {
            failed = true;
            if (lane == 0) atomicOr(fault, 1u);
        }
    };

    for (; u < n_units; u += stride) {
        // ---------------- landmarks (Algorithm 1 step 1) ----------------
        wait(barQK);
        wide_landmarks<T, M, N, RS>(Qs, qbar, d, c * 32 + lane, CW * 32);
        wide_landmarks<T, M, N, RS>(Ks, kbar, d, c * 32 + lane, CW * 32);
        wait(barV);
        if (named_barrier_or(bar, CW * 32, failed)) break;
        pend = false;
        phase ^= 1u;
        // ---------------- S_U, m_U and W of landmarks 16c .. 16c + 15 ----------------
        float w[NTO][4], run0 = -INFINITY, run1 = -INFINITY;
        {
            typename Opnd<T>::DReg aq[2][4];
            qbar_afrag<T>(qbar, c, g, t, aq);
#pragma unroll
            for (int j = 0; j < NTO; ++j) w[j][0] = w[j][1] = w[j][2] = w[j][3] = 0.f;
#pragma unroll 1
            for (int ch = 0; ch < N / 64; ++ch)
                su_w_chunk<T, NCOL, false, RS>(aq, Ks + ch * 64 * d, Vs + ch * 64 * d, d, g, t, sl2, true, true, w,
                                               run0, run1, N > 64);
        }
        // ---------------- core ----------------
        // (its first write to the K and V rows comes after a barrier of its own)
        const T* yT = sc_core<T, M, NCOL, true>(qbar, kbar, run0, run1, w, nullptr, gb + Lay::G_KV,
                                                gb + Lay::G_KV + Sc::MAT, reinterpret_cast<float*>(gb + Lay::G_QV),
                                                reinterpret_cast<float*>(gb + Lay::G_AUX), iters, sl2, c, lane, bar);
        gsync();
        // ---------------- output, in place over Q ----------------
#pragma unroll 1
        for (int tile = c; tile < N / 16; tile += CW)
            wide_output_tile<T, M, NCOL, RS>(Qs + ((tile >> 2) * 64 + mtok<RS>(tile & 3, g)) * d, kbar, yT, d, t, lane,
                                             sl2);
        fence_proxy_async_smem();  // this lane's accesses precede the bulk store and the next copies
        gsync();
        const long long un = u + stride;
        pend = un < n_units;
        if (leader) {
            bulk_s2g(out + (size_t)u * td, Qs, bytes);
            bulk_commit();
            if (pend) {
                mbar_arrive_expect_tx(barQK, 2u * bytes);
                issue_kv(un);
            }
            bulk_wait_read_all();
            if (pend) issue_q(un);
        }
        __syncwarp();
    }
    if (leader) bulk_wait_all();  // output stores complete before exit
    // Fault path only: copies still in flight land before the CTA's memory is released.
    if (pend) {
        (void)__all_sync(0xffffffffu, mbar_wait_bounded(barQK, phase, kWaitNs));
        (void)__all_sync(0xffffffffu, mbar_wait_bounded(barV, phase, kWaitNs));
    }
}

template <typename T, int M, int NCOL, int N, int DC>
cudaError_t launch_wide_dc(const void* q, const void* k, const void* v, void* out, long long n_units, int d, int iters,
                           cudaStream_t stream, unsigned int* fault) {
    using Lay = WideLayout<T, M, NCOL, N>;
    constexpr int kGroups = Lay::GROUPS, kThreads = kGroups * Lay::CW * 32;
    auto kern = nystra_wide_kernel<T, M, NCOL, N, DC>;
    const size_t smem = (size_t)kGroups * Lay::GROUP;
    static std::atomic<int> s_blocks[kMaxDevices];  // persistent grid size per device
    int blocks = 0;
    if (cudaError_t e = persistent_grid(kern, kThreads, smem, s_blocks, &blocks); e != cudaSuccess) return e;
    // the fewest groups per CTA that still reach the minimal number of rounds
    // contend least for the SM
    const long long rounds = (n_units + blocks * kGroups - 1) / (blocks * kGroups);
    int active = (int)((n_units + blocks * rounds - 1) / (blocks * rounds));
    active = active < 1 ? 1 : (active > kGroups ? kGroups : active);
    const long long want = (n_units + active - 1) / active;
    const long long grid = want < blocks ? want : blocks;
    const float sl2 = 1.4426950408889634f / sqrtf((float)d);
    kern<<<(unsigned)grid, kThreads, smem, stream>>>((const T*)q, (const T*)k, (const T*)v, (T*)out, n_units, d, iters,
                                                     sl2, fault, active);
    return cudaGetLastError();
}

// The common head widths get kernels with d_h as a compile-time constant.
template <typename T, int M, int NCOL, int N>
cudaError_t launch_wide(const void* q, const void* k, const void* v, void* out, long long n_units, int d, int iters,
                        cudaStream_t stream, unsigned int* fault) {
    constexpr int DC = NCOL == 32 ? 30 : 32;
    if (d == DC) return launch_wide_dc<T, M, NCOL, N, DC>(q, k, v, out, n_units, d, iters, stream, fault);
    return launch_wide_dc<T, M, NCOL, N, 0>(q, k, v, out, n_units, d, iters, stream, fault);
}

}  // namespace tc
}  // namespace nystra
