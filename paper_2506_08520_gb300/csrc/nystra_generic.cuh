// Generic PnP-Nystra kernel: any N <= 1024, m | N with m <= 64, d_h <= 64.
// Included by one translation unit per landmark bound (nystra_generic_m*.cu).
//
// One CTA per (window, head) unit, all arithmetic in fp32 with expf.  Tokens
// are staged in chunks as fp32, so shared memory holds a chunk of Q, K or V,
// its scores and the O(m^2 + m d) state:
//   pass 1  Qbar (segment or square-patch means, Algorithm 1 step 1);
//   pass 2  K and V chunks: Kbar's sums, S_U = s Qbar K^T with a running row
//           max m_U, and W = G_U^n [V | 1] accumulated with the usual online
//           rescaling, so that at the end W = exp(S_U - m_U) [V | 1] for the
//           final m_U;
//   core    G_A^n = exp(s Qbar Kbar^T - m_U), the third-order iteration for
//           Z ~ (G_A^n)^+ (step 4), Y = Z W;
//   pass 3  Q chunks: G_L^n = exp(S_L - m_L) and O = (G_L^n Y_:d) / (G_L^n Y_d)
//           (steps 5-7, re-associated as G_L^n (Z (G_U^n [V | 1]))).
// This is the always-available path (and the fp32-exact one); shape-specialised
// tensor-core kernels take the common shapes.
//
// Every product is A B^T over rows that are contiguous along the contraction
// (right factors are stored transposed), in register tiles of 4 x 4 results:
// eight 16-byte shared loads feed 32 packed FMAs (fma.rn.f32x2, the even and
// odd terms of a dot product summed apart).  Row strides are an odd number of
// 16-byte granules and a tile's rows lie a whole group of tiles apart, so the
// lanes of a warp read neighbouring rows, free of bank conflicts.  A score
// tile stays in registers from the product through its row maximum (shuffles)
// and exponentials, and is stored once.  Up to 16 landmarks the m x m core is
// one warp's (no CTA barriers); the other CTAs of the SM fill its wait.
//
// What bounds it: instruction issue and shared-memory latency (12x12 windows,
// m = 16, fp16: 43,000 warp instructions per unit, 0.51 issued per cycle, 19
// warps per SM, DRAM 6%), so chunks are as long as one score tile per thread
// allows: chunks of 72 and 88 tokens with more CTAs per SM were 4-12% slower.
// Measured: 6144 units of 16x16 windows, d_h = 30, m = 16, fp32 1.52 -> 0.62 ms
// (1.2 TB/s of Q, K, V, O); 11094 units of 12x12, fp16 1.62 -> 0.76 ms; 1668
// units of 16x16, d_h = 32, m = 32 with a score bias 3.94 -> 0.40 ms, against a
// kernel with one shared load per operand and 32-token chunks.
#pragma once

#include "simt.cuh"

namespace nystra {
namespace generic {

using namespace simt;

// Per landmark bound MP (8, 16, 32, 64): groups of four landmarks (the lanes
// that share a token group), the longest token chunk (one score tile per
// thread) and the row stride of anything with landmark columns.
template <int MP>
struct Bound {
    static constexpr int JG = MP / 4;
    static constexpr int CH = MP <= 16 ? 160 : (MP == 32 ? 128 : 64);
    static constexpr int MS = MP + 4;
    static_assert((MS / 4) % 2 == 1, "odd granules");
    // W's tiles (17 column groups at d_h = 64) may outnumber the score tiles
    static constexpr int kTiles = JG * 17 > CH / 4 * JG ? JG * 17 : CH / 4 * JG;
    static constexpr int kThreads = kTiles > 128 ? (kTiles + 31) / 32 * 32 : 128;
    static constexpr int kCtas = MP <= 16 ? 4 : (MP == 32 ? 2 : 1);
};

// Region sizes in floats for one call; DS: row stride of d_h columns.
template <int MP, int DS>
struct Shape {
    using B = Bound<MP>;
    int ch, c4, ks, threads;  // chunk, groups of four columns of [V | 1], token splits of W, CTA size
    int ns;                   // row stride of anything with token columns: odd granules
    int kv, p;
    static constexpr int kLm = MP * DS, kMat = MP * B::MS;
    __host__ __device__ Shape(int N, int d, int min_threads) {
        const int chunks = (N + B::CH - 1) / B::CH;
        ch = 4 * ((N + 4 * chunks - 1) / (4 * chunks));
        ns = 4 * ((ch / 4) | 1);
        c4 = d / 4 + 1;
        const int tiles = B::JG * c4;
        threads = ch / 4 * B::JG;
        threads = ((threads > tiles ? threads : tiles) + 31) / 32 * 32;
        ks = threads / tiles;  // (before min_threads: a unit's sums do not depend on how many units there are)
        if (ks > ch / 4) ks = ch / 4;
        threads = threads > min_threads ? threads : min_threads;
        kv = ch * DS;                                               // Q or K rows
        if (4 * c4 * ns > kv) kv = 4 * c4 * ns;                     // V^T
        if (ks * 4 * c4 * B::MS > kv) kv = ks * 4 * c4 * B::MS;     // W^T's splits
        if (6 * kMat > kv) kv = 6 * kMat;                           // the core's matrices
        p = MP * ns > ch * B::MS ? MP * ns : ch * B::MS;
    }
    __host__ __device__ int wt() const { return 4 * c4 * B::MS; }
    __host__ __device__ size_t bytes() const {
        return sizeof(float) * (size_t)(kv + p + 2 * kLm + 2 * wt() + 2 * MP + 4 + ch + 9 * MP);
    }
};

__device__ __forceinline__ float warp_max(float x) {
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// ---- the m x m core ----
// put(i, j, (A B^T)[i][j]) for i < m4 and j < rb (multiples of four), by
// threads 0 .. n - 1.
template <int TI, int MS, int KU, typename Put>
__device__ __forceinline__ void product(const float* A, const float* Bt, int m4, int rb, int id, int n, Put put) {
    const int gi = m4 / TI, gj = rb >> 2;
    for (int it = id; it < gi * gj; it += n) {
        const int i0 = it / gj, j0 = it - i0 * gj;
        f32x2 acc[TI][4];
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
        tile_nt<TI, 4, KU>(A + i0 * MS, gi * MS, Bt + j0 * MS, gj * MS, m4 >> 2, acc);
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) put(i0 + i * gi, j0 + j * gj, sum2(acc[i][j]));
    }
}

// `iters` steps Z <- Z (13I - X (15I - X (7I - X))) / 4, X = A Z, and
// Y^T = (Z W)^T from W^T.  mats: A row-major, then five more matrices; alpha
// scales Z_0 = alpha A^T.  Right factors are kept transposed, Z both ways.
template <int MP, bool ONE_WARP>
__device__ __forceinline__ void core(float* mats, float alpha, const float* Wt, float* Yt, int c4, int m, int m4,
                                     int iters, int id, int n) {
    constexpr int MS = Bound<MP>::MS, kMat = MP * MS, TI = MP <= 32 ? 2 : 4, KU = ONE_WARP ? MP / 4 : 2;
    if constexpr (ONE_WARP) m4 = MP, n = 32;  // constant loops; the padding is zero
    auto sync = [] {
        if constexpr (ONE_WARP) __syncwarp();
        else __syncthreads();
    };
    const float* A = mats;
    float* Zr = mats + kMat;
    float* Zt = mats + 2 * kMat;
    float* X = mats + 3 * kMat;
    float* T1 = mats + 4 * kMat;
    float* T2 = mats + 5 * kMat;
    for (int it = id; it < m4 * m4; it += n) {
        const int i = it / m4, j = it - i * m4;
        const float z = alpha * A[i * MS + j];
        Zt[i * MS + j] = z;
        Zr[j * MS + i] = z;
    }
    sync();
    for (int it = 0; it < iters; ++it) {
        product<TI, MS, KU>(A, Zt, m4, m4, id, n, [&](int i, int j, float p) {  // X and 7I - X
            X[i * MS + j] = p;
            T1[j * MS + i] = (i == j && i < m ? 7.f : 0.f) - p;
        });
        sync();
        product<TI, MS, KU>(X, T1, m4, m4, id, n,  // 15I - X(7I - X)
                        [&](int i, int j, float p) { T2[j * MS + i] = (i == j && i < m ? 15.f : 0.f) - p; });
        sync();
        product<TI, MS, KU>(X, T2, m4, m4, id, n,  // 13I - X(15I - ...)
                        [&](int i, int j, float p) { T1[j * MS + i] = (i == j && i < m ? 13.f : 0.f) - p; });
        sync();
        product<TI, MS, KU>(Zr, T1, m4, m4, id, n, [&](int i, int j, float p) {
            T2[i * MS + j] = 0.25f * p;
            Zt[j * MS + i] = 0.25f * p;
        });
        sync();
        float* z = Zr;
        Zr = T2;
        T2 = z;
    }
    product<TI, MS, KU>(Zr, Wt, m4, 4 * c4, id, n, [&](int j, int c, float p) { Yt[c * MS + j] = p; });
}

template <int MP, int DS, typename T>
__device__ __forceinline__ void run(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                    T* __restrict__ out, long long n_units, int N, int d, int m, int iters, int pw,
                                    float scale, const NystraBias& bias, float* sm) {
    using B = Bound<MP>;
    constexpr int JG = B::JG, MS = B::MS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nth = blockDim.x, NW = nth >> 5;
    const Shape<MP, DS> G(N, d, nth);
    const int ch = G.ch, ns = G.ns, c4 = G.c4, ks = G.ks, L = N / m, m4 = (m + 3) & ~3;
    const int kg = (d + 3) >> 2, pl = 4 * kg <= 16 ? 3 : (4 * kg <= 32 ? 4 : 5);
    float* KV = sm;                 // Q or K rows (DS), V^T (ns), W^T's splits, the core's matrices, O rows
    float* P = KV + G.kv;           // exponentials: [MP][ns] (U side) or [ch][MS] (L side)
    float* qbar = P + G.p;          // MP rows, zero beyond m and d
    float* kbar = qbar + G.kLm;     // MP rows
    float* Wt = kbar + G.kLm;       // 4 c4 rows: (G_U^n [V | 1])^T
    float* Yt = Wt + G.wt();        // 4 c4 rows: (Z W)^T
    float* mU = Yt + G.wt();        // MP
    float* rs = mU + MP;            // MP      rescale factors
    float* red = rs + MP;           // 4       1/(||A||_1 ||A||_inf)
    float* rowv = red + 4;          // ch      1 / denominators
    float* wmax = rowv + ch;        // [warps][MP] partial row maxima

    // score tile of this thread: landmarks j0 + JG i, tokens t0 + tg i
    const int j0 = tid % JG, t0 = tid / JG;
    // W tile: split ws of the tokens, landmarks wj + JG i, columns wc + c4 i
    const int ws = tid / (JG * c4), wj = (tid - ws * JG * c4) / c4, wc = tid - (ws * JG + wj) * c4;

    // Landmark j covers `rows` runs of `len` tokens, `pw` apart: a segment of
    // L tokens, or (pw > 0) a pb x pb patch of the pw-wide window, pb^2 = L.
    int pb = 1, pp = 1;
    if (pw > 0) {
        while ((pp + 1) * (pp + 1) <= m) ++pp;
        pb = pw / pp;
    }
    const int rows = pw > 0 ? pb : 1, len = pw > 0 ? pb : L;
    // adds the tokens c0 .. c0 + nt - 1 (rows at KV) to the landmark sums
    auto add_landmarks = [&](float* sums, int c0, int nt) {
        for (int i = tid; i < m * kg; i += nth) {
            const int j = i / kg, c = 4 * (i - j * kg);
            const int f = (pw > 0 ? (j / pp) * pb * pw + (j % pp) * pb : j * L) - c0;
            float4 a = *reinterpret_cast<const float4*>(sums + j * DS + c);
            for (int r = 0; r < rows; ++r) {
                const int lo = max(f + r * pw, 0), hi = min(f + r * pw + len, nt);
                for (int t = lo; t < hi; ++t) {
                    const float4 x = *reinterpret_cast<const float4*>(KV + t * DS + c);
                    a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
                }
            }
            *reinterpret_cast<float4*>(sums + j * DS + c) = a;
        }
    };
    auto put_rows = [&](int r, int c, float2 x) { *reinterpret_cast<float2*>(KV + r * DS + c) = x; };
    // s[i][j] = scale a_(j0 + JG j) . x_(t0 + tg i) + bias, -inf outside the landmarks and tokens;
    // bias of landmark j and token t at b[j * bj + t * bt]
    auto scores = [&](const float* a, int tg, int nt, const float* __restrict__ b, int bj, int bt, float (&s)[4][4]) {
        f32x2 acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
        if (t0 < tg) tile_nt<4, 4>(KV + t0 * DS, tg * DS, a + j0 * DS, JG * DS, kg, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int t = t0 + i * tg, jj = j0 + j * JG;
                s[i][j] = -INFINITY;
                if (t0 < tg && t < nt && jj < m) {
                    s[i][j] = scale * sum2(acc[i][j]);
                    if (b) s[i][j] += __ldg(b + (size_t)jj * bj + (size_t)t * bt);
                }
            }
    };

    for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
        const size_t base = (size_t)u * N * d;
        const T* qu = q + base;
        const T* ku = k + base;
        const T* vu = v + base;
        T* ou = out + base;
        // score bias through the landmarks (null without one): slice of this unit
        const long long bs = bias.per_window ? u : u % bias.heads;
        const float* bLu = bias.L ? bias.L + (size_t)bs * N * m : nullptr;
        const float* bUu = bias.U ? bias.U + (size_t)bs * m * N : nullptr;
        const float* bAu = bias.A ? bias.A + (size_t)bs * m * m : nullptr;

        // K and V will be wanted soon: bring them to L2 while Q is pooled
        for (int i = tid; i * 128 < N * d * (int)sizeof(T); i += nth) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(ku) + i * 128));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(vu) + i * 128));
        }

        // ---- pass 1: Qbar ----
        for (int i = tid; i < 2 * G.kLm; i += nth) qbar[i] = 0.f;  // and kbar
        for (int c0 = 0; c0 < N; c0 += ch) {
            const int nt = min(ch, N - c0), tg = (nt + 3) >> 2;
            load_rows<T>(qu + (size_t)c0 * d, nt, tg, d, 4 * kg, pl, put_rows);
            __syncthreads();
            add_landmarks(qbar, c0, nt);
            __syncthreads();
        }
        for (int i = tid; i < G.kLm; i += nth) qbar[i] = qbar[i] / (float)L;

        // ---- pass 2: Kbar's sums, S_U, running m_U, W = G_U^n [V | 1] ----
        float run[4], w[4][4];  // m_U of landmarks j0 + JG j; this thread's tile of W
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            run[i] = -INFINITY;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[i][j] = 0.f;
        }
        for (int c0 = 0; c0 < N; c0 += ch) {
            const int nt = min(ch, N - c0), tg = (nt + 3) >> 2;
            load_rows<T>(ku + (size_t)c0 * d, nt, tg, d, 4 * kg, pl, put_rows);
            __syncthreads();
            float s[4][4];
            scores(qbar, tg, nt, bUu ? bUu + c0 : nullptr, N, 1, s);
            add_landmarks(kbar, c0, nt);
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // row maxima: this thread, its warp, the CTA
                float mx = fmaxf(fmaxf(s[0][j], s[1][j]), fmaxf(s[2][j], s[3][j]));
#pragma unroll
                for (int o = 16; o >= JG; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane < JG) wmax[warp * MP + j0 + j * JG] = mx;
            }
            __syncthreads();  // K has been read: V may take its place
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int jj = j0 + j * JG;
                float mx = run[j];
                for (int x = 0; x < NW; ++x) mx = fmaxf(mx, wmax[x * MP + jj]);
                if (tid < JG) {
                    rs[jj] = (run[j] == -INFINITY) ? 0.f : expf(run[j] - mx);
                    mU[jj] = mx;
                }
                run[j] = mx;
                if (t0 < tg) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        P[jj * ns + t0 + i * tg] = (t0 + i * tg < nt && jj < m) ? expf(s[i][j] - mx) : 0.f;
                }
            }
            load_rows<T>(vu + (size_t)c0 * d, nt, tg, d, d, pl, [&](int r, int c, float2 x) {
                KV[c * ns + r] = x.x;
                if (c + 1 < d) KV[(c + 1) * ns + r] = x.y;
            });
            for (int i = tid; i < 4 * tg; i += nth) {
                KV[d * ns + i] = i < nt ? 1.f : 0.f;
                for (int c = d + 1; c < 4 * c4; ++c) KV[c * ns + i] = 0.f;
            }
            __syncthreads();
            if (ws < ks) {
                const int g0 = ws * tg / ks, g1 = (ws + 1) * tg / ks;  // this split's groups of four tokens
                f32x2 acc[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float f = rs[wj + JG * i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = __float_as_uint(w[i][j] * f);  // (w f, 0)
                }
                tile_nt<4, 4>(P + wj * ns + 4 * g0, JG * ns, KV + wc * ns + 4 * g0, c4 * ns, g1 - g0, acc);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) w[i][j] = sum2(acc[i][j]);
            }
            __syncthreads();
        }
        // W^T's splits, then their sum; Kbar's means
        if (ws < ks) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) KV[ws * G.wt() + (wc + c4 * j) * MS + wj + JG * i] = w[i][j];
        }
        for (int i = tid; i < G.kLm; i += nth) kbar[i] = kbar[i] / (float)L;
        __syncthreads();
        for (int i = tid; i < 4 * c4 * MP; i += nth) {
            const int e = i / MP * MS + i % MP;
            float a = KV[e];
            for (int x = 1; x < ks; ++x) a += KV[x * G.wt() + e];
            Wt[e] = a;
        }
        __syncthreads();

        // ---- core: G_A^n, pseudo-inverse iteration, Y = Z W ----
        float* A = KV;
        for (int i = tid; i < (MP <= 16 ? MP : m4) * MP; i += nth) {
            const int r = i / MP, j = i % MP;
            float e = 0.f;
            if (r < m && j < m) {
                f32x2 a[1][1] = {{0ull}};
                tile_nt<1, 1>(qbar + r * DS, 0, kbar + j * DS, 0, kg, a);
                e = expf(scale * sum2(a[0][0]) + (bAu ? __ldg(bAu + r * m + j) : 0.f) - mU[r]);
            }
            A[r * MS + j] = e;
        }
        __syncthreads();
        if (warp == 0) {
            // ||A||_1 (max column sum) and ||A||_inf (max row sum); A > 0.
            float cmax = 0.f, rmax = 0.f;
            for (int j = lane; j < m; j += 32) {
                float cs = 0.f, rsum = 0.f;
#pragma unroll 4
                for (int i = 0; i < m; ++i) {
                    cs += A[i * MS + j];
                    rsum += A[j * MS + i];
                }
                cmax = fmaxf(cmax, cs);
                rmax = fmaxf(rmax, rsum);
            }
            cmax = warp_max(cmax);
            rmax = warp_max(rmax);
            const float alpha = 1.f / (cmax * rmax);
            // up to 16 landmarks one warp keeps all tiles busy, without CTA barriers
            if constexpr (MP <= 16) core<MP, true>(A, alpha, Wt, Yt, c4, m, m4, iters, lane, 32);
            else if (lane == 0) red[0] = alpha;
        }
        __syncthreads();
        if constexpr (MP > 16) {
            core<MP, false>(A, red[0], Wt, Yt, c4, m, m4, iters, tid, nth);
            __syncthreads();
        }

        // ---- pass 3: G_L^n and the normalised output ----
        for (int c0 = 0; c0 < N; c0 += ch) {
            const int nt = min(ch, N - c0), tg = (nt + 3) >> 2;
            load_rows<T>(qu + (size_t)c0 * d, nt, tg, d, 4 * kg, pl, put_rows);
            __syncthreads();
            float s[4][4];
            scores(kbar, tg, nt, bLu ? bLu + (size_t)c0 * m : nullptr, 1, m, s);
            float yd[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) yd[j] = j0 + j * JG < m ? Yt[d * MS + j0 + j * JG] : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float mx = fmaxf(fmaxf(s[i][0], s[i][1]), fmaxf(s[i][2], s[i][3])), den = 0.f;
#pragma unroll
                for (int o = JG >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float p = j0 + j * JG < m ? expf(s[i][j] - mx) : 0.f;
                    den = fmaf(p, yd[j], den);
                    if (t0 < tg) P[(t0 + i * tg) * MS + j0 + j * JG] = p;
                }
#pragma unroll
                for (int o = JG >> 1; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
                if (j0 == 0 && t0 < tg) rowv[t0 + i * tg] = 1.f / den;
            }
            __syncthreads();
            for (int it = tid; it < tg * kg; it += nth) {  // over the Q rows, which the scores have read
                const int r = it / kg, c = 4 * (it - r * kg);
                f32x2 acc[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
                tile_nt<4, 4>(P + r * MS, tg * MS, Yt + c * MS, MS, m4 >> 2, acc);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float inv = rowv[r + i * tg];
                    *reinterpret_cast<float4*>(KV + (r + i * tg) * DS + c) =
                        make_float4(sum2(acc[i][0]) * inv, sum2(acc[i][1]) * inv, sum2(acc[i][2]) * inv,
                                    sum2(acc[i][3]) * inv);
                }
            }
            __syncthreads();
            {
                const int c = 2 * (tid & ((1 << pl) - 1));
                T* oc = ou + (size_t)c0 * d;
                if (c < d)
                    for (int r = tid >> pl; r < nt; r += nth >> pl) {
                        const float2 x = *reinterpret_cast<const float2*>(KV + r * DS + c);
                        st_pair<T>(oc + (size_t)r * d, c, d, x.x, x.y);
                    }
            }
            __syncthreads();
        }
    }
}

// One kernel per type: with the three in one, the 16-bit ones' loops lay apart and
// a unit waited for instructions (12 units of 4x4 windows, d_h = 16, m = 4: fp32
// 14.4 us, bf16 19.7, by itself 14.5; of 8x8, d_h = 20, m = 4, bf16, 20.7 and 16.3).
template <int MP, int DS, typename T>
__global__ void __launch_bounds__(Bound<MP>::kThreads, Bound<MP>::kCtas)
nystra_generic_kernel(const T* q, const T* k, const T* v, T* out, long long n_units, int N, int d, int m, int iters,
                      int pw, float scale, NystraBias bias) {
    extern __shared__ __align__(16) float sm[];
    run<MP, DS, T>(q, k, v, out, n_units, N, d, m, iters, pw, scale, bias, sm);
}

template <int MP, int DS, typename T>
cudaError_t launch_ds(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d, int m,
                      int iters, int pool, cudaStream_t stream, const NystraBias& bias) {
    static std::atomic<int> s_sms[kMaxDevices];
    auto kern = nystra_generic_kernel<MP, DS, T>;
    int sms = 0;
    if (cudaError_t e = opt_in_smem(kern, s_sms, &sms); e != cudaSuccess) return e;
    int pw = 0;  // window width for square patches
    if (pool != 0)
        while ((pw + 1) * (pw + 1) <= N) ++pw;
    // Few units, up to four CTAs per SM: at least four warps, for a unit's latency
    // (108 units of 7x7 windows, m = 7: 33 us with one warp, 22 with four); else the
    // tiles' threads only, for more CTAs per SM.
    const Shape<MP, DS> G(N, d, n_units <= 4LL * sms ? 128 : 32);
    const long long grid = n_units < (1LL << 30) ? n_units : (1LL << 30);
    kern<<<(unsigned)grid, G.threads, G.bytes(), stream>>>((const T*)q, (const T*)k, (const T*)v, (T*)out, n_units, N, d,
                                                           m, iters, pw, 1.0f / sqrtf((float)d), bias);
    return cudaGetLastError();
}

// m <= MP.  Row strides: the d_h columns and (V's) one more, in an odd number
// of granules: up to 19, 35 and 67 columns.
template <int MP, typename T>
cudaError_t launch_t(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d, int m,
                     int iters, int pool, cudaStream_t stream, const NystraBias& bias) {
    if (d < 20) return launch_ds<MP, 20, T>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
    if (d < 36) return launch_ds<MP, 36, T>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
    return launch_ds<MP, 68, T>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
}

template <int MP>
cudaError_t launch(const void* q, const void* k, const void* v, void* out, long long n_units, int N, int d, int m,
                   int iters, int pool, int dtype, cudaStream_t stream, const NystraBias& bias) {
    if (dtype == 0) return launch_t<MP, float>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
    if (dtype == 1) return launch_t<MP, __nv_bfloat16>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
    return launch_t<MP, __half>(q, k, v, out, n_units, N, d, m, iters, pool, stream, bias);
}

}  // namespace generic
}  // namespace nystra

// One translation unit per landmark bound.
#define NYSTRA_GENERIC_DEFINE(MP)                                                                                \
    namespace nystra_host {                                                                                      \
    cudaError_t launch_nystra_generic_m##MP(const void* q, const void* k, const void* v, void* out,              \
                                            long long n_units, int N, int d, int m, int iters, int pool,         \
                                            int dtype, cudaStream_t stream, const nystra::NystraBias& bias) {    \
        return nystra::generic::launch<MP>(q, k, v, out, n_units, N, d, m, iters, pool, dtype, stream, bias);    \
    }                                                                                                            \
    }
