// The m x m core of m = 32 and 64 on CW = m/16 warps, with symmetric products.
// Included by nystra_tc.cuh after the one-warp core, whose fragment helpers it
// uses.
#pragma once

#include "ptx.cuh"

namespace nystra {
namespace tc {

// The m x m operands no longer fit one warp's registers: warp c owns rows 16c ..
// 16c + 15.  The arithmetic is core_warp's: X = A Z_k and Z are carried, T2 = 15I -
// 7X + XX, T3 = 13I - X T2, Z <- Z T3/4, X <- X T3/4.  T2, T3 and X are
// polynomials in X_0 = a A A^T and symmetric: of a warp's 2 CW tiles of 16 x 8 in
// each of their products only one triangle's CW + 1 are computed, and mirrored,
// which also removes antisymmetric round-off (m = 64: 23 tile products per warp
// and step instead of 32; m = 32: 13 instead of 16).  Z's own rows stay in
// registers at a power of two per warp, so no step needs a maximum over the
// warps.
//
// A warp computes its diagonal block (two tiles), m = 64: the block to its right,
// cyclically (two tiles), and one tile of the blocks two apart (m = 32: of the
// only off-diagonal block), whose left rows it keeps as a second A operand.  X's
// k-blocks and Z's tiles are taken in the cyclic order of those columns, so that
// register indexes are constant.
//
// Right factors are read from two shared-memory matrices (hi and lo planes,
// rows padded to m + 8 halves so ldmatrix is conflict-free) that alternate
// roles: X in one, -T2/4 in the other, T3/4 over X once every warp has used X,
// the next X over -T2/4 once every warp has used it; three barriers per step.
// Z is carried in fp32 between the steps (and split at a power of two per warp
// for its product), and Y = Z W is a split-tf32 product of fp32 Z and W: neither
// factor's entries have a bounded range, and both parts of a tf32 split have
// fp32's exponent, while fp16 pairs lose bits of entries 2^13 below the largest.
//
// What bounds it: the tensor pipe's mma.sync rate and, between two barriers,
// a chain of 6 or 12 dependent MMAs with the split and store of their results.
// Measured (bf16) against full products and scales agreed on over the warps:
// m = 64, 4096 units of 16x16 windows, d_h = 32, 925 -> 452 us (in the wide
// kernel, with three groups per SM instead of two), 1024 of 32x32 499 -> 377;
// m = 32, 8192 units of 16x16, d_h = 30, 354 -> 283 us (d_h = 32 now in the team
// kernel too: 560 -> 294); 1024 units of 32x32, d_h = 32, 145 -> 133, the step mostly
// in the token loads.  Y = Z W from fp16 pairs, W's scaled by a power of two per
// column, was no faster (453, 372, 292, 306 and 135 us).  At m = 64, carrying V = Z W
// instead (V <- T3 V/4 with X = Z A: d_h + 1 columns instead of m, 20 tile
// products a step, but V's column scales to agree on in every step) took 0.51 and
// 0.46 ms, and was less accurate: under sharp attention (logit std 4) its
// error was up to twice as large, since Z T3 meets W's small parts exactly.

template <int M>
__device__ __forceinline__ void sc_store(unsigned char* mat, int row, int col, const H2Pair& p) {
    constexpr int SS = ScScratch<M>::SS;
    *reinterpret_cast<uint32_t*>(mat + ((size_t)row * SS + col) * 2) = p.hi;
    *reinterpret_cast<uint32_t*>(mat + ScScratch<M>::PLANE + ((size_t)row * SS + col) * 2) = p.lo;
}

// Own rows of acc (already scaled) into a scratch matrix.
template <int M>
__device__ __forceinline__ void sc_put(unsigned char* mat, const float (&acc)[M / 8][4], int c, int g, int t) {
#pragma unroll
    for (int n = 0; n < M / 8; ++n) {
        sc_store<M>(mat, 16 * c + g, 8 * n + 2 * t, split_h2(acc[n][0], acc[n][1]));
        sc_store<M>(mat, 16 * c + g + 8, 8 * n + 2 * t, split_h2(acc[n][2], acc[n][3]));
    }
}

// The tiles of one warp (see above): columns 8 n(i) .. 8 n(i) + 7 of its own
// rows for i < OWN, of row block r5 for the last.
template <int M>
struct ScTiles {
    static constexpr int CW = M / 16, N = CW + 1, OWN = N - 1;
    static_assert(CW == 4 || CW == 2, "the splits are those of four and two row blocks");
    int c, r5, b5, h5;  // own block; the last tile's row block, column block and half
    __device__ __forceinline__ explicit ScTiles(int c_) : c(c_) {
        r5 = CW == 4 ? (c & 1) : 0;
        b5 = CW == 4 ? r5 + 2 : 1;
        h5 = CW == 4 ? (c >> 1) : c;
    }
    __device__ __forceinline__ int row(int i) const { return i < OWN ? c : r5; }
    __device__ __forceinline__ int col(int i) const { return i < OWN ? 2 * ((c + i / 2) % CW) + (i & 1) : 2 * b5 + h5; }
};

// The symmetric matrix of which acc (scaled by s) holds this warp's tiles.
template <int M>
__device__ __forceinline__ void sc_put_sym(unsigned char* mat, const float (&acc)[M / 16 + 1][4], float s,
                                             const ScTiles<M>& tl, int g, int t, uint32_t sel) {
#pragma unroll
    for (int i = 0; i < ScTiles<M>::N; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int R = 2 * tl.row(i) + h, n = tl.col(i);  // 8x8 block (R, n)
            if (i < 2 && h < i) continue;                    // the diagonal block's upper right quarter
            H2Pair p = split_h2(s * acc[i][2 * h], s * acc[i][2 * h + 1]);
            const H2Pair q = {movmatrix_trans(p.hi), movmatrix_trans(p.lo)};
            if (i < 2 && h == i) {  // on the diagonal: mirror the lower triangle
                p.hi = prmt(p.hi, q.hi, sel);
                p.lo = prmt(p.lo, q.lo, sel);
            } else {
                sc_store<M>(mat, 8 * n + g, 8 * R + 2 * t, q);
            }
            sc_store<M>(mat, 8 * R + g, 8 * n + 2 * t, p);
        }
}

// A operand of row block rb (TR: of the transpose's) from a scratch matrix,
// k-step j = block (b0 + j) mod CW.
template <int M, bool TR>
__device__ __forceinline__ void sc_load_a(const unsigned char* mat, H2Pair (&a)[M / 16][4], int rb, int b0,
                                            int lane) {
    constexpr int SS = ScScratch<M>::SS, CW = M / 16;
    const int blk = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int j = 0; j < CW; ++j) {
        const int kk = (b0 + j) % CW;
        const int row = TR ? 16 * kk + 8 * (blk >> 1) + rr : 16 * rb + 8 * (blk & 1) + rr;
        const int col = TR ? 16 * rb + 8 * (blk & 1) : 16 * kk + 8 * (blk >> 1);
        uint32_t h[4], l[4];
        const unsigned char* ph = mat + ((size_t)row * SS + col) * 2;
        if (TR) {
            ldsm_x4_t(h, ph);
            ldsm_x4_t(l, ph + ScScratch<M>::PLANE);
        } else {
            ldsm_x4(h, ph);
            ldsm_x4(l, ph + ScScratch<M>::PLANE);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) a[j][r] = H2Pair{h[r], l[r]};
    }
}

// D[i] += A_i B_i over the pair's significant products (lo hi, hi lo, hi hi),
// tile by tile within each so that consecutive MMAs are independent.
template <int NTL>
__device__ __forceinline__ void sc_mma(float (*const (&D)[NTL])[4], const H2Pair (*const (&A)[NTL])[4],
                                         const uint32_t (*const (&bh)[NTL]), const uint32_t (*const (&bl)[NTL])) {
    using H = Mma16<__half>;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int i = 0; i < NTL; ++i) {
            const H2Pair(&a)[4] = *A[i];
            const uint32_t hi[4] = {a[0].hi, a[1].hi, a[2].hi, a[3].hi}, lo[4] = {a[0].lo, a[1].lo, a[2].lo, a[3].lo};
            const uint32_t* b = p == 1 ? bl[i] : bh[i];
            if (p == 0) H::k16(*D[i], lo, b[0], b[1]);
            else H::k16(*D[i], hi, b[0], b[1]);
        }
}

// This warp's tiles of A P^T (P in mat): acc += ...; Ao, A5: A operands of the
// own rows and of row block r5, in the cyclic k order of sc_load_a from block c
// and b5.
template <int M>
__device__ __forceinline__ void sc_sym_mm(const H2Pair (&Ao)[M / 16][4], const H2Pair (&A5)[M / 16][4],
                                          const unsigned char* mat, float (&acc)[M / 16 + 1][4],
                                          const ScTiles<M>& tl, int lane) {
    constexpr int SS = ScScratch<M>::SS, CW = M / 16, OWN = CW;
    constexpr size_t PL = ScScratch<M>::PLANE;
    const int blk = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int j = 0; j < CW; ++j) {
        // B fragments of the own tiles, two at a time (16 columns), and of the last tile
        uint32_t bh[OWN / 2][4], bl[OWN / 2][4], eh[2], el[2];
        const int kk = (tl.c + j) % CW, k5 = (tl.b5 + j) % CW;
#pragma unroll
        for (int p = 0; p < OWN / 2; ++p) {
            const int cb = (tl.c + p) % CW;
            const unsigned char* ph = mat + ((size_t)(16 * cb + 8 * (blk >> 1) + rr) * SS + 16 * kk + 8 * (blk & 1)) * 2;
            ldsm_x4(bh[p], ph);
            ldsm_x4(bl[p], ph + PL);
        }
        const unsigned char* p5 = mat + ((size_t)(8 * tl.col(OWN) + rr) * SS + 16 * k5 + 8 * (blk & 1)) * 2;
        ldsm_x2(eh, p5);
        ldsm_x2(el, p5 + PL);
        float(*D[OWN + 1])[4];
        const H2Pair(*A[OWN + 1])[4];
        const uint32_t *ph[OWN + 1], *pl[OWN + 1];
#pragma unroll
        for (int i = 0; i < OWN; ++i) {
            D[i] = &acc[i];
            A[i] = &Ao[j];
            ph[i] = bh[i / 2] + 2 * (i & 1);
            pl[i] = bl[i / 2] + 2 * (i & 1);
        }
        D[OWN] = &acc[OWN];
        A[OWN] = &A5[j];
        ph[OWN] = eh;
        pl[OWN] = el;
        sc_mma<OWN + 1>(D, A, ph, pl);
    }
}

// All tiles of the own rows of A P^T (P in mat), column block (c + i / 2) mod CW
// in tiles i, i + 1: acc = A P^T; A in the cyclic k order from block c, as the
// C-layout tiles of such a product hold it.
template <int M>
__device__ __forceinline__ void sc_row_mm(const H2Pair (&A)[M / 16][4], const unsigned char* mat,
                                          float (&acc)[M / 8][4], int c, int lane) {
    constexpr int SS = ScScratch<M>::SS, CW = M / 16, NT = M / 8;
    constexpr size_t PL = ScScratch<M>::PLANE;
    const int blk = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int i = 0; i < NT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll
    for (int j = 0; j < CW; ++j) {
        const int kk = (c + j) % CW;
#pragma unroll
        for (int q = 0; q < CW; q += 2) {  // four tiles at a time
            uint32_t bh[2][4], bl[2][4];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int cb = (c + q + p) % CW;
                const unsigned char* ph =
                    mat + ((size_t)(16 * cb + 8 * (blk >> 1) + rr) * SS + 16 * kk + 8 * (blk & 1)) * 2;
                ldsm_x4(bh[p], ph);
                ldsm_x4(bl[p], ph + PL);
            }
            float(*D[4])[4];
            const H2Pair(*Ap[4])[4];
            const uint32_t *ph[4], *pl[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                D[i] = &acc[2 * q + i];
                Ap[i] = &A[j];
                ph[i] = bh[i / 2] + 2 * (i & 1);
                pl[i] = bl[i / 2] + 2 * (i & 1);
            }
            sc_mma<4>(D, Ap, ph, pl);
        }
    }
}

// x as two tf32 values, both rounded to nearest: hi + lo equals x to within
// 2^-22 |x| (a NaN stays one in lo).
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
    hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi)) + 0x1000u;  // (the tensor core ignores the low bits)
}

// Own rows of Z W: acc = z W, z as sc_row_mm leaves it, W fp32 with row stride
// NCOL + 4 (so that a B fragment's loads fall into 32 banks).  A step of eight
// landmarks takes columns 2t and 2t + 1 of z's tile as its k = t and t + 4, and
// the rows of W likewise.
template <int M, int NCOL>
__device__ __forceinline__ void sc_w_mm(const float (&z)[M / 8][4], const float* W, float (&acc)[NCOL / 8][4], int c,
                                        int g, int t) {
    constexpr int WS = NCOL + 4, CW = M / 16, NTO = NCOL / 8;
#pragma unroll
    for (int n = 0; n < NTO; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
    for (int i = 0; i < M / 8; ++i) {
        uint32_t ah[4], al[4], bh[NTO][2], bl[NTO][2];
#pragma unroll
        for (int e = 0; e < 4; ++e) split_tf32(z[i][2 * (e & 1) + (e >> 1)], ah[e], al[e]);
        const float* w = W + (16 * ((c + i / 2) % CW) + 8 * (i & 1) + 2 * t) * WS + g;
#pragma unroll
        for (int n = 0; n < NTO; ++n) {
            split_tf32(w[8 * n], bh[n][0], bl[n][0]);
            split_tf32(w[8 * n + WS], bh[n][1], bl[n][1]);
        }
#pragma unroll
        for (int n = 0; n < NTO; ++n) mma_tf32(acc[n], al[0], al[1], al[2], al[3], bh[n][0], bh[n][1]);
#pragma unroll
        for (int n = 0; n < NTO; ++n) mma_tf32(acc[n], ah[0], ah[1], ah[2], ah[3], bl[n][0], bl[n][1]);
#pragma unroll
        for (int n = 0; n < NTO; ++n) mma_tf32(acc[n], ah[0], ah[1], ah[2], ah[3], bh[n][0], bh[n][1]);
    }
}

// Core on CW = M/16 warps (warp c of them calls with its index; bar_id is a
// named barrier reserved for these warps; mat0, mat1, aux: ScScratch areas):
// G_A^n from the landmarks and the m_U of the own rows (mu0, mu1: rows 16c + g
// and + 8, log2 domain), the iteration of step 4, Y = Z W (W: fp32, row stride
// NCOL + 4) stored as Y^T at yT, or where yT is null over the scratch matrix that
// is free by then; returns its place.  WREG: w holds the own rows of W on entry
// (C layout), and W, which may overlay Qbar, is first written after every warp
// has read its rows.  yT may overlay W.  As in core_warp, A is split at 2^ea
// with its largest entry in [2^10, 2^11); X, -T2/4 and T3/4 are split at the
// fixed scale 2^10 (their entries stay within a few units, since X's
// eigenvalues lie in [0, 1]).  Scalar factors of Z cancel in step 7 and are
// dropped; the warps' powers of two are taken back.
template <typename T, int M, int NCOL, bool WREG>
__device__ __forceinline__ T* sc_core(const T* qbar, const T* kbar, float mu0, float mu1, float (&w)[NCOL / 8][4],
                                      T* yT, unsigned char* mat0, unsigned char* mat1, float* W, float* aux, int iters,
                                      float sl2, int c, int lane, int bar_id) {
    using S = ScScratch<M>;
    using O = Opnd<T>;
    using D = typename O::DReg;
    constexpr int CW = S::CW, KT = M / 16, NT = M / 8, LS = LmS<T>::LS, LO = LmS<T>::LO, NTO = NCOL / 8,
                  YS = YtS<T, M>::YS, YLO = YtS<T, M>::LO, NTL = ScTiles<M>::N;
    const int g = lane >> 2, t = lane & 3;
    unsigned char* cur = mat0;
    unsigned char* oth = mat1;
    float* cols = aux;                // [CW][M] column-sum partials
    float* slots = aux + CW * M;      // [4][CW] maxima
    auto csync = [&]() { named_barrier(bar_id, CW * 32); };
    const uint32_t sel = tril_selector(g, t);
    const ScTiles<M> tl(c);
    constexpr float kS = 1024.f, kS2 = 1048576.f;  // fixed scale 2^10 of X, -T2/4, T3/4 (and its square)
    H2Pair Xa[KT][4], X5[KT][4];
    float acc[NTL][4], z[NT][4];  // z: the own rows of 2^ez Z, tiles as in sc_row_mm
    int ez = 0;
    float alpha;  // a A A^T = alpha (2^ea A)(2^ea A)^T
    {
        float a[NT][4];
        // ---- G_A^n's own rows ----
        {
            D aq[2][4];
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
                const T* r0 = qbar + (16 * c + g) * LS + 16 * kk + 2 * t;
                aq[kk][0] = DSt<T>::ld(r0, LO);
                aq[kk][1] = DSt<T>::ld(r0 + 8 * LS, LO);
                aq[kk][2] = DSt<T>::ld(r0 + 8, LO);
                aq[kk][3] = DSt<T>::ld(r0 + 8 * LS + 8, LO);
            }
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                float sa[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                    const T* kr = kbar + (8 * n + g) * LS + 16 * kk + 2 * t;
                    O::mma(sa, aq[kk], DSt<T>::ld(kr, LO), DSt<T>::ld(kr + 8, LO));
                }
                a[n][0] = fmaf(sa[0], sl2, -mu0);  // log2 of G_A^n
                a[n][1] = fmaf(sa[1], sl2, -mu0);
                a[n][2] = fmaf(sa[2], sl2, -mu1);
                a[n][3] = fmaf(sa[3], sl2, -mu1);
            }
        }
        // 2^ea G_A^n with its largest entry in [2^10, 2^11) (the shift enters the
        // exponent, as in core_warp)
        {
            float lm = -INFINITY;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) lm = fmaxf(lm, a[n][e]);
            lm = warp_max_f(lm);
            if (lane == 0) slots[3 * CW + c] = lm;
            csync();  // every warp has read its rows of Qbar
            float lmax = -INFINITY;
#pragma unroll
            for (int x = 0; x < CW; ++x) lmax = fmaxf(lmax, slots[3 * CW + x]);
            const float fa = (lmax > -INFINITY && lmax < INFINITY) ? (float)(10 - (int)floorf(lmax)) : 0.f;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[n][e] = ex2(a[n][e] + fa);
        }
        // ---- ||A||_inf, ||A||_1 (A > 0), A and W into scratch ----
        {
            float r0 = 0.f, r1 = 0.f;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                r0 += a[n][0] + a[n][1];
                r1 += a[n][2] + a[n][3];
            }
            r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
            r0 += __shfl_xor_sync(0xffffffffu, r0, 2);
            r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
            r1 += __shfl_xor_sync(0xffffffffu, r1, 2);
            const float rm = warp_max_nonneg(fmaxf(r0, r1));
            if (lane == 0) slots[c] = rm;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float cs = a[n][e] + a[n][e + 2];
                    cs += __shfl_xor_sync(0xffffffffu, cs, 4);
                    cs += __shfl_xor_sync(0xffffffffu, cs, 8);
                    cs += __shfl_xor_sync(0xffffffffu, cs, 16);
                    if (g == 0) cols[c * M + 8 * n + 2 * t + e] = cs;
                }
        }
        sc_put<M>(cur, a, c, g, t);  // 2^ea A
        if constexpr (WREG) {
#pragma unroll
            for (int n = 0; n < NTO; ++n)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<float2*>(W + (16 * c + g + 8 * h) * (NCOL + 4) + 8 * n + 2 * t) =
                        make_float2(w[n][2 * h], w[n][2 * h + 1]);
        }
        csync();
        float rmax = 0.f, cmax = 0.f;
#pragma unroll
        for (int x = 0; x < CW; ++x) rmax = fmaxf(rmax, slots[x]);
        for (int col = lane; col < M; col += 32) {
            float cs = 0.f;
#pragma unroll
            for (int x = 0; x < CW; ++x) cs += cols[x * M + col];
            cmax = fmaxf(cmax, cs);
        }
        alpha = 1.f / (rmax * warp_max_nonneg(cmax));
    }
    auto zero = [&]() {
#pragma unroll
        for (int i = 0; i < NTL; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    };
    auto add_diag = [&](float s) {  // acc += s I
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (8 * (e >> 1) + g == 8 * i + (e & 1) + 2 * t) acc[i][e] += s;
    };
    // C-layout entries (rows 8h + g, columns 2t, 2t + 1 of half n of k-step kk) of an A operand
    auto entries = [&](const H2Pair (&a)[KT][4], int kk, int n, int h) -> float2 {
        const H2Pair p = n == 0 ? a[kk][h] : a[kk][2 + h];
        const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&p.hi));
        const float2 y = __half22float2(*reinterpret_cast<const __half2*>(&p.lo));
        return make_float2(x.x + y.x, x.y + y.y);
    };
    // ---- Z_0 = (2^ea A)^T (a and 2^ea dropped), X_0 = alpha (2^ea A)(2^ea A)^T ----
    sc_load_a<M, false>(cur, Xa, c, c, lane);
    sc_load_a<M, false>(cur, X5, tl.r5, tl.b5, lane);
    zero();
    sc_sym_mm<M>(Xa, X5, cur, acc, tl, lane);
    {
        H2Pair Za[KT][4];
        sc_load_a<M, true>(cur, Za, c, c, lane);
#pragma unroll
        for (int j = 0; j < KT; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float2 v = entries(Za, j, r >> 1, r & 1);
                z[2 * j + (r >> 1)][2 * (r & 1)] = v.x;
                z[2 * j + (r >> 1)][2 * (r & 1) + 1] = v.y;
            }
    }
    sc_put_sym<M>(oth, acc, kS * alpha, tl, g, t, sel);  // kS X_0
    csync();
    {
        unsigned char* tmp = cur;
        cur = oth;
        oth = tmp;
    }
    // ---- iteration (step 4): X in cur ----
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        sc_load_a<M, false>(cur, Xa, c, c, lane);
        sc_load_a<M, false>(cur, X5, tl.r5, tl.b5, lane);
        // kS^2 T2 = kS^2 (15I - 7X + X X); X's entries of a tile are its k-step i / 2's (the last tile's: 0's)
#pragma unroll
        for (int i = 0; i < NTL; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 x;
                if (i < NTL - 1) x = entries(Xa, i / 2, i & 1, h);
                else {
                    const float2 x0 = entries(X5, 0, 0, h), x1 = entries(X5, 0, 1, h);
                    x = tl.h5 ? x1 : x0;
                }
                acc[i][2 * h] = -7.f * kS * x.x;
                acc[i][2 * h + 1] = -7.f * kS * x.y;
            }
        add_diag(15.f * kS2);
        sc_sym_mm<M>(Xa, X5, cur, acc, tl, lane);
        sc_put_sym<M>(oth, acc, -0.25f / kS, tl, g, t, sel);  // kS (-T2/4)
        csync();
        zero();
        add_diag(3.25f * kS2);
        sc_sym_mm<M>(Xa, X5, oth, acc, tl, lane);          // kS^2 T3/4
        sc_put_sym<M>(cur, acc, 1.f / kS, tl, g, t, sel);  // kS T3/4 (every warp is done with X)
        csync();
        const bool more = it + 1 < iters;
        if (more) {
            zero();
            sc_sym_mm<M>(Xa, X5, cur, acc, tl, lane);          // kS^2 X T3/4
            sc_put_sym<M>(oth, acc, 1.f / kS, tl, g, t, sel);  // every warp is done with -T2/4
        }
        {
            float zm = 0.f;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) zm = fmaxf(zm, fabsf(z[n][e]));
            const int e = h2_exponent(warp_max_nonneg(zm));
            const float s = pow2i(e);
            ez += e + 10;  // and kS
            H2Pair Za[KT][4];
#pragma unroll
            for (int j = 0; j < KT; ++j)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int n = 2 * j + (r >> 1), v = 2 * (r & 1);
                    Za[j][r] = split_h2(s * z[n][v], s * z[n][v + 1]);
                }
            sc_row_mm<M>(Za, cur, z, c, lane);  // kS Z T3/4
        }
        if (more) {
            csync();
            unsigned char* tmp = cur;
            cur = oth;
            oth = tmp;
        }
    }
    // ---- Y = Z W, own rows, without the warp's power of two, stored as Y^T ----
    sc_w_mm<M, NCOL>(z, W, w, c, g, t);
    const float sz = pow2i(-ez);
#pragma unroll
    for (int n = 0; n < NTO; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) w[n][e] *= sz;
    float scale = 1.f;
    if (O::kNarrowRange) {
        float ym = 0.f;
#pragma unroll
        for (int j = 0; j < NTO; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) ym = fmaxf(ym, fabsf(w[j][e]));
        ym = warp_max_nonneg(ym);
        if (lane == 0) slots[2 * CW + c] = ym;
        csync();
        float ymax = 0.f;
#pragma unroll
        for (int x = 0; x < CW; ++x) ymax = fmaxf(ymax, slots[2 * CW + x]);
        if (ymax > 0.f && ymax < INFINITY) scale = pow2i(14 - ilogbf(ymax));
    } else if (yT) csync();  // Y^T may overlay W, which every warp reads in full
    // free: after the last step -T2/4's matrix (its readers have passed a
    // barrier since), without steps A's
    if constexpr (YtS<T, M>::bytes(NCOL) <= S::MAT)  // (m = 32: the caller has a place)
        if (!yT) yT = reinterpret_cast<T*>(oth);
#pragma unroll
    for (int j = 0; j < NTO; ++j) {
        const int rr = 16 * c + g, cc = 8 * j + 2 * t;
        DSt<T>::put(yT + cc * YS + rr, YLO, w[j][0] * scale);
        DSt<T>::put(yT + (cc + 1) * YS + rr, YLO, w[j][1] * scale);
        DSt<T>::put(yT + cc * YS + rr + 8, YLO, w[j][2] * scale);
        DSt<T>::put(yT + (cc + 1) * YS + rr + 8, YLO, w[j][3] * scale);
    }
    return yT;
}

}  // namespace tc
}  // namespace nystra
