// FP32 block kernels shared by the dense products (la.cu) and the H-matrix
// level products (hmatrix.cu).
#pragma once

#include "lsw_internal.cuh"

namespace lsw {

// out (m x n, column-major) = A^H B over `rows` rows (A: m columns, ld lda; B:
// n columns, ld ldb), m, n <= 64, by a CTA of 256 threads.  Rows go through
// shared memory in tiles of 32, stored row-major with odd strides (conflict-
// free transposing stores); a thread keeps MA x 4 outputs, ti + mtr a,
// tj + mtn b (a warp's loads are contiguous), over every G-th row of a tile,
// and the row groups are summed in shared memory at the end.  MA = 8 makes an
// inner step 128 multiply-adds on 12 loads (4 x 4 blocks, 64 on 8, are bound
// by shared-memory wavefronts); MA = 5 wastes less where m is 10, 20, 30 or
// so, the usual ranks (cn_block_ma).  The next tile is fetched into registers
// during the products.  NPRE >= max(m rounded up, n) / 8.
template <int NPRE, int MA>
__device__ __forceinline__ void cn_block_f32(int m, int n, const float2* __restrict__ A, long long lda,
                                             const float2* __restrict__ B, long long ldb, int rows, float2* sm,
                                             float2* __restrict__ out) {
    constexpr int TR = 32;
    const int ms = (m + MA - 1) / MA * MA, ns = (n + 3) & ~3;
    const int asd = ms + 1, bsd = ns + 1;
    float2* As = sm;
    float2* Bs = As + TR * asd;
    float2* Red = As;                               // G x m x n, after the products
    const int mtr = ms / MA, mtn = ns / 4, nmt = mtr * mtn;
    const int G = min(TR, 256 / nmt);
    const int mt = threadIdx.x % nmt, rg = threadIdx.x / nmt;
    const bool active = rg < G;
    const int ti = mt % mtr, tj = mt / mtr;
    float2 acc[MA][4];
#pragma unroll
    for (int a = 0; a < MA; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = make_float2(0.f, 0.f);
    // tile entry: row rr0 of columns cc0 + 8 u
    const int rr0 = threadIdx.x & 31, cc0 = threadIdx.x >> 5;
    float2 pa[NPRE], pb[NPRE];
    auto fetch = [&](int r0) {
        const int r = r0 + rr0;
#pragma unroll
        for (int u = 0; u < NPRE; ++u) {
            const int cc = cc0 + 8 * u;
            pa[u] = r < rows && cc < m ? A[cc * lda + r] : make_float2(0.f, 0.f);
            pb[u] = r < rows && cc < n ? B[cc * ldb + r] : make_float2(0.f, 0.f);
        }
    };
    fetch(0);
    for (int r0 = 0; r0 < rows; r0 += TR) {
#pragma unroll
        for (int u = 0; u < NPRE; ++u) {
            const int cc = cc0 + 8 * u;
            if (cc < ms) As[rr0 * asd + cc] = pa[u];
            if (cc < ns) Bs[rr0 * bsd + cc] = pb[u];
        }
        __syncthreads();
        if (r0 + TR < rows) fetch(r0 + TR);
        if (active) {
            for (int rr = rg; rr < TR; rr += G) {
                float2 x[MA], y[4];
#pragma unroll
                for (int a = 0; a < MA; ++a) x[a] = As[rr * asd + ti + mtr * a];
#pragma unroll
                for (int c = 0; c < 4; ++c) y[c] = Bs[rr * bsd + tj + mtn * c];
#pragma unroll
                for (int a = 0; a < MA; ++a)
#pragma unroll
                    for (int c = 0; c < 4; ++c) cfmac(acc[a][c], x[a], y[c]);
            }
        }
        __syncthreads();
    }
    const int nout = m * n;
    if (active) {
#pragma unroll
        for (int a = 0; a < MA; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int i = ti + mtr * a, j = tj + mtn * c;
                if (i < m && j < n) Red[(long long)rg * nout + j * m + i] = acc[a][c];
            }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nout; e += 256) {
        float2 sacc = make_float2(0.f, 0.f);
        for (int g = 0; g < G; ++g) sacc = cadd(sacc, Red[(long long)g * nout + e]);
        out[e] = sacc;
    }
}

// Outputs per thread along m: the choice with the larger useful share of the
// CTA's multiply-adds (columns beyond m, idle threads, rows beyond the tile's
// last full round), MA = 5 counted at 0.85 for its 9 loads per 80.
inline int cn_block_ma(int m, int n) {
    const int ns = (n + 3) & ~3;
    auto share = [&](int ma) {
        const int ms = (m + ma - 1) / ma * ma, nmt = (ms / ma) * (ns / 4);
        const int q = 256 / nmt, G = q < 32 ? q : 32;
        return (double)m / ms * (G * nmt / 256.0) * (32.0 / (G * ((32 + G - 1) / G)));
    };
    return 0.85 * share(5) > share(8) ? 5 : 8;
}

// columns to fetch per thread (NPRE) and shared memory (at most 66 KB)
inline int cn_block_npre(int m, int n, int ma) {
    const int ms = (m + ma - 1) / ma * ma, ns = (n + 3) & ~3, most = ms > ns ? ms : ns;
    return most <= 16 ? 2 : most <= 32 ? 4 : 9;
}
inline size_t cn_block_smem(int m, int n, int ma) {
    const int ms = (m + ma - 1) / ma * ma, ns = (n + 3) & ~3;
    const int q = 256 / ((ms / ma) * (ns / 4)), G = q < 32 ? q : 32;
    const size_t tiles = 32 * (size_t)(ms + ns + 2), red = (size_t)G * m * n;
    return sizeof(float2) * (tiles > red ? tiles : red);
}

}  // namespace lsw
