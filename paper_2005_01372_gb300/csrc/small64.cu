// FP64 arithmetic of the randomized sketches (Algorithm 1/2): the Gram
// matrices of sketch blocks, the thin QR of the complex64 sketches by
// shifted Cholesky QR, and the Hermitian eigen-decomposition of the small
// Gram matrix that truncates Q Yt^H to rank r.  The tall factors (Y, Q, Yt)
// stay in the working precision; every k x k matrix derived from them
// (k <= 64 columns) is formed and factored with FP64 accuracy.
//
// FP64 on this GPU runs at 1/62 of the FP32 rate (1.25 against 78 TFLOP/s,
// measured) and its dependent chains are slow, so long serial FP64 code is
// avoided: the Gram of a complex64 block is accumulated with
// error-free transformations in FP32 arithmetic: every product a*b is split
// exactly into p + e (p = fl(a b), e = fma(a, b, -p)) and summed with
// TwoSum, which is Dot2 of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26,
// 2005): over a tile of 32 rows the result is as accurate as a sum in twice
// the working precision; tiles and row chunks are then added in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>

#include "lsw_internal.cuh"

namespace lsw {

namespace {

constexpr int GT_ROWS = 32;   // rows per tile (one compensated sum)
constexpr int GT_MAXQ = 9;    // pairs per thread: 256 * 9 >= 64 * 65 / 2

// Row chunks per block for the Gram and the product kernels: down to one
// tile of 32 rows per CTA, about 1216 CTAs (8 per SM) over the batch, so
// that a few small blocks (the recompressions on the inversion's critical
// path) still spread over the GPU.
int sketch_chunks(int m, int batch) {
    return std::max(1, std::min((m + GT_ROWS - 1) / GT_ROWS, std::max(1, 1216 / batch)));
}

int grid_small(long long n, int bs = 256) {
    long long g = (n + bs - 1) / bs;
    return (int)std::max<long long>(1, std::min<long long>(g, 152LL * 32));
}

// ------------------------------------------------------ compensated Gram
// s + c accumulates a * b: p + e = a * b exactly, (s, q) = TwoSum(s, p),
// c += q + e.  The round-to-nearest intrinsics keep the compiler from
// contracting a product into a neighbouring add.
__device__ __forceinline__ void dot2(float a, float b, float& s, float& c) {
    const float p = __fmul_rn(a, b);
    const float e = __fmaf_rn(a, b, -p);
    const float t = __fadd_rn(s, p);
    const float z = __fsub_rn(t, s);
    const float q = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    s = t;
    c = __fadd_rn(c, __fadd_rn(q, e));
}

// upper-triangle pair index p -> (i, j), i <= j, p = j (j + 1) / 2 + i
__device__ __forceinline__ void tri_pair(int p, int& i, int& j) {
    int jj = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((jj + 1) * (jj + 2) / 2 <= p) ++jj;
    while (jj * (jj + 1) / 2 > p) --jj;
    j = jj;
    i = p - jj * (jj + 1) / 2;
}


// Partial Gram of rows [r0, r1) of block b: part[(b * nchunk + ch) * npair + p]
// for the upper-triangle pairs p.  Columns are staged in shared memory in
// tiles of 32 rows (odd stride: the lanes of a warp read different banks).
__global__ void __launch_bounds__(256)
k_gram_c64(const float2* __restrict__ Y, int m, int k, long long sY, int nchunk, double2* __restrict__ part,
           const int* __restrict__ active) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2* sy = reinterpret_cast<float2*>(sm_raw);   // k columns x (GT_ROWS + 1)
    const int b = blockIdx.y, ch = blockIdx.x;
    if (active && !active[b]) return;                 // this block needs no second pass
    const int rows_per = (m + nchunk - 1) / nchunk;
    const int r0 = ch * rows_per, r1 = min(m, r0 + rows_per);
    const float2* Yb = Y + (long long)b * sY;
    const int npair = k * (k + 1) / 2;
    int pi[GT_MAXQ], pj[GT_MAXQ];
    double2 acc[GT_MAXQ];
#pragma unroll
    for (int q = 0; q < GT_MAXQ; ++q) {
        const int p = threadIdx.x + q * 256;
        pi[q] = 0;
        pj[q] = 0;
        if (p < npair) tri_pair(p, pi[q], pj[q]);
        acc[q] = make_double2(0.0, 0.0);
    }
    for (int rr = r0; rr < r1; rr += GT_ROWS) {
        const int nr = min(GT_ROWS, r1 - rr);
        for (int e = threadIdx.x; e < GT_ROWS * k; e += 256) {
            const int c = e / GT_ROWS, r = e - c * GT_ROWS;
            sy[c * (GT_ROWS + 1) + r] = r < nr ? Yb[(long long)c * m + rr + r] : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < GT_MAXQ; ++q) {
            if (threadIdx.x + q * 256 < npair) {
                const float2* yi = sy + pi[q] * (GT_ROWS + 1);
                const float2* yj = sy + pj[q] * (GT_ROWS + 1);
                float sre = 0.f, cre = 0.f, sim = 0.f, cim = 0.f;
                for (int r = 0; r < nr; ++r) {
                    const float2 a = yi[r], v = yj[r];
                    // conj(a) * v = (ax vx + ay vy) + i (ax vy - ay vx)
                    dot2(a.x, v.x, sre, cre);
                    dot2(a.y, v.y, sre, cre);
                    dot2(a.x, v.y, sim, cim);
                    dot2(-a.y, v.x, sim, cim);
                }
                acc[q].x += (double)sre + (double)cre;
                acc[q].y += (double)sim + (double)cim;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < GT_MAXQ; ++q) {
        const int p = threadIdx.x + q * 256;
        if (p < npair) part[((long long)b * nchunk + ch) * npair + p] = acc[q];
    }
}

// G_b (k x k, full Hermitian, column-major) = sum over chunks, in FP64.
__global__ void k_gram_c64_reduce(const double2* __restrict__ part, int nchunk, int k, int batch, double2* G) {
    const int npair = k * (k + 1) / 2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < batch * k * k; e += gridDim.x * blockDim.x) {
        const int b = e / (k * k), ij = e - b * k * k;
        const int j = ij / k, i = ij - j * k;
        const int lo = min(i, j), hi = max(i, j);
        const int p = hi * (hi + 1) / 2 + lo;
        // eight interleaved partial sums: short FP64 dependency chains
        double2 acc[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = make_double2(0.0, 0.0);
        const double2* src = part + (long long)b * nchunk * npair + p;
        int c = 0;
        for (; c + 8 <= nchunk; c += 8) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const double2 v = src[(long long)(c + u) * npair];
                acc[u].x += v.x;
                acc[u].y += v.y;
            }
        }
        for (int u = 0; c < nchunk; ++c, ++u) {
            const double2 v = src[(long long)c * npair];
            acc[u].x += v.x;
            acc[u].y += v.y;
        }
        double2 s = make_double2(((acc[0].x + acc[1].x) + (acc[2].x + acc[3].x)) + ((acc[4].x + acc[5].x) + (acc[6].x + acc[7].x)),
                                 ((acc[0].y + acc[1].y) + (acc[2].y + acc[3].y)) + ((acc[4].y + acc[5].y) + (acc[6].y + acc[7].y)));
        if (i > j) s.y = -s.y;   // G(i, j) = conj(G(j, i))
        G[e] = s;
    }
}

// The same for many chunks of few blocks: a CTA takes 32 consecutive pairs of a
// block (contiguous in a chunk), its 32 warps every 32nd chunk (one block of
// 1024 chunks took 24 us with one thread's chain of loads per entry).
__global__ void __launch_bounds__(1024)
k_gram_c64_reduce_few(const double2* __restrict__ part, int nchunk, int k, double2* __restrict__ G) {
    __shared__ double2 red[32][33];
    const int npair = k * (k + 1) / 2, b = blockIdx.y;
    const int p = blockIdx.x * 32 + threadIdx.x;
    double2 s = make_double2(0.0, 0.0);
    if (p < npair) {
        const double2* src = part + (long long)b * nchunk * npair + p;
#pragma unroll 8
        for (int c = threadIdx.y; c < nchunk; c += 32) {
            const double2 v = src[(long long)c * npair];
            s.x += v.x;
            s.y += v.y;
        }
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    for (int h = 16; h > 0; h >>= 1) {
        if (threadIdx.y < h) {
            const double2 v = red[threadIdx.y + h][threadIdx.x];
            red[threadIdx.y][threadIdx.x].x += v.x;
            red[threadIdx.y][threadIdx.x].y += v.y;
        }
        __syncthreads();
    }
    if (threadIdx.y || p >= npair) return;
    int i, j;
    tri_pair(p, i, j);
    const double2 v = red[0][threadIdx.x];
    double2* Gb = G + (long long)b * k * k;
    Gb[j * k + i] = v;
    if (i != j) Gb[i * k + j] = make_double2(v.x, -v.y);    // G(j, i) = conj(G(i, j))
}

// ------------------------------------------- Cholesky and R^-1 (FP64)
// One CTA per matrix: G + shift I = Lt D Lt^H (Lt unit lower triangular, D
// diagonal: the square-root-free Cholesky), with Xt = Lt^-1 formed alongside,
// and R^-1 = Xt^H D^-1/2 (R = D^1/2 Lt^H, so R^H R = G + shift I).
// Written for the rate and latency of FP64 on this GPU (2 FP64 lanes per
// cycle per SM): every multiply-add a thread issues is useful (the trailing
// triangle is enumerated through a table, not masked out of a square), a
// step waits on one barrier-separated phase of independent multiply-adds,
// the pivot's reciprocal (an FP32 estimate and two Newton steps, no FP64
// division) is formed by the thread that finishes the pivot while the
// others finish the step, and the square roots of D are taken once, at the
// end, for all columns at once.
// A non-positive pivot restarts the factorisation with a larger shift
// (1e-15 tr(G) / k, then x100, at most 12 times).  A block with tr(G) = 0
// gets Rinv = 0 (its Q is zero, which the truncation keeps as a zero block).
__device__ __forceinline__ double rsqrt64(double d) {
    float f = (float)d;
    double y = (f > 1e-37f && f < 1e37f) ? (double)rsqrtf(f) : 1.0 / sqrt(d);
    // y <- y (3 - d y^2) / 2, twice: relative error ~1e-7 -> ~1e-14 -> rounding
    for (int it = 0; it < 2; ++it) {
        const double e = fma(-d * y, y, 1.0);
        y = fma(0.5 * y, e, y);
    }
    return y;
}

__device__ __forceinline__ double rcp64(double d) {
    float f = (float)d;
    double y = (f > 1e-37f && f < 1e37f) ? (double)(1.0f / f) : 1.0 / d;
    // y <- y (2 - d y), twice
    for (int it = 0; it < 2; ++it) {
        const double e = fma(-d, y, 1.0);
        y = fma(y, e, y);
    }
    return y;
}

constexpr int CH_NT = 256;   // threads per matrix

template <typename C>
__global__ void __launch_bounds__(CH_NT)
k_chol_rinv(const double2* __restrict__ Gall, int k, int batch, double shift_rel, C* __restrict__ Rall,
            const int* __restrict__ active, int* __restrict__ need2) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int tid = threadIdx.x;
    const int mat = blockIdx.x;
    if (active && !active[mat]) return;
    const int ld = k + 1;
    // A: lower triangle = the matrix being factored (then Lt D), upper
    // triangle = U(j, l) = conj(Lt(l, j)), written as each column finishes
    double2* A = reinterpret_cast<double2*>(sm_raw);
    double2* X = A + (size_t)k * ld;                            // Xt = Lt^-1, lower
    double* dinv = reinterpret_cast<double*>(X + (size_t)k * ld);  // 1 / D(j)
    short2* tri = reinterpret_cast<short2*>(dinv + k);          // p -> (a, b), a <= b
    __shared__ double red[CH_NT / 32];
    __shared__ int fail;
    const double2* G = Gall + (long long)mat * k * k;
    C* Rout = Rall + (long long)mat * k * k;
    const int ntri = k * (k - 1) / 2;
    for (int p = tid; p < ntri; p += CH_NT) {
        int bb = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
        while ((bb + 1) * (bb + 2) / 2 <= p) ++bb;
        while (bb * (bb + 1) / 2 > p) --bb;
        tri[p] = make_short2((short)(p - bb * (bb + 1) / 2), (short)bb);
    }
    double tr = 0.0;
    for (int i = tid; i < k; i += CH_NT) tr += G[i * k + i].x;
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if ((tid & 31) == 0) red[tid >> 5] = tr;
    __syncthreads();
    tr = 0.0;
    for (int w = 0; w < CH_NT / 32; ++w) tr += red[w];
    tr /= k;
    if (!(tr > 0.0) || !isfinite(tr)) {
        const double fill = (tr == 0.0) ? 0.0 : NAN;
        for (int e = tid; e < k * k; e += CH_NT) { Rout[e].x = fill; Rout[e].y = fill; }
        if (need2 && tid == 0) need2[mat] = 0;
        return;
    }
    double shift = shift_rel * tr;
    const bool shifted0 = shift > 0.0;
    int attempts = 0;
    bool ok = false;
    for (int attempt = 0; attempt < 13 && !ok; ++attempt) {
        for (int e = tid; e < k * k; e += CH_NT) {
            const int j = e / k, i = e - j * k;
            if (i < j) continue;
            double2 v = G[e];
            if (i == j) { v.x += shift; v.y = 0.0; }
            A[j * ld + i] = v;
        }
        for (int e = tid; e < k * ld; e += CH_NT) {
            const int c = e / ld, i = e - c * ld;
            X[e] = make_double2(i == c ? 1.0 : 0.0, 0.0);
        }
        if (tid == 0) {
            const double d0 = G[0].x + shift;
            fail = (d0 > 0.0 && isfinite(d0)) ? 0 : 1;
            dinv[0] = rcp64(d0);
        }
        __syncthreads();
        for (int j = 0; j < k - 1 && !fail; ++j) {
            // column j of Lt, kept conjugated in row j: U(j, i) = conj(A(i, j)) / D(j)
            const double dj = dinv[j];
            for (int i = j + 1 + tid; i < k; i += CH_NT) {
                const double2 v = A[j * ld + i];
                A[i * ld + j] = make_double2(v.x * dj, -v.y * dj);
            }
            __syncthreads();
            // trailing triangle: A(i, l) -= A(i, j) U(j, l), j < l <= i; item
            // 0 (the next pivot) first, on thread 0, which then forms 1 / D(j+1).
            // In the same phase Xt = Lt^-1 in axpy form: Xt starts as I, row j
            // is final in every column c <= j by now, and step j removes it
            // from the rows below: Xt(i, c) -= Lt(i, j) Xt(j, c), Lt(i, j) =
            // conj(U(j, i)).  Together a step has about k^2 / 2 items whatever j.
            const int nt = k - 1 - j, T = nt * (nt + 1) / 2, items = T + nt * (j + 1);
            const float rnt = 1.0f / (float)nt;
            for (int p = tid; p < items; p += CH_NT) {
                if (p < T) {
                    const short2 ab = tri[T - 1 - p];
                    const int i = j + nt - ab.x, l = j + nt - ab.y;
                    const double2 a = A[j * ld + i], u = A[l * ld + j];
                    double2 v = A[l * ld + i];
                    v.x = fma(-a.x, u.x, v.x);
                    v.x = fma(a.y, u.y, v.x);
                    v.y = fma(-a.x, u.y, v.y);
                    v.y = fma(-a.y, u.x, v.y);
                    A[l * ld + i] = v;
                    if (p == 0) {
                        const double d = v.x;
                        if (!(d > 0.0) || !isfinite(d)) fail = 1;
                        dinv[j + 1] = rcp64(d);
                    }
                } else {
                    // e = c * nt + (i - j - 1); the float quotient is exact here
                    // (e < 4096, nt < 64: the fraction is at least 1 / (2 nt) from an integer)
                    const int e = p - T;
                    const int c = (int)(((float)e + 0.5f) * rnt), i = j + 1 + (e - c * nt);
                    const double2 u = A[i * ld + j], xt = X[c * ld + j];
                    double2 v = X[c * ld + i];
                    // v -= conj(u) xt
                    v.x = fma(-u.x, xt.x, v.x);
                    v.x = fma(-u.y, xt.y, v.x);
                    v.y = fma(-u.x, xt.y, v.y);
                    v.y = fma(u.y, xt.x, v.y);
                    X[c * ld + i] = v;
                }
            }
            __syncthreads();
        }
        ok = fail == 0;
        __syncthreads();
        if (!ok) shift = shift > 0.0 ? shift * 100.0 : 1e-15 * tr;
        ++attempts;
    }
    if (!ok) {
        for (int e = tid; e < k * k; e += CH_NT) { Rout[e].x = NAN; Rout[e].y = NAN; }
        if (need2 && tid == 0) need2[mat] = 0;
        return;
    }
    // D^-1/2 for every column at once (reuses dinv)
    for (int j = tid; j < k; j += CH_NT) dinv[j] = rsqrt64(A[j * ld + j].x);
    __syncthreads();
    // Rinv(i, j) = conj(Xt(j, i)) D(j)^-1/2, upper triangular
    double fro = 0.0;
    for (int e = tid; e < k * k; e += CH_NT) {
        const int j = e / k, i = e - j * k;
        C v;
        if (i <= j) {
            const double2 xv = X[i * ld + j];
            const double s = dinv[j];
            v.x = xv.x * s;
            v.y = -xv.y * s;
            fro += (double)v.x * v.x + (double)v.y * v.y;
        } else {
            v.x = 0;
            v.y = 0;
        }
        Rout[e] = v;
    }
    if (need2) {
        // kappa_F = ||Y||_F ||R^-1||_F >= kappa_2(Y).  One pass of Cholesky QR
        // with an FP64-accurate Gram and product leaves Q^H Q - I ~ 1e-16
        // kappa^2: a second pass is needed above kappa ~ 1e3 (and after any
        // shift, which perturbs the factor on purpose).
        for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = fro;
        __syncthreads();
        if (tid == 0) {
            double rf = 0.0;
            for (int w = 0; w < CH_NT / 32; ++w) rf += red[w];
            const double kap2 = tr * k * rf;
            need2[mat] = (shifted0 || attempts > 0 || !(kap2 <= 1e6)) ? 1 : 0;
        }
    }
}

// Q = Y R^-1 in place, formed with FP64 accuracy in FP32 arithmetic: R^-1
// (FP64, upper triangular) is split into two FP32 parts, the products with
// the high part are summed by Dot2 and those with the low part are added to
// the compensation; the result is rounded to FP32 once.  Rows are
// independent, so each CTA loads a tile of rows into shared memory and
// writes its result over it.  Blocks whose active flag is 0 are skipped.
__global__ void __launch_bounds__(256)
k_rmul_dot2(float2* __restrict__ Y, int m, int k, long long sY, const double2* __restrict__ Rall,
            const int* __restrict__ active) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    float2* Rh = reinterpret_cast<float2*>(sm_raw);   // k x k
    float2* Rl = Rh + k * k;
    float2* yt = Rl + k * k;                           // k columns x (GT_ROWS + 1)
    const double2* R = Rall + (long long)b * k * k;
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
        const double2 v = R[e];
        const float hx = (float)v.x, hy = (float)v.y;
        Rh[e] = make_float2(hx, hy);
        Rl[e] = make_float2((float)(v.x - (double)hx), (float)(v.y - (double)hy));
    }
    float2* Yb = Y + (long long)b * sY;
    const int rows_per = (m + gridDim.x - 1) / gridDim.x;
    const int r0 = blockIdx.x * rows_per, r1 = min(m, r0 + rows_per);
    for (int rr = r0; rr < r1; rr += GT_ROWS) {
        const int nr = min(GT_ROWS, r1 - rr);
        __syncthreads();
        for (int e = threadIdx.x; e < GT_ROWS * k; e += blockDim.x) {
            const int c = e / GT_ROWS, r = e - c * GT_ROWS;
            yt[c * (GT_ROWS + 1) + r] = r < nr ? Yb[(long long)c * m + rr + r] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < GT_ROWS * k; e += blockDim.x) {
            const int j = e / GT_ROWS, r = e - j * GT_ROWS;
            if (r >= nr) continue;
            float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
            for (int t = 0; t <= j; ++t) {
                const float2 a = yt[t * (GT_ROWS + 1) + r], h = Rh[j * k + t], l = Rl[j * k + t];
                dot2(a.x, h.x, sr, cr);
                dot2(-a.y, h.y, sr, cr);
                dot2(a.x, h.y, si, ci);
                dot2(a.y, h.x, si, ci);
                cr = fmaf(a.x, l.x, fmaf(-a.y, l.y, cr));
                ci = fmaf(a.x, l.y, fmaf(a.y, l.x, ci));
            }
            Yb[(long long)j * m + rr + r] = make_float2(__fadd_rn(sr, cr), __fadd_rn(si, ci));
        }
    }
}

// --------------------------- eigenvectors of a Gram matrix (FP64 accuracy)
// The eigenvectors of G = Y^H Y (FP64-accurate, eigenvalues spread over up to
// 16 decades) are the left singular vectors of its Cholesky factor L, and
// one-sided Jacobi on L's columns finds those in FP32 however small their
// singular values are against the largest: the factor carries the square roots
// of the eigenvalues column by column, and a pair of columns is rotated by
// their own inner product alone (Veselic and Hari, Numer. Math. 56, 1989).
// One CTA per matrix.
//   1. The trace is scaled to 1 and the indices sorted by the diagonal's
//      thousands (2^10): a sketch's own order is nearly decreasing and saves
//      sweeps, and a block's empty columns come last.
//   2. G = Lt D Lt^H in FP64 (square-root-free, as in k_chol_rinv), without
//      further pivoting.  A pivot not above 1e-15, the accuracy of G itself,
//      becomes 1e-15 with nothing below it: no restart.  What is dropped below it
//      can be as large as 3e-8 (columns nearly equal to earlier ones ahead of
//      independent ones), but it couples directions of no weight: for the matrix
//      G' that is factored, v^H G v <= (p + 1) v^H G' v after p such pivots
//      (||v||_S <= ||v_j||_d + ||rest||_R for a positive S with diagonal
//      blocks d and R), so directions that the truncation leaves out for their
//      small eigenvalues in G' carry no more than p + 1 times as much of G.
//   3. W = L, times 2^20 so that all squares are normal FP32 numbers.  Rounds of
//      disjoint column pairs (circle method), sixteen lanes per pair: the
//      pair's norms and inner product (four shuffles), the rotation, the update, one
//      barrier per round.  A pair is left alone below 3e-7 of its
//      norms (twice the rounding of a 64-term inner product); a sweep without a
//      rotation ends.
//   4. Columns divided by their norms, by decreasing norm, rows put back.
// Bound by latency: for 30 x 30 about 25 us of FP64 chains in 2 and 8.5 us per
// sweep in 3 (0.3 us a round), 5 to 6 sweeps, 78 us in all (one GB300).  A
// coarse FP32 two-sided Jacobi, a Rayleigh-Ritz projection in split FP32 and a
// second Jacobi that resolved the small eigenvalues took 67 + 16 + 122 us and a
// product, and left complex64 sketches 1e-6 to 1e-5 from their FP64
// counterparts where this leaves 3e-7 to 2e-6.
__device__ __forceinline__ float rsqrt_newton(float a) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return fmaf(0.5f * y, fmaf(-a * y, y, 1.f), y);
}

template <int RPL>
__global__ void __launch_bounds__(RPL * 128)
k_eig_gram(const double2* __restrict__ Gall, float2* __restrict__ Vall, int k) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    constexpr int LW = 16 * RPL + 1;                                // rows of W, zero beyond k, and a pad
    const int ld = k + 1;
    double2* A = reinterpret_cast<double2*>(sm_raw);                // k x ld, then
    double* dinv = reinterpret_cast<double*>(A + (size_t)k * ld);   // 1 / D(j), 0 for a floored pivot
    double* dval = dinv + k;                                        // D(j)
    const int m = (k + 1) & ~1;
    float2* W = reinterpret_cast<float2*>(dval + k);                // m columns of LW
    short2* tri = reinterpret_cast<short2*>(W + (size_t)m * LW);    // p -> (a, b), a <= b
    __shared__ double trs;
    __shared__ int order[64];
    __shared__ float key[64];
    __shared__ int rotated;
    const double2* G = Gall + (long long)blockIdx.x * k * k;
    const int ntri = k * (k - 1) / 2;
    for (int p = tid; p < ntri; p += nt) {
        int a, b;
        tri_pair(p, a, b);
        tri[p] = make_short2((short)a, (short)b);
    }
    if (warp == 0) {
        double t = 0;
        for (int i = lane; i < k; i += 32) t += fabs(G[i * k + i].x);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) trs = t > 0 ? 1.0 / t : 0.0;
    }
    // position of each index by decreasing key (ties by index, NaN last)
    auto sort_keys = [&]() {
        for (int i = tid; i < k; i += nt) {
            const float a = isnan(key[i]) ? -INFINITY : key[i];
            int pos = 0;
            for (int j = 0; j < k; ++j) {
                const float b = isnan(key[j]) ? -INFINITY : key[j];
                pos += (b > a || (b == a && j < i)) ? 1 : 0;
            }
            order[pos] = i;
        }
    };
    __syncthreads();
    for (int i = tid; i < k; i += nt) {
        const float d = (float)(G[i * k + i].x * trs);
        key[i] = d > 0.f ? (float)(ilogbf(d) / 10) : d == 0.f ? -100.f : d;
    }
    __syncthreads();
    sort_keys();
    __syncthreads();
    const int row0 = lane < k ? order[lane] : 0, row1 = lane + 32 < k ? order[lane + 32] : 0;
    for (int e = tid; e < k * k; e += nt) {
        const int j = e / k, i = e - j * k;
        if (i < j) continue;
        const double2 v = G[order[j] * k + order[i]];
        A[j * ld + i] = make_double2(v.x * trs, i == j ? 0.0 : v.y * trs);
    }
    __syncthreads();
    constexpr double tiny = 1e-15;
    if (tid == 0) {
        const double d = A[0].x;
        dval[0] = d > tiny ? d : tiny;
        dinv[0] = d > tiny ? rcp64(d) : 0.0;
    }
    __syncthreads();
    for (int j = 0; j < k - 1; ++j) {
        // column j of Lt, kept conjugated in row j: U(j, i) = conj(A(i, j)) / D(j)
        const double dj = dinv[j];
        for (int i = j + 1 + tid; i < k; i += nt) {
            const double2 v = A[j * ld + i];
            A[i * ld + j] = make_double2(v.x * dj, -v.y * dj);
        }
        __syncthreads();
        // trailing triangle: A(i, l) -= A(i, j) U(j, l); item 0, the next pivot, first
        const int n = k - 1 - j, T = n * (n + 1) / 2;
        for (int p = tid; p < T; p += nt) {
            const short2 ab = tri[T - 1 - p];
            const int i = j + n - ab.x, l = j + n - ab.y;
            const double2 a = A[j * ld + i], u = A[l * ld + j];
            double2 v = A[l * ld + i];
            v.x = fma(-a.x, u.x, v.x);
            v.x = fma(a.y, u.y, v.x);
            v.y = fma(-a.x, u.y, v.y);
            v.y = fma(-a.y, u.x, v.y);
            A[l * ld + i] = v;
            if (p == 0) {
                dval[j + 1] = v.x > tiny ? v.x : tiny;
                dinv[j + 1] = v.x > tiny ? rcp64(v.x) : 0.0;
            }
        }
        __syncthreads();
    }
    // W(i, j) = Lt(i, j) sqrt(D(j)) 2^20, zero above the diagonal and beyond k
    for (int e = tid; e < m * LW; e += nt) {
        const int j = e / LW, i = e - j * LW;
        float2 w = make_float2(0.f, 0.f);
        if (i >= j && i < k) {
            const float s = sqrtf((float)dval[j]) * 1048576.f;
            if (i == j) w.x = s;
            else w = make_float2((float)A[i * ld + j].x * s, -(float)A[i * ld + j].y * s);
        }
        W[e] = w;
    }
    if (tid == 0) rotated = 0;
    __syncthreads();
    // pair i of round r: columns (m - 1, r) or (r + i, r - i) mod m - 1; an
    // odd k's extra column is zero and never rotates
    const int i = tid >> 4, l16 = tid & 15;
    const bool live = i < m / 2;
    const int lim = (m - 1) * LW;
    for (int sweep = 0; sweep < 20; ++sweep) {
        int po = (i == 0 ? m - 1 : i) * LW, qo = (live && i > 0 ? m - 1 - i : 0) * LW;
        if (!live) po = 0;
        for (int r = 0; r < m - 1; ++r) {
            float2 *wp = W + po + l16, *wq = W + qo + l16;
            float2 a[RPL], b[RPL];
#pragma unroll
            for (int u = 0; u < RPL; ++u) {
                a[u] = wp[16 * u];
                b[u] = wq[16 * u];
            }
            if (i) { po += LW; if (po == lim) po = 0; }
            qo += LW;
            if (qo == lim) qo = 0;
            // norms and w_p^H w_q
            float al = 0.f, be = 0.f;
            float2 ga = make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < RPL; ++u) {
                al = fmaf(a[u].x, a[u].x, fmaf(a[u].y, a[u].y, al));
                be = fmaf(b[u].x, b[u].x, fmaf(b[u].y, b[u].y, be));
                cfmac(ga, a[u], b[u]);
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                al += __shfl_xor_sync(0xffffffffu, al, o);
                be += __shfl_xor_sync(0xffffffffu, be, o);
                ga.x += __shfl_xor_sync(0xffffffffu, ga.x, o);
                ga.y += __shfl_xor_sync(0xffffffffu, ga.y, o);
            }
            const float g2 = fmaf(ga.x, ga.x, ga.y * ga.y);
            if (live && g2 > 9e-14f * (al * be)) {
                // the rotation that makes w_p, w_q orthogonal, by the half angle:
                // h = sqrt(d^2 + 4 |g|^2), cos^2 = (1 + |d| / h) / 2, sin cos = |g| / h
                const float d = be - al, rg = rsqrt_newton(g2);
                const float rh = rsqrt_newton(fmaf(4.f, g2, d * d));
                const float x = fmaf(0.5f * fabsf(d), rh, 0.5f), rx = rsqrt_newton(x);
                const float cs = x * rx, sn = (d >= 0 ? g2 : -g2) * rg * rh * rx;
                const float2 em = make_float2(ga.x * rg, -ga.y * rg);       // e^{-i phi}, g = |g| e^{i phi}
#pragma unroll
                for (int u = 0; u < RPL; ++u) {
                    const float2 e = cmul(em, b[u]);
                    wp[16 * u] = make_float2(cs * a[u].x - sn * e.x, cs * a[u].y - sn * e.y);
                    wq[16 * u] = make_float2(sn * a[u].x + cs * e.x, sn * a[u].y + cs * e.y);
                }
                if (l16 == 0) rotated = sweep + 1;
            }
            __syncthreads();
        }
        if (rotated != sweep + 1) break;        // every thread reads it between the same two barriers
        __syncthreads();
    }
    // norms (squared) as sort keys, columns normalised, rows back in place
    float2* Vo = Vall + (long long)blockIdx.x * k * k;
    for (int j = warp; j < k; j += nt >> 5) {
        const float2 a0 = lane < k ? W[j * LW + lane] : make_float2(0.f, 0.f);
        const float2 a1 = lane + 32 < k ? W[j * LW + lane + 32] : make_float2(0.f, 0.f);
        float s = fmaf(a0.x, a0.x, a0.y * a0.y) + fmaf(a1.x, a1.x, a1.y * a1.y);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float f = rsqrt_newton(s);
        if (lane < k) W[j * LW + lane] = make_float2(a0.x * f, a0.y * f);
        if (lane + 32 < k) W[j * LW + lane + 32] = make_float2(a1.x * f, a1.y * f);
        if (lane == 0) key[j] = s;
    }
    __syncthreads();
    sort_keys();
    __syncthreads();
    for (int j = warp; j < k; j += nt >> 5) {
        const float2* w = W + order[j] * LW;
        if (lane < k) Vo[j * k + row0] = w[lane];
        if (lane + 32 < k) Vo[j * k + row1] = w[lane + 32];
    }
}

__global__ void k_up64(const float2* __restrict__ s, long long sS, double2* __restrict__ d, long long n, int batch) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * batch; e += (long long)gridDim.x * blockDim.x) {
        const long long b = e / n, i = e - b * n;
        const float2 v = s[b * sS + i];
        d[e] = make_double2(v.x, v.y);
    }
}

__global__ void k_down32(const double2* __restrict__ s, float2* __restrict__ d, long long sD, long long n, int batch) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * batch; e += (long long)gridDim.x * blockDim.x) {
        const long long b = e / n, i = e - b * n;
        const double2 v = s[e];
        d[b * sD + i] = make_float2((float)v.x, (float)v.y);
    }
}

}  // namespace

lsw_status gram64_c64(const float2* Y, int m, int k, long long sY, int batch, double2* G, cudaStream_t st,
                      const int* active) {
    if (batch <= 0 || k <= 0) return LSW_OK;
    if (k > 64) return LSW_ERR_INVALID_ARG;
    const int nchunk = sketch_chunks(m, batch);
    const int npair = k * (k + 1) / 2;
    DevBuf part;
    LSW_TRY(part.alloc(sizeof(double2) * (size_t)batch * nchunk * npair, st));
    KTimer kt("gram", st, 8.0 * batch * (double)m * k, 0.0);
    k_gram_c64<<<dim3(nchunk, batch), 256, sizeof(float2) * (GT_ROWS + 1) * k, st>>>(Y, m, k, sY, nchunk,
                                                                                        part.as<double2>(), active);
    LSW_LAUNCH_CHECK();
    // many chunks go with few blocks (sketch_chunks): enough CTAs either way
    if (nchunk >= 32)
        k_gram_c64_reduce_few<<<dim3((npair + 31) / 32, batch), dim3(32, 32), 0, st>>>(part.as<double2>(), nchunk, k, G);
    else
        k_gram_c64_reduce<<<grid_small((long long)batch * k * k), 256, 0, st>>>(part.as<double2>(), nchunk, k, batch, G);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

template <typename R>
lsw_status chol_rinv(const double2* G, int k, int batch, double shift_rel, typename Cx<R>::T* Rinv, cudaStream_t st,
                     const int* active, int* need2) {
    typedef typename Cx<R>::T C;
    if (batch <= 0 || k <= 0) return LSW_OK;
    if (k > 64) return LSW_ERR_INVALID_ARG;
    const size_t per = sizeof(double2) * 2 * (size_t)k * (k + 1) + sizeof(double) * k +
                       sizeof(short2) * (size_t)(k * (k - 1) / 2 + 1);
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        LSW_CUDA(cudaFuncSetAttribute(k_chol_rinv<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr.store(true);
    }
    KTimer kt("chol", st, 0.0, 0.0);
    k_chol_rinv<C><<<batch, CH_NT, per, st>>>(G, k, batch, shift_rel, Rinv, active, need2);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

lsw_status heev_c64(const double2* G, float2* V, int k, int batch, cudaStream_t st) {
    if (batch <= 0 || k <= 0) return LSW_OK;
    if (k > 64) return LSW_ERR_INVALID_ARG;
    // algorithmic work: the classical count of a Hermitian eigen-decomposition
    // with eigenvectors, 9 k^3 real flops for real symmetric, four times that
    // for complex (reads and writes of the k x k matrices only, in bytes)
    KTimer kt("heev", st, 24.0 * (double)k * k * batch, 36.0 * (double)k * k * k * batch);
    const int rpl = k <= 32 ? 2 : 4;
    const size_t smem = sizeof(double2) * (size_t)k * (k + 1) + 2 * sizeof(double) * k +
                        sizeof(float2) * (size_t)((k + 1) & ~1) * (16 * rpl + 1) +
                        sizeof(short2) * (size_t)(k * (k - 1) / 2 + 1);
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        LSW_CUDA(cudaFuncSetAttribute(k_eig_gram<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 120 * 1024));
        LSW_CUDA(cudaFuncSetAttribute(k_eig_gram<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 120 * 1024));
        attr.store(true);
    }
    if (rpl == 2) k_eig_gram<2><<<batch, 256, smem, st>>>(G, V, k);
    else k_eig_gram<4><<<batch, 512, smem, st>>>(G, V, k);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

// Thin QR of complex64 sketch blocks, Q returned in place of A (m x k, ld m,
// block stride sA).  Tall blocks (m >= 4k): Cholesky QR with FP64-accurate
// arithmetic in every step (Yamamoto, Nakatsukasa, Yanagisawa, Fukaya 2015,
// with the Gram and the product both accurate to ~1e-16): G = Y^H Y by
// Dot2, G + s I = R^H R in FP64 (s = 0, raised only on breakdown), Q = Y R^-1
// by Dot2 products in place.  Then Q^H Q - I ~ 1e-16 kappa(Y)^2 + u32, so a
// second identical pass on Q runs only for the blocks whose estimate
// kappa_F = ||Y||_F ||R^-1||_F exceeds 1e3 or whose factor needed a shift
// (a per-block flag on the device; the other blocks skip it).  Short blocks:
// Householder QR in FP64 on an upcast copy.
lsw_status qr_sketch_c64(float2* A, int m, int k, long long sA, int batch, cudaStream_t st) {
    if (batch <= 0 || k <= 0 || m <= 0) return LSW_OK;
    if (k > 64) return LSW_ERR_INVALID_ARG;
    const long long mk = (long long)m * k;
    if (m < 4 * k) {
        DevBuf w;
        LSW_TRY(w.alloc(sizeof(double2) * (size_t)mk * batch, st));
        k_up64<<<grid_small(mk * batch), 256, 0, st>>>(A, sA, w.as<double2>(), mk, batch);
        LSW_LAUNCH_CHECK();
        LSW_TRY(qr_explicit<double>(w.as<double2>(), m, k, mk, batch, nullptr, st));
        k_down32<<<grid_small(mk * batch), 256, 0, st>>>(w.as<double2>(), A, sA, mk, batch);
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    }
    KTimer kt("qr", st, 8.0 * batch * (double)mk * 4, 2.0 * batch * (8.0 * m * k * (k + 1) / 2 * 5 * 2));
    DevBuf G, Ri, flag;
    LSW_TRY(G.alloc(sizeof(double2) * (size_t)batch * k * k, st));
    LSW_TRY(Ri.alloc(sizeof(double2) * (size_t)batch * k * k, st));
    LSW_TRY(flag.alloc(sizeof(int) * (size_t)batch, st));
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        LSW_CUDA(cudaFuncSetAttribute(k_rmul_dot2, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
        attr.store(true);
    }
    const size_t smp = sizeof(float2) * (2 * (size_t)k * k + (size_t)(GT_ROWS + 1) * k);
    const int nchunk = sketch_chunks(m, batch);
    auto pass = [&](const int* active, int* need2) -> lsw_status {
        LSW_TRY(gram64_c64(A, m, k, sA, batch, G.as<double2>(), st, active));
        LSW_TRY(chol_rinv<double>(G.as<double2>(), k, batch, 0.0, Ri.as<double2>(), st, active, need2));
        k_rmul_dot2<<<dim3(nchunk, batch), 256, smp, st>>>(A, m, k, sA, Ri.as<double2>(), active);
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    };
    LSW_TRY(pass(nullptr, flag.as<int>()));
    LSW_TRY(pass(flag.as<int>(), nullptr));
    return LSW_OK;
}

template lsw_status chol_rinv<float>(const double2*, int, int, double, float2*, cudaStream_t, const int*, int*);
template lsw_status chol_rinv<double>(const double2*, int, int, double, double2*, cudaStream_t, const int*, int*);

}  // namespace lsw
