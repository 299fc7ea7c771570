// Fourier neural operator used as a learned right preconditioner: forward,
// backward (G = dL/dRe + i dL/dIm convention), Adam, and the preconditioner
// apply, all in FP32 complex: fused passes (fno_passes.cuh) and the library's
// batched GEMMs.
//
// Network (complex): v = P x + p;  v <- sigma(K_l v + W_l v + b_l) for
// l < L (no sigma on the last layer);  y = x0 + Q v + q.  K_l keeps the 2m x 2m
// modes kz, kx in {0..m-1} U {n-m..n-1} of the 2D DFT and mixes channels per
// mode with R_l[mode] (W x W).  sigma: GELU on real and imaginary parts.
// The output adds the input's residual channel x0: y = x0 + Q v + q.
//
// Layouts.  A field is nz x nx, strip order; a batch of samples holds W
// fields per sample, sample after sample, so sample b is the column-major
// n x W matrix V_b.  Parameters live in one buffer in this order (all
// column-major complex): P^T (2 x W), p (W), then per layer R (4m^2 modes,
// each W_out x W_in), W^T (W x W), b (W), then Q^T (W x 1), q (1).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <new>
#include <vector>

#include "fno_passes.cuh"
#include "lsw_internal.cuh"

struct lsw_fno {
    int nz, nx, W, m, L;
    long long n;                 // nz * nx
    int M;                       // 2m modes per axis, M * M modes
    float2* params = nullptr;    // np entries
    float2* grads = nullptr;
    float2* adam_m = nullptr;
    float2* adam_v = nullptr;    // (second moments of re, im)
    long long np = 0;
    float2* Fz = nullptr;        // M x nz   rows of the DFT
    float2* FxT = nullptr;       // nx x M   (F_x)^T
    float2* Fxc = nullptr;       // M x nx   conj(F_x)
    bool fast = false;           // truncated transforms by register DFTs (fno_passes.cuh)
    float2* twz = nullptr;       // their line twiddles, nz and nx entries (inside Fz's and FxT's arrays)
    float2* twx = nullptr;
    // offsets into params
    long long oPT, op, oQT, oq;
    std::vector<long long> oR, oWT, ob;
};

namespace lsw {
namespace {

int gridn(long long n, int bs = 256) {
    long long g = (n + bs - 1) / bs;
    return (int)std::max<long long>(1, std::min<long long>(g, 152LL * 32));
}

__host__ __device__ inline float2 c1() { return make_float2(1.f, 0.f); }
__host__ __device__ inline float2 c0() { return make_float2(0.f, 0.f); }

// rows of the DFT for the retained wavenumbers: F[a][i] = exp(-2 pi i k_a i / n)
__global__ void k_dft_rows(float2* F, int n, int m, int ld_rows_first) {
    const int M = 2 * m;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M * n; e += gridDim.x * blockDim.x) {
        const int a = e % M, i = e / M;
        const int k = a < m ? a : n - 2 * m + a;
        double s, c;
        sincospi(-2.0 * (double)((long long)k * i % n) / n, &s, &c);
        const float2 v = make_float2((float)c, (float)s);
        // ld_rows_first: store M x n (element (a, i) at a + M i), else n x M transposed (i + n a)
        if (ld_rows_first) F[a + (long long)M * i] = v;
        else F[i + (long long)n * a] = v;
    }
}

__global__ void k_conj(const float2* a, float2* b, long long n) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        b[e] = make_float2(a[e].x, -a[e].y);
}

// v[b][w][i] += bias[w]
__global__ void k_bias(float2* v, const float2* __restrict__ bias, long long n, int W, int B) {
    const long long tot = n * W * B;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const int w = (int)((e / n) % W);
        v[e].x += bias[w].x;
        v[e].y += bias[w].y;
    }
}

// v = split-GELU(z + bias) (or z + bias)
__global__ void k_bias_act(const float2* __restrict__ z, const float2* __restrict__ bias, float2* __restrict__ v,
                           long long n, int W, int B, int act) {
    const long long tot = n * W * B;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const int w = (int)((e / n) % W);
        float2 t = z[e];
        t.x += bias[w].x;
        t.y += bias[w].y;
        v[e] = act ? make_float2(gelu_f(t.x), gelu_f(t.y)) : t;
    }
}

// [b][w][mode] <-> [mode][b][w]: per mode a W x B column-major matrix
__global__ void k_bwm_to_mwb(const float2* __restrict__ s, float2* __restrict__ d, int B, int W, int MM) {
    const long long tot = (long long)B * W * MM;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const int md = (int)(e % MM);
        const long long r = e / MM;
        const int w = (int)(r % W), b = (int)(r / W);
        d[((long long)md * B + b) * W + w] = s[e];
    }
}
__global__ void k_mwb_to_bwm(const float2* __restrict__ s, float2* __restrict__ d, int B, int W, int MM) {
    const long long tot = (long long)B * W * MM;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const int md = (int)(e % MM);
        const long long r = e / MM;
        const int w = (int)(r % W), b = (int)(r / W);
        d[e] = s[((long long)md * B + b) * W + w];
    }
}

// G_y = 2 (y - t) / count; per-block partial sums of |y - t|^2
__global__ void k_loss(const float2* __restrict__ y, const float2* __restrict__ t, float2* __restrict__ g, long long tot,
                       float scale, double* part) {
    double s = 0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const float dx = y[e].x - t[e].x, dy = y[e].y - t[e].y;
        g[e] = make_float2(2.f * dx * scale, 2.f * dy * scale);
        s += (double)dx * dx + (double)dy * dy;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0;
        for (int i = 0; i < 8; ++i) a += red[i];
        part[blockIdx.x] = a;
    }
}

// out = sum over b of part[b] (count elements each)
__global__ void k_batch_sum(const float2* __restrict__ part, float2* __restrict__ out, long long count, int B) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count; e += (long long)gridDim.x * blockDim.x) {
        float2 a = c0();
        for (int b = 0; b < B; ++b) { a.x += part[b * count + e].x; a.y += part[b * count + e].y; }
        out[e] = a;
    }
}

__global__ void k_adam(float2* __restrict__ w, const float2* __restrict__ g, float2* __restrict__ m, float2* __restrict__ v,
                       long long n, float lr, float b1, float b2, float eps, float c1_, float c2_) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const float2 gg = g[e];
        float2 mm = m[e], vv = v[e];
        mm.x = b1 * mm.x + (1 - b1) * gg.x;
        mm.y = b1 * mm.y + (1 - b1) * gg.y;
        vv.x = b2 * vv.x + (1 - b2) * gg.x * gg.x;
        vv.y = b2 * vv.y + (1 - b2) * gg.y * gg.y;
        m[e] = mm;
        v[e] = vv;
        float2 ww = w[e];
        ww.x -= lr * (mm.x / c1_) / (sqrtf(vv.x / c2_) + eps);
        ww.y -= lr * (mm.y / c1_) / (sqrtf(vv.y / c2_) + eps);
        w[e] = ww;
    }
}

// Input channels of the preconditioner apply: x0 = v / s_b, x1 = chi / k0^2 + i k0 h
template <typename C>
__global__ void k_fno_input(const C* __restrict__ v, const double* __restrict__ inv_norm, const double* __restrict__ chi,
                            double ik02, float k0h, float2* __restrict__ x, long long n, int B) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * B; e += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(e / n);
        const long long i = e - (long long)b * n;
        const double s = inv_norm[b];
        x[((long long)b * 2) * n + i] = make_float2((float)(v[e].x * s), (float)(v[e].y * s));
        x[((long long)b * 2 + 1) * n + i] = make_float2((float)(chi[i] * ik02), k0h);
    }
}

template <typename C>
__global__ void k_fno_output(const float2* __restrict__ y, const double* __restrict__ norm, C* __restrict__ z, long long n,
                             int B) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * B; e += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(e / n);
        C o;
        o.x = y[e].x * norm[b];
        o.y = y[e].y * norm[b];
        z[e] = o;
    }
}

// t_b = e_b / ||r_b|| (complex128 or complex64 in, complex64 out)
template <typename C>
__global__ void k_scale_rows(const C* __restrict__ e, const double* __restrict__ inv_norm, float2* __restrict__ t,
                             long long n, int B) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * B; q += (long long)gridDim.x * blockDim.x) {
        const double s = inv_norm[q / n];
        t[q] = make_float2((float)(e[q].x * s), (float)(e[q].y * s));
    }
}

// x_b channel 0 and t_b times exp(i phi_b)
__global__ void k_rotate_pairs(float2* __restrict__ x, float2* __restrict__ t, const float2* __restrict__ rot,
                               long long n, int B) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * B; q += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(q / n);
        const long long i = q - (long long)b * n;
        const float2 w = rot[b];
        float2* xv = x + (long long)b * 2 * n + i;
        const float2 a = *xv, c = t[q];
        *xv = make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
        t[q] = make_float2(c.x * w.x - c.y * w.y, c.x * w.y + c.y * w.x);
    }
}

// per-block partial sums of |y - t|^2 and |t|^2 in FP64
__global__ void __launch_bounds__(256) k_err_sums(const float2* __restrict__ y, const float2* __restrict__ t,
                                                  long long tot, double* __restrict__ part) {
    __shared__ double sn[8], sd[8];
    double num = 0.0, den = 0.0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < tot; q += (long long)gridDim.x * blockDim.x) {
        const float2 a = y[q], c = t[q];
        const double dx = (double)a.x - c.x, dy = (double)a.y - c.y;
        num += dx * dx + dy * dy;
        den += (double)c.x * c.x + (double)c.y * c.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if ((threadIdx.x & 31) == 0) { sn[threadIdx.x >> 5] = num; sd[threadIdx.x >> 5] = den; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < 8; ++w) { a += sn[w]; b += sd[w]; }
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = b;
    }
}

__global__ void k_scale(float2* p, long long n, float a) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        p[e].x *= a;
        p[e].y *= a;
    }
}

__global__ void k_sqrt_inv(const double* __restrict__ n2, double* __restrict__ nrm, double* __restrict__ inv, int B) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const double s = sqrt(n2[b]);
    nrm[b] = s;
    inv[b] = s > 0 ? 1.0 / s : 0.0;
}

}  // namespace

// ------------------------------------------------------------- forward
// Activations: the scratch of a forward pass and, when keep is set, what the
// backward pass reads.
struct FnoTape {
    int B = 0;
    bool keep = false;
    std::vector<DevBuf*> bufs;
    std::vector<float2*> v, z, Vt;     // v[0..L], z[0..L-2], Vt[0..L-1] ([mode][b][w])
    ~FnoTape() { for (auto* b : bufs) delete b; }
    float2* get(size_t elems, cudaStream_t st, lsw_status* s) {
        DevBuf* b = new (std::nothrow) DevBuf();
        if (!b) { *s = LSW_ERR_OOM; return nullptr; }
        bufs.push_back(b);
        const lsw_status r = b->alloc(sizeof(float2) * elems, st);
        if (r != LSW_OK) { *s = r; return nullptr; }
        return b->as<float2>();
    }
};

namespace {

bool fno_fast(int nz, int nx, int M) {
    if (M != 8 && M != 16 && M != 32) return false;
    if (nz % M || nx % M) return false;
    const int qz = nz / M, qx = nx / M;
    return is_pow2(qz) && is_pow2(qx) && qz <= M && qx <= M &&
           sizeof(float2) * M * (size_t)(nx + 1) <= 200 * 1024;
}

// scratch of the spectral passes
struct SpecWork {
    float2 *T1, *Vh, *Zt, *Zh;
};

// Vt[mode][b][w] = scale * truncated transform of the B W fields of v
lsw_status fno_analysis(const lsw_fno* f, const float2* v, int B, float scale, const SpecWork& wk, float2* Vt,
                        cudaStream_t st) {
    const int W = f->W, M = f->M, MM = M * M, nz = f->nz, nx = f->nx;
    if (f->fast) {
        const size_t smem = sizeof(float2) * M * (size_t)(nx + 1);
        static std::atomic<bool> attr{false};
        if (!attr.load()) {
            for (auto k : {k_fno_analysis<8>, k_fno_analysis<16>, k_fno_analysis<32>})
                LSW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
            attr.store(true);
        }
        auto k = M == 8 ? k_fno_analysis<8> : M == 16 ? k_fno_analysis<16> : k_fno_analysis<32>;
        k<<<B * W, 256, smem, st>>>(v, nz, nx, B * W, f->twz, f->twx, scale, Vt);
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    }
    // Vh = Fz v FxT   (per sample and channel: M x M)
    LSW_TRY(gemm<float>('N', 'N', M, nx, nz, c1(), f->Fz, M, 0, v, nz, f->n, c0(), wk.T1, M, (long long)M * nx, B * W, st));
    LSW_TRY(gemm<float>('N', 'N', M, M, nx, make_float2(scale, 0.f), wk.T1, M, (long long)M * nx, f->FxT, nx, 0, c0(),
                        wk.Vh, M, MM, B * W, st));
    k_bwm_to_mwb<<<gridn((long long)B * W * MM), 256, 0, st>>>(wk.Vh, Vt, B, W, MM);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

// out = sigma(inverse transform of Zt / scale^-1 + pointwise map of v + bias)
lsw_status fno_synthesis(const lsw_fno* f, const float2* Zt, int B, float scale, const SpecWork& wk, float2* zin,
                         PointwiseArgs a, cudaStream_t st) {
    const int W = f->W, M = f->M, MM = M * M, nz = f->nz, nx = f->nx, og = (W + 7) / 8;
    a.n = f->n;
    a.nz = nz;
    a.W = W;
    // the fused z transform needs whole columns in a tile
    const int cells = 4 * pw_cells(og);
    const bool fused = f->fast && cells % nz == 0;
    if (f->fast) {
        auto k = M == 8 ? k_fno_synth_x<8> : M == 16 ? k_fno_synth_x<16> : k_fno_synth_x<32>;
        k<<<B * W, 256, 0, st>>>(Zt, nx, B * W, f->twx, scale, wk.T1);
        LSW_LAUNCH_CHECK();
    } else {
        k_mwb_to_bwm<<<gridn((long long)B * W * MM), 256, 0, st>>>(Zt, wk.Zh, B, W, MM);
        LSW_LAUNCH_CHECK();
        LSW_TRY(gemm<float>('N', 'N', M, nx, M, make_float2(scale, 0.f), wk.Zh, M, MM, f->Fxc, M, 0, c0(), wk.T1, M,
                            (long long)M * nx, B * W, st));
    }
    if (!fused)
        LSW_TRY(gemm<float>('C', 'N', nz, nx, M, c1(), f->Fz, M, 0, wk.T1, M, (long long)M * nx, c0(), zin, nz, f->n,
                            B * W, st));
    a.T1 = wk.T1;
    a.twz = f->twz;
    a.zin = zin;
    const int nt = pw_threads(og);
    const int Mk = fused ? M : 0;
    const size_t smem = sizeof(float2) * W * (size_t)(8 * og + cells + 8);
    const dim3 grid((unsigned)((f->n + cells - 1) / cells), B);
    typedef void (*Kern)(PointwiseArgs);
    static const Kern kerns[2][4] = {{k_fno_pointwise<0, 256>, k_fno_pointwise<8, 256>, k_fno_pointwise<16, 256>,
                                      k_fno_pointwise<32, 256>},
                                     {k_fno_pointwise<0, 512>, k_fno_pointwise<8, 512>, k_fno_pointwise<16, 512>,
                                      k_fno_pointwise<32, 512>}};
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        for (auto& by_m : kerns)
            for (Kern k : by_m)
                LSW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr.store(true);
    }
    const Kern k = kerns[nt == 512][Mk == 0 ? 0 : Mk == 8 ? 1 : Mk == 16 ? 2 : 3];
    k<<<grid, nt, smem, st>>>(a);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

bool fno_zin_needed(const lsw_fno* f) { return !f->fast || (4 * pw_cells((f->W + 7) / 8)) % f->nz != 0; }

lsw_status fno_spec_work(const lsw_fno* f, int B, FnoTape& tp, SpecWork* wk, cudaStream_t st) {
    lsw_status s = LSW_OK;
    const size_t modes = (size_t)B * f->W * f->M * f->M;
    wk->T1 = tp.get((size_t)B * f->W * f->M * f->nx, st, &s);
    wk->Zt = tp.get(modes, st, &s);
    wk->Vh = wk->Zh = nullptr;
    if (!f->fast) {
        wk->Vh = tp.get(modes, st, &s);
        wk->Zh = tp.get(modes, st, &s);
    }
    return s;
}

}  // namespace

static lsw_status fno_forward(const lsw_fno* f, const float2* x, float2* y, int B, FnoTape& tp, cudaStream_t st) {
    const long long n = f->n;
    const int W = f->W, M = f->M, MM = M * M;
    const float2* P = f->params;
    lsw_status s = LSW_OK;
    tp.B = B;
    tp.v.assign(f->L + 1, nullptr);
    tp.z.assign(f->L, nullptr);
    tp.Vt.assign(f->L, nullptr);
    SpecWork wk;
    LSW_TRY(fno_spec_work(f, B, tp, &wk, st));
    const size_t act = (size_t)B * W * n, modes = (size_t)B * W * MM;
    float2* zin = fno_zin_needed(f) ? tp.get(act, st, &s) : nullptr;
    for (int l = 0; l <= f->L; ++l)     // without keep the pointwise map works in place
        tp.v[l] = l == 0 || tp.keep ? tp.get(act, st, &s) : tp.v[0];
    for (int l = 0; l < f->L; ++l) {
        if (tp.keep && l < f->L - 1) tp.z[l] = tp.get(act, st, &s);
        tp.Vt[l] = l == 0 || tp.keep ? tp.get(modes, st, &s) : tp.Vt[0];
    }
    if (s != LSW_OK) return s;
    const dim3 cells((unsigned)((n + 255) / 256), B);
    k_fno_lift<<<cells, 256, 0, st>>>(x, P + f->oPT, P + f->op, tp.v[0], n, W);
    LSW_LAUNCH_CHECK();
    const size_t smix = sizeof(float2) * ((size_t)W * W + W * 32);
    for (int l = 0; l < f->L; ++l) {
        LSW_TRY(fno_analysis(f, tp.v[l], B, 1.f, wk, tp.Vt[l], st));
        // Zt[mode] = R[mode] Vt[mode]
        k_fno_mix<<<MM, 256, smix, st>>>(P + f->oR[l], tp.Vt[l], wk.Zt, W, B);
        LSW_LAUNCH_CHECK();
        PointwiseArgs a = {};
        a.v = tp.v[l];
        a.wt = P + f->oWT[l];
        a.bias = P + f->ob[l];
        a.z = tp.z[l];
        a.out = tp.v[l + 1];
        a.act = l < f->L - 1;
        LSW_TRY(fno_synthesis(f, wk.Zt, B, 1.f / (float)n, wk, zin, a, st));
    }
    k_fno_project<<<cells, 256, 0, st>>>(x, tp.v[f->L], P + f->oQT, P + f->oq, y, n, W);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

// The forward pass for complex128 vectors (fno_apply_precond): the same network
// as a chain of dense products.  The arithmetic is FP32 either way, but its
// results leave as complex128, and callers compare and store them to the digits
// of that type, where the rounding of every sum shows.  So for this type the
// products, the order of their sums and with them every bit stay as they are;
// the fused passes round differently (1e-6 of the result).
static lsw_status fno_forward_dense(const lsw_fno* f, const float2* x, float2* y, int B, FnoTape& tp, cudaStream_t st) {
    const long long n = f->n;
    const int W = f->W, M = f->M, MM = M * M, nz = f->nz, nx = f->nx;
    const float2* P = f->params;
    lsw_status s = LSW_OK;
    const size_t act = (size_t)B * W * n, modes = (size_t)B * W * MM;
    float2* v = tp.get(act, st, &s);
    float2* z = tp.get(act, st, &s);
    float2* T1 = tp.get((size_t)B * W * M * nx, st, &s);
    float2* Vh = tp.get(modes, st, &s);         // [b][w][mode]
    float2* Vt = tp.get(modes, st, &s);         // [mode][b][w]
    float2* Zt = tp.get(modes, st, &s);
    if (s != LSW_OK) return s;
    // lift: V_b (n x W) = X_b (n x 2) P^T (2 x W) + p
    LSW_TRY(gemm<float>('N', 'N', (int)n, W, 2, c1(), x, (int)n, 2 * n, P + f->oPT, 2, 0, c0(), v, (int)n, W * n, B, st, true));
    k_bias<<<gridn(n * W * B), 256, 0, st>>>(v, P + f->op, n, W, B);
    LSW_LAUNCH_CHECK();
    for (int l = 0; l < f->L; ++l) {
        // Vh = Fz v FxT   (per sample and channel: M x M)
        LSW_TRY(gemm<float>('N', 'N', M, nx, nz, c1(), f->Fz, M, 0, v, nz, n, c0(), T1, M, (long long)M * nx, B * W, st, true));
        LSW_TRY(gemm<float>('N', 'N', M, M, nx, c1(), T1, M, (long long)M * nx, f->FxT, nx, 0, c0(), Vh, M, MM, B * W, st,
                            true));
        k_bwm_to_mwb<<<gridn((long long)B * W * MM), 256, 0, st>>>(Vh, Vt, B, W, MM);
        LSW_LAUNCH_CHECK();
        // Zt[mode] = R[mode] Vt[mode]
        LSW_TRY(gemm<float>('N', 'N', W, B, W, c1(), P + f->oR[l], W, (long long)W * W, Vt, W, (long long)W * B, c0(), Zt,
                            W, (long long)W * B, MM, st, true));
        k_mwb_to_bwm<<<gridn((long long)B * W * MM), 256, 0, st>>>(Zt, Vh, B, W, MM);
        LSW_LAUNCH_CHECK();
        // z = Fz^H (Zh conj(Fx)) / n
        LSW_TRY(gemm<float>('N', 'N', M, nx, M, c1(), Vh, M, MM, f->Fxc, M, 0, c0(), T1, M, (long long)M * nx, B * W, st,
                            true));
        LSW_TRY(gemm<float>('C', 'N', nz, nx, M, make_float2(1.f / (float)n, 0.f), f->Fz, M, 0, T1, M, (long long)M * nx,
                            c0(), z, nz, n, B * W, st, true));
        // z += V W^T;  v = sigma(z + b)
        LSW_TRY(gemm<float>('N', 'N', (int)n, W, W, c1(), v, (int)n, W * n, P + f->oWT[l], W, 0, c1(), z, (int)n, W * n, B,
                            st, true));
        k_bias_act<<<gridn(n * W * B), 256, 0, st>>>(z, P + f->ob[l], v, n, W, B, l < f->L - 1);
        LSW_LAUNCH_CHECK();
    }
    // project: y_b (n x 1) = x0_b + V_b Q^T + q  (the residual channel passes through)
    LSW_CUDA(cudaMemcpy2DAsync(y, sizeof(float2) * n, x, sizeof(float2) * 2 * n, sizeof(float2) * n, B,
                               cudaMemcpyDeviceToDevice, st));
    LSW_TRY(gemm<float>('N', 'N', (int)n, 1, W, c1(), v, (int)n, W * n, P + f->oQT, W, 0, c1(), y, (int)n, n, B, st, true));
    k_bias<<<gridn(n * B), 256, 0, st>>>(y, P + f->oq, n, 1, B);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

static lsw_status fno_backward(lsw_fno* f, const float2* x, const float2* Gy, int B, FnoTape& tp, cudaStream_t st) {
    const long long n = f->n;
    const int W = f->W, M = f->M, MM = M * M;
    const float2* P = f->params;
    float2* G = f->grads;
    lsw_status s = LSW_OK;
    FnoTape own;
    SpecWork wk;
    LSW_TRY(fno_spec_work(f, B, own, &wk, st));
    float2* Gv = own.get((size_t)B * W * n, st, &s);        // the activations' gradient, layer by layer in place
    float2* zin = fno_zin_needed(f) ? own.get((size_t)B * W * n, st, &s) : nullptr;
    float2* GZt = own.get((size_t)B * W * MM, st, &s);
    const int chunks = (int)((n + kFnoSumChunk - 1) / kFnoSumChunk);
    // per-sample partial weight gradients (W x W at most), summed over samples
    float2* part = own.get((size_t)B * std::max<long long>({(long long)W * W, 2LL * W, (long long)W * chunks}), st, &s);
    if (s != LSW_OK) return s;
    const dim3 cells((unsigned)((n + 255) / 256), B);
    // Q^T: sum_b V_b^H Gy_b;  q: sum Gy;  G = Gy conj(Q)
    LSW_TRY(gemm<float>('C', 'N', W, 1, (int)n, c1(), tp.v[f->L], (int)n, W * n, Gy, (int)n, n, c0(), part, W, W, B, st));
    k_batch_sum<<<gridn(W), 256, 0, st>>>(part, G + f->oQT, W, B);
    LSW_LAUNCH_CHECK();
    // the sums read g through the kernel's in-place argument and leave it alone (z NULL)
    auto channel_sums = [&](float2* g, const float2* z, int chan, float2* out) -> lsw_status {
        k_fno_act_sum<<<dim3(chunks, chan * B), 256, 0, st>>>(g, z, n, part);
        LSW_LAUNCH_CHECK();
        k_fno_sum_channels<<<chan, 32, 0, st>>>(part, chunks, chan, B, out);
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    };
    LSW_TRY(channel_sums(const_cast<float2*>(Gy), nullptr, 1, G + f->oq));
    k_fno_project_grad<<<cells, 256, 0, st>>>(Gy, P + f->oQT, Gv, n, W);
    LSW_LAUNCH_CHECK();
    const size_t smix = sizeof(float2) * ((size_t)W * (W + 1) + 2 * W * 32);
    static std::atomic<bool> attr{false};
    if (!attr.load()) {
        LSW_CUDA(cudaFuncSetAttribute(k_fno_mix_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
        attr.store(true);
    }
    for (int l = f->L - 1; l >= 0; --l) {
        // Gz = Gv sigma'(z) and its channel sums
        LSW_TRY(channel_sums(Gv, l < f->L - 1 ? tp.z[l] : nullptr, W, G + f->ob[l]));
        // W^T: sum_b V_b^H Gz_b
        LSW_TRY(gemm<float>('C', 'N', W, W, (int)n, c1(), tp.v[l], (int)n, W * n, Gv, (int)n, W * n, c0(), part, W,
                            (long long)W * W, B, st));
        k_batch_sum<<<gridn((long long)W * W), 256, 0, st>>>(part, G + f->oWT[l], (long long)W * W, B);
        LSW_LAUNCH_CHECK();
        // G_Zh = Fz Gz FxT / n;  G_R[mode] = GZt[mode] Vt[mode]^H, GVt[mode] = R[mode]^H GZt[mode]
        LSW_TRY(fno_analysis(f, Gv, B, 1.f / (float)n, wk, GZt, st));
        k_fno_mix_grad<<<MM, 256, smix, st>>>(P + f->oR[l], tp.Vt[l], GZt, G + f->oR[l], wk.Zt, W, B);
        LSW_LAUNCH_CHECK();
        // Gv = Fz^H GVh conj(Fx)  +  Gz (W^T)^H
        PointwiseArgs a = {};
        a.v = Gv;
        a.wt = P + f->oWT[l];
        a.adjoint = 1;
        a.out = Gv;
        LSW_TRY(fno_synthesis(f, wk.Zt, B, 1.f, wk, zin, a, st));
    }
    // lift: P^T: sum_b X_b^H Gv_b ; p: sum Gv
    LSW_TRY(channel_sums(Gv, nullptr, W, G + f->op));
    LSW_TRY(gemm<float>('C', 'N', 2, W, (int)n, c1(), x, (int)n, 2 * n, Gv, (int)n, W * n, c0(), part, 2, 2LL * W, B, st));
    k_batch_sum<<<gridn(2LL * W), 256, 0, st>>>(part, G + f->oPT, 2LL * W, B);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

bool fno_matches(const lsw_fno* f, const lsw_green* g) { return g->nz == f->nz && g->nx == f->nx; }

lsw_status fno_apply_precond(const lsw_fno* f, const lsw_green* g, const double* chi, const void* v, void* z, int nb,
                             int prec, cudaStream_t st) {
    const long long n = f->n;
    if (!fno_matches(f, g)) return LSW_ERR_INVALID_ARG;
    DevBuf x, y, n2, nrm, inv;
    LSW_TRY(x.alloc(sizeof(float2) * 2 * n * nb, st));
    LSW_TRY(y.alloc(sizeof(float2) * n * nb, st));
    LSW_TRY(n2.alloc(sizeof(double) * nb, st));
    LSW_TRY(nrm.alloc(sizeof(double) * nb, st));
    LSW_TRY(inv.alloc(sizeof(double) * nb, st));
    if (prec == LSW_C128) LSW_TRY(norms2<double>((const double2*)v, n, nb, n2.as<double>(), st));
    else LSW_TRY(norms2<float>((const float2*)v, n, nb, n2.as<double>(), st));
    k_sqrt_inv<<<(nb + 255) / 256, 256, 0, st>>>(n2.as<double>(), nrm.as<double>(), inv.as<double>(), nb);
    LSW_LAUNCH_CHECK();
    const double ik02 = 1.0 / (g->k * g->k);
    const float k0h = (float)(g->k * g->h);
    if (prec == LSW_C128)
        k_fno_input<double2><<<gridn(n * nb), 256, 0, st>>>((const double2*)v, inv.as<double>(), chi, ik02, k0h,
                                                          x.as<float2>(), n, nb);
    else
        k_fno_input<float2><<<gridn(n * nb), 256, 0, st>>>((const float2*)v, inv.as<double>(), chi, ik02, k0h,
                                                         x.as<float2>(), n, nb);
    LSW_LAUNCH_CHECK();
    FnoTape tp;
    if (prec == LSW_C128) LSW_TRY(fno_forward_dense(f, x.as<float2>(), y.as<float2>(), nb, tp, st));
    else LSW_TRY(fno_forward(f, x.as<float2>(), y.as<float2>(), nb, tp, st));
    if (prec == LSW_C128)
        k_fno_output<double2><<<gridn(n * nb), 256, 0, st>>>(y.as<float2>(), nrm.as<double>(), (double2*)z, n, nb);
    else
        k_fno_output<float2><<<gridn(n * nb), 256, 0, st>>>(y.as<float2>(), nrm.as<double>(), (float2*)z, n, nb);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

}  // namespace lsw

using namespace lsw;

extern "C" {

lsw_status lsw_fno_create(const lsw_fno_params* p, void* stream, lsw_fno** out) {
    if (!p || !out) return LSW_ERR_INVALID_ARG;
    *out = nullptr;
    if (p->nz < 2 || p->nx < 2 || p->width < 1 || p->width > 64 || p->modes < 1 || p->layers < 1 || p->layers > 16 ||
        2 * p->modes > p->nz || 2 * p->modes > p->nx)
        return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    lsw_fno* f = new (std::nothrow) lsw_fno();
    if (!f) return LSW_ERR_OOM;
    f->nz = p->nz; f->nx = p->nx; f->W = p->width; f->m = p->modes; f->L = p->layers;
    f->n = (long long)p->nz * p->nx;
    f->M = 2 * p->modes;
    const long long W = f->W, MM = (long long)f->M * f->M;
    long long o = 0;
    f->oPT = o; o += 2 * W;
    f->op = o; o += W;
    for (int l = 0; l < f->L; ++l) {
        f->oR.push_back(o); o += MM * W * W;
        f->oWT.push_back(o); o += W * W;
        f->ob.push_back(o); o += W;
    }
    f->oQT = o; o += W;
    f->oq = o; o += 1;
    f->np = o;
    lsw_status s = LSW_OK;
    auto al = [&](float2** ptr, long long cnt) {
        if (s == LSW_OK && cudaMalloc(ptr, sizeof(float2) * cnt) != cudaSuccess) s = LSW_ERR_OOM;
    };
    al(&f->params, f->np); al(&f->grads, f->np); al(&f->adam_m, f->np); al(&f->adam_v, f->np);
    f->fast = fno_fast(f->nz, f->nx, f->M);
    // the line twiddles of the register transforms lie behind Fz and FxT
    al(&f->Fz, (long long)(f->M + f->fast) * f->nz);
    al(&f->FxT, (long long)(f->M + f->fast) * f->nx);
    al(&f->Fxc, (long long)f->M * f->nx);
    if (s != LSW_OK) { lsw_fno_destroy(f); return s; }
    cudaMemsetAsync(f->grads, 0, sizeof(float2) * f->np, st);
    cudaMemsetAsync(f->adam_m, 0, sizeof(float2) * f->np, st);
    cudaMemsetAsync(f->adam_v, 0, sizeof(float2) * f->np, st);
    k_dft_rows<<<gridn((long long)f->M * f->nz), 256, 0, st>>>(f->Fz, f->nz, f->m, 1);
    k_dft_rows<<<gridn((long long)f->M * f->nx), 256, 0, st>>>(f->FxT, f->nx, f->m, 0);
    {
        // Fxc = conj(F_x) as M x nx: conjugate-transpose of FxT via a temporary
        DevBuf tmp;
        s = tmp.alloc(sizeof(float2) * f->M * f->nx, st);
        if (s == LSW_OK) {
            k_dft_rows<<<gridn((long long)f->M * f->nx), 256, 0, st>>>(tmp.as<float2>(), f->nx, f->m, 1);
            k_conj<<<gridn((long long)f->M * f->nx), 256, 0, st>>>(tmp.as<float2>(), f->Fxc, (long long)f->M * f->nx);
        }
    }
    if (f->fast) {
        f->twz = f->Fz + (long long)f->M * f->nz;
        f->twx = f->FxT + (long long)f->M * f->nx;
        k_line_twiddles<<<gridn(f->nz + f->nx), 256, 0, st>>>(f->twz, f->nz, f->twx, f->nx, f->M);
    }
    // Gaussian initial weights (Philox), scaled per tensor by 1/sqrt(fan-in); biases zero
    if (s == LSW_OK) {
        DevBuf w2, w3;
        s = w2.alloc(sizeof(uint32_t), st);
        if (s == LSW_OK) s = w3.alloc(sizeof(uint32_t), st);
        if (s == LSW_OK) {
            cudaMemsetAsync(w2.p, 0, 4, st);
            cudaMemsetAsync(w3.p, 0, 4, st);
            s = gaussian_fill<float>(f->params, (int)f->np, 1, f->np, 1, p->seed, w2.as<uint32_t>(), w3.as<uint32_t>(), st);
        }
        if (s == LSW_OK) {
            // fan-in scaling per tensor; biases start at zero
            auto scale = [&](long long off, long long cnt, float sc) {
                k_scale<<<gridn(cnt), 256, 0, st>>>(f->params + off, cnt, sc);
            };
            auto zero = [&](long long off, long long cnt) {
                cudaMemsetAsync(f->params + off, 0, sizeof(float2) * cnt, st);
            };
            scale(f->oPT, 2 * W, 1.f / std::sqrt(2.f));
            zero(f->op, W);
            for (int l = 0; l < f->L; ++l) {
                scale(f->oR[l], MM * W * W, 1.f / (float)W);
                scale(f->oWT[l], W * W, 1.f / std::sqrt((float)W));
                zero(f->ob[l], W);
            }
            scale(f->oQT, W, 1.f / std::sqrt((float)W));
            zero(f->oq, 1);
        }
    }
    if (s == LSW_OK && cudaGetLastError() != cudaSuccess) s = LSW_ERR_CUDA;
    if (s != LSW_OK) { lsw_fno_destroy(f); return s; }
    *out = f;
    return LSW_OK;
}

lsw_status lsw_fno_destroy(lsw_fno* f) {
    if (!f) return LSW_ERR_INVALID_ARG;
    for (float2* p : {f->params, f->grads, f->adam_m, f->adam_v, f->Fz, f->FxT, f->Fxc})
        if (p) device_free(p);
    delete f;
    return LSW_OK;
}

lsw_status lsw_fno_num_params(const lsw_fno* f, int64_t* count) {
    if (!f || !count) return LSW_ERR_INVALID_ARG;
    *count = f->np;
    return LSW_OK;
}

lsw_status lsw_fno_state(lsw_fno* f, int which, void* dst, const void* src, void* stream) {
    if (!f || (!dst && !src) || which < 0 || which > 3) return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    float2* buf = which == 0 ? f->params : which == 1 ? f->grads : which == 2 ? f->adam_m : f->adam_v;
    if (dst) LSW_CUDA(cudaMemcpyAsync(dst, buf, sizeof(float2) * f->np, cudaMemcpyDeviceToDevice, st));
    if (src) LSW_CUDA(cudaMemcpyAsync(buf, src, sizeof(float2) * f->np, cudaMemcpyDeviceToDevice, st));
    return LSW_OK;
}

lsw_status lsw_fno_forward(const lsw_fno* f, const void* x, void* y, int batch, void* stream) {
    if (!f || !x || !y || batch <= 0) return LSW_ERR_INVALID_ARG;
    FnoTape tp;
    return fno_forward(f, (const float2*)x, (float2*)y, batch, tp, reinterpret_cast<cudaStream_t>(stream));
}

lsw_status lsw_fno_loss_grad(lsw_fno* f, const void* x, const void* target, int batch, double* loss, void* grad,
                             void* stream) {
    if (!f || !x || !target || batch <= 0) return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const long long tot = f->n * batch;
    DevBuf y, gy, part;
    LSW_TRY(y.alloc(sizeof(float2) * tot, st));
    LSW_TRY(gy.alloc(sizeof(float2) * tot, st));
    const int nblk = 512;
    LSW_TRY(part.alloc(sizeof(double) * nblk, st));
    FnoTape tp;
    tp.keep = true;
    LSW_TRY(fno_forward(f, (const float2*)x, y.as<float2>(), batch, tp, st));
    k_loss<<<nblk, 256, 0, st>>>(y.as<float2>(), (const float2*)target, gy.as<float2>(), tot, 1.f / (float)tot,
                                 part.as<double>());
    LSW_LAUNCH_CHECK();
    LSW_TRY(fno_backward(f, (const float2*)x, gy.as<float2>(), batch, tp, st));
    if (grad) LSW_CUDA(cudaMemcpyAsync(grad, f->grads, sizeof(float2) * f->np, cudaMemcpyDeviceToDevice, st));
    if (loss) {
        std::vector<double> h(nblk);
        LSW_CUDA(cudaMemcpyAsync(h.data(), part.p, sizeof(double) * nblk, cudaMemcpyDeviceToHost, st));
        LSW_CUDA(cudaStreamSynchronize(st));
        double s = 0;
        for (double v : h) s += v;
        *loss = s / (double)tot;
    }
    return LSW_OK;
}

lsw_status lsw_fno_adam_step(lsw_fno* f, float lr, int32_t t, void* stream) {
    if (!f || !(lr > 0) || t < 1) return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const double b1 = 0.9, b2 = 0.999;
    const float c1_ = (float)(1.0 - std::pow(b1, (double)t)), c2_ = (float)(1.0 - std::pow(b2, (double)t));
    k_adam<<<gridn(f->np), 256, 0, st>>>(f->params, f->grads, f->adam_m, f->adam_v, f->np, lr, (float)b1, (float)b2,
                                         1e-8f, c1_, c2_);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

lsw_status lsw_fno_pairs(const lsw_green* g, const double* chi, const void* r, const void* e, int nbatch, int prec,
                         void* x, void* t, void* stream) {
    if (!g || !chi || !r || !e || !x || !t || nbatch <= 0 || (prec != LSW_C128 && prec != LSW_C64))
        return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const long long n = (long long)g->nz * g->nx;
    DevBuf n2, nrm, inv;
    LSW_TRY(n2.alloc(sizeof(double) * nbatch, st));
    LSW_TRY(nrm.alloc(sizeof(double) * nbatch, st));
    LSW_TRY(inv.alloc(sizeof(double) * nbatch, st));
    if (prec == LSW_C128) LSW_TRY(norms2<double>((const double2*)r, n, nbatch, n2.as<double>(), st));
    else LSW_TRY(norms2<float>((const float2*)r, n, nbatch, n2.as<double>(), st));
    k_sqrt_inv<<<(nbatch + 255) / 256, 256, 0, st>>>(n2.as<double>(), nrm.as<double>(), inv.as<double>(), nbatch);
    LSW_LAUNCH_CHECK();
    const double ik02 = 1.0 / (g->k * g->k);
    const float k0h = (float)(g->k * g->h);
    if (prec == LSW_C128) {
        k_fno_input<double2><<<gridn(n * nbatch), 256, 0, st>>>((const double2*)r, inv.as<double>(), chi, ik02, k0h,
                                                               (float2*)x, n, nbatch);
        LSW_LAUNCH_CHECK();
        k_scale_rows<double2><<<gridn(n * nbatch), 256, 0, st>>>((const double2*)e, inv.as<double>(), (float2*)t, n,
                                                                nbatch);
    } else {
        k_fno_input<float2><<<gridn(n * nbatch), 256, 0, st>>>((const float2*)r, inv.as<double>(), chi, ik02, k0h,
                                                              (float2*)x, n, nbatch);
        LSW_LAUNCH_CHECK();
        k_scale_rows<float2><<<gridn(n * nbatch), 256, 0, st>>>((const float2*)e, inv.as<double>(), (float2*)t, n,
                                                               nbatch);
    }
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

lsw_status lsw_fno_rotate(void* x, void* t, int nbatch, int64_t n, const float* phases, void* stream) {
    if (!x || !t || !phases || nbatch <= 0 || n <= 0) return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    std::vector<float2> w(nbatch);
    for (int b = 0; b < nbatch; ++b) w[b] = make_float2((float)std::cos((double)phases[b]), (float)std::sin((double)phases[b]));
    DevBuf rot;
    LSW_TRY(rot.alloc(sizeof(float2) * nbatch, st));
    LSW_CUDA(cudaMemcpyAsync(rot.p, w.data(), sizeof(float2) * nbatch, cudaMemcpyHostToDevice, st));
    k_rotate_pairs<<<gridn((long long)n * nbatch), 256, 0, st>>>((float2*)x, (float2*)t, rot.as<float2>(), n, nbatch);
    LSW_LAUNCH_CHECK();
    // the host array w is read by the copy: wait before it goes out of scope
    LSW_CUDA(cudaStreamSynchronize(st));
    return LSW_OK;
}

lsw_status lsw_fno_error(const lsw_fno* f, const void* x, const void* t, int batch, double* num, double* den,
                         void* stream) {
    if (!f || !x || !t || !num || !den || batch <= 0) return LSW_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const long long tot = f->n * batch;
    DevBuf y, part;
    LSW_TRY(y.alloc(sizeof(float2) * tot, st));
    const int nblk = 256;
    LSW_TRY(part.alloc(sizeof(double) * 2 * nblk, st));
    FnoTape tp;
    LSW_TRY(fno_forward(f, (const float2*)x, y.as<float2>(), batch, tp, st));
    k_err_sums<<<nblk, 256, 0, st>>>(y.as<float2>(), (const float2*)t, tot, part.as<double>());
    LSW_LAUNCH_CHECK();
    std::vector<double> h(2 * nblk);
    LSW_CUDA(cudaMemcpyAsync(h.data(), part.p, sizeof(double) * 2 * nblk, cudaMemcpyDeviceToHost, st));
    LSW_CUDA(cudaStreamSynchronize(st));
    double a = 0.0, b = 0.0;
    for (int i = 0; i < nblk; ++i) { a += h[2 * i]; b += h[2 * i + 1]; }
    *num = a;
    *den = b;
    return LSW_OK;
}

lsw_status lsw_fno_apply(const lsw_fno* f, const lsw_green* g, const double* chi, const void* v, void* z, int nbatch,
                         int prec, void* stream) {
    if (!f || !g || !chi || !v || !z || nbatch <= 0 || (prec != LSW_C128 && prec != LSW_C64)) return LSW_ERR_INVALID_ARG;
    return fno_apply_precond(f, g, chi, v, z, nbatch, prec, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
