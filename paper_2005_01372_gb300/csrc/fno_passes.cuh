// Fused passes of the Fourier neural operator (fno.cu): spectral transforms
// of whole fields, the per-mode channel mixing, and the pointwise map with
// everything that is added to it.  All complex FP32 on the CUDA cores.
//
// Truncated transforms.  With M = 2m retained wavenumbers k_a (a < m: a, else
// n - M + a) per axis and n = q M, mode a is k_a mod M = a, and
//     X[a] = sum_{b < q} w_n^(b k_a) DFT_M(x[q j + b])[a]
//     x[q j + b] = IDFT_M(conj(w_n^(b k_a)) X[a])[j]
// so a line costs q register DFTs of M points instead of the 8 M n flops of a
// product with the M x n matrix (11 times less at n = 256, M = 32).
// Used for M = 8, 16, 32 and q a power of two, q <= M (fno_fast); other sizes
// go through dense products.
#pragma once

#include "fft.cuh"
#include "lsw_internal.cuh"

namespace lsw {

// tw[a q + b] = w_n^(b k_a), for both axes
__global__ void k_line_twiddles(float2* twz, int nz, float2* twx, int nx, int M) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < nz + nx; g += gridDim.x * blockDim.x) {
        const int n = g < nz ? nz : nx, e = g < nz ? g : g - nz, q = n / M;
        const int a = e / q, b = e - a * q;
        const int k = a < M / 2 ? a : a - M;
        double s, c;
        sincospi(-2.0 * (double)(k * b) / n, &s, &c);
        (g < nz ? twz : twx)[e] = make_float2((float)c, (float)s);
    }
}

// One truncated line held by q lanes of a warp, lane b owning y[j] =
// x[q j + b]: afterwards y[j], j < M / q, is X[b (M / q) + j].  The sum over
// the lanes halves the entries each lane keeps at every step.
template <int M>
__device__ __forceinline__ void trunc_dft(float2 (&y)[M], int q, int b, const float2* __restrict__ tw) {
    reg_dft<M, false>(y);
#pragma unroll
    for (int a = 0; a < M; ++a) y[a] = cmul(y[a], tw[a * q + b]);
#pragma unroll
    for (int t = 0; (2 << t) <= M; ++t) {
        const int s = q >> (t + 1);
        if (s == 0) break;
        const int half = M >> (t + 1);
        const bool up = b & s;
#pragma unroll
        for (int j = 0; j < half; ++j) {
            const float2 send = up ? y[j] : y[j + half], keep = up ? y[j + half] : y[j];
            y[j].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, s);
            y[j].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, s);
        }
    }
}

// Truncated 2D transform of one field per CTA, times scale:
// out[(a + M kx) B W + field] (mode-major, as the mixing reads it).
// The z modes of all columns (M x nx) stay in shared memory between the two
// axes.  Bound by the latency of reading the fields once at 16 warps per SM:
// 1024 fields of 256^2 in 147 us (3.6 TB/s); the dense products took 550 us.
template <int M>
__global__ void __launch_bounds__(256, 2)
k_fno_analysis(const float2* __restrict__ v, int nz, int nx, int nfield, const float2* __restrict__ twz,
               const float2* __restrict__ twx, float scale, float2* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2* T1 = reinterpret_cast<float2*>(sm_raw);          // M rows of nx + 1
    const int f = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int qz = nz / M, qx = nx / M, ld = nx + 1;
    const float2* vf = v + (long long)f * nz * nx;
    float2 y[M];
    {
        const int b = lane & (qz - 1), c = lane / qz, cpw = 32 / qz, keep = M / qz;
        for (int i0 = w * cpw; i0 < nx; i0 += 8 * cpw) {
            const int ix = i0 + c;
            const float2* p = vf + (long long)min(ix, nx - 1) * nz + b;
#pragma unroll
            for (int j = 0; j < M; ++j) y[j] = __ldcs(p + qz * j);
            trunc_dft<M>(y, qz, b, twz);
            if (ix < nx) {
#pragma unroll
                for (int j = 0; j < M; ++j)
                    if (j < keep) T1[(b * keep + j) * ld + ix] = y[j];
            }
        }
    }
    __syncthreads();
    {
        const int b = lane & (qx - 1), r = lane / qx, rpw = 32 / qx, keep = M / qx;
        for (int a0 = w * rpw; a0 < M; a0 += 8 * rpw) {
            const int a = a0 + r;
            const float2* p = T1 + min(a, M - 1) * ld + b;
#pragma unroll
            for (int j = 0; j < M; ++j) y[j] = p[qx * j];
            trunc_dft<M>(y, qx, b, twx);
            if (a < M) {
#pragma unroll
                for (int j = 0; j < M; ++j)
                    if (j < keep)
                        out[(long long)(a + M * (b * keep + j)) * nfield + f] = make_float2(y[j].x * scale, y[j].y * scale);
            }
        }
    }
}

// The x half of the inverse: T1[field][ix][a] = scale sum_kx Zh[a + M kx]
// conj(w_nx^(kx ix)), one CTA per field, Zh mode-major.
template <int M>
__global__ void __launch_bounds__(256)
k_fno_synth_x(const float2* __restrict__ Zt, int nx, int nfield, const float2* __restrict__ twx, float scale,
              float2* __restrict__ T1) {
    __shared__ float2 zs[M * M];
    const int f = blockIdx.x, qx = nx / M;
    for (int e = threadIdx.x; e < M * M; e += 256) {
        const float2 z = Zt[(long long)e * nfield + f];
        zs[e] = make_float2(z.x * scale, z.y * scale);
    }
    __syncthreads();
    float2* o = T1 + (long long)f * nx * M;
    for (int e = threadIdx.x; e < M * qx; e += 256) {
        const int a = e % M, b = e / M;
        float2 y[M];
#pragma unroll
        for (int k = 0; k < M; ++k) y[k] = cmulc(twx[k * qx + b], zs[k * M + a]);
        reg_dft<M, true>(y);
#pragma unroll
        for (int j = 0; j < M; ++j) o[(long long)(qx * j + b) * M + a] = y[j];
    }
}

// Z[mode] = R[mode] V[mode] (W x W times W x B, column-major), a CTA per mode.
__global__ void __launch_bounds__(256)
k_fno_mix(const float2* __restrict__ R, const float2* __restrict__ V, float2* __restrict__ Z, int W, int B) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2* rs = reinterpret_cast<float2*>(sm_raw);      // W x W
    float2* vs = rs + W * W;                             // W x 32
    const long long md = blockIdx.x;
    for (int e = threadIdx.x; e < W * W; e += 256) rs[e] = R[md * W * W + e];
    for (int b0 = 0; b0 < B; b0 += 32) {
        const int nb = min(32, B - b0);
        __syncthreads();
        for (int e = threadIdx.x; e < W * 32; e += 256) vs[e] = e < W * nb ? V[(md * B + b0) * W + e] : make_float2(0.f, 0.f);
        __syncthreads();
        for (int e = threadIdx.x; e < W * 8; e += 256) {
            const int o = e % W, q = e / W * 4;
            if (q >= nb) continue;
            float2 acc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int i = 0; i < W; ++i) {
                const float2 r = rs[o + W * i];
#pragma unroll
                for (int u = 0; u < 4; ++u) cfma(acc[u], r, vs[i + W * (q + u)]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q + u < nb) Z[(md * B + b0 + q + u) * W + o] = acc[u];
        }
    }
}

// Its adjoints: GR[mode] = GZ V^H and GV[mode] = R^H GZ, a CTA per mode.
__global__ void __launch_bounds__(256)
k_fno_mix_grad(const float2* __restrict__ R, const float2* __restrict__ V, const float2* __restrict__ GZ,
               float2* __restrict__ GR, float2* __restrict__ GV, int W, int B) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int ld = W + 1;                                // rows and columns of R are both walked
    float2* rs = reinterpret_cast<float2*>(sm_raw);      // W x W, ld
    float2* vs = rs + W * ld;                            // W x 32
    float2* gs = vs + W * 32;                            // W x 32
    const long long md = blockIdx.x;
    for (int e = threadIdx.x; e < W * W; e += 256) rs[e / W * ld + e % W] = R[md * W * W + e];
    float2 gr[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) gr[u] = make_float2(0.f, 0.f);
    for (int b0 = 0; b0 < B; b0 += 32) {
        const int nb = min(32, B - b0);
        __syncthreads();
        for (int e = threadIdx.x; e < W * 32; e += 256) {
            const bool in = e < W * nb;
            vs[e] = in ? V[(md * B + b0) * W + e] : make_float2(0.f, 0.f);
            gs[e] = in ? GZ[(md * B + b0) * W + e] : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int e = threadIdx.x + 256 * u;
            if (e < W * W) {
                const int o = e % W, i = e / W;
                float2 a = gr[u];
#pragma unroll 4
                for (int b = 0; b < nb; ++b) cfmac(a, vs[i + W * b], gs[o + W * b]);
                gr[u] = a;
            }
        }
        for (int e = threadIdx.x; e < W * 8; e += 256) {
            const int i = e % W, q = e / W * 4;
            if (q >= nb) continue;
            float2 acc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int o = 0; o < W; ++o) {
                const float2 r = rs[o + ld * i];
#pragma unroll
                for (int u = 0; u < 4; ++u) cfmac(acc[u], r, gs[o + W * (q + u)]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q + u < nb) GV[(md * B + b0 + q + u) * W + i] = acc[u];
        }
    }
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const int e = threadIdx.x + 256 * u;
        if (e < W * W) GR[md * W * W + e] = gr[u];
    }
}

__device__ __forceinline__ float gelu_f(float t) { return t * 0.5f * (1.f + erff(t * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_g(float t) {
    return 0.5f * (1.f + erff(t * 0.70710678118654752f)) + t * expf(-0.5f * t * t) * 0.3989422804014327f;
}

// The pointwise map of one sample, with all that is added to it:
//   z[o] = spectral part[o] + sum_i w[o][i] v[i] + bias[o],   out = sigma(z)
// A CTA takes a tile of cells and every channel: thread (cell thread, group of
// 8 outputs) keeps 4 cells x 8 outputs, the input tile and the weights are in
// shared memory, and 32 products cost 4 loads of the tile and 4 of two weights.
// M > 0: the spectral part is the z half of the inverse transform, from
// T1[field][ix][a]; the tile holds whole columns, and the transform's results
// go through the space the input tile takes next.  M == 0: it is read from zin.
// z may be NULL (not kept); v and out may be the same buffer (a CTA reads its
// whole tile before it writes).  Bound by FP32 issue (70% of the issue slots
// busy, 48% with the products' 8 W^2 flops per cell): 32 samples of 256^2 cells
// and 32 channels take 620 us with bias, GELU and both outputs, 460 us for the
// adjoint, where the dense z transform, the product and the elementwise kernel
// took 1.17 ms.
struct PointwiseArgs {
    const float2* v;
    const float2* wt;        // W^T: entry (i, o) at i + W o
    int adjoint;             // out[i] = sum_o conj(w[o][i]) v[o]
    const float2* bias;      // may be NULL
    const float2* T1;
    const float2* twz;
    const float2* zin;
    float2* z;
    float2* out;
    int act;
    long long n;
    int nz, W;
};
// cell threads of a CTA and its threads, by the number of output groups
__host__ __device__ constexpr int pw_cells(int og) { return og == 1 ? 256 : og == 2 ? 128 : 64; }
__host__ __device__ constexpr int pw_threads(int og) { return og > 4 ? 512 : 256; }

template <int M, int NT>
__global__ void __launch_bounds__(NT, (NT == 256 ? 2 : 1))
k_fno_pointwise(PointwiseArgs p) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int W = p.W, og = (W + 7) / 8;
    const int CT = pw_cells(og), cells = 4 * CT, ld = cells + 8;
    float2* ws = reinterpret_cast<float2*>(sm_raw);              // W x 8 og weights
    float2* tile = reinterpret_cast<float2*>(ws + W * 8 * og);   // W x ld
    const long long c0 = (long long)blockIdx.x * cells;
    const int nc = (int)min((long long)cells, p.n - c0);
    const long long base = (long long)blockIdx.y * W * p.n + c0;
    for (int e = threadIdx.x; e < W * 8 * og; e += NT) {
        const int i = e / (8 * og), o = e - i * 8 * og;
        float2 w = make_float2(0.f, 0.f);
        if (o < W) {
            if (p.adjoint) w = cconj(p.wt[o + W * i]);
            else w = p.wt[i + W * o];
        }
        ws[e] = w;
    }
    const int ct = threadIdx.x % CT, g = threadIdx.x / CT;
    const bool live = g < og;
    float2 acc[4][8];
    // the input tile; rows start on 16 bytes when n is even (c0 is)
    auto load_tile = [&]() {
        if ((p.n & 1) == 0) {
            const int per = nc / 2;
            for (int i = threadIdx.x / 32; i < W; i += NT / 32)
                for (int c = threadIdx.x & 31; c < per; c += 32)
                    cp_async<16>(tile + i * ld + 2 * c, p.v + base + i * p.n + 2 * c);
        } else {
            for (int i = threadIdx.x / 32; i < W; i += NT / 32)
                for (int c = threadIdx.x & 31; c < nc; c += 32) cp_async<8>(tile + i * ld + c, p.v + base + i * p.n + c);
        }
    };
    if constexpr (M > 0) {
        const int q = p.nz / M, cols = nc / p.nz;
        const long long ix0 = c0 / p.nz, nx = p.n / p.nz;
        for (int e = threadIdx.x; e < cols * W * q; e += NT) {
            const int b = e % q, r = e / q;
            const int o = r % W, c = r / W;
            const float4* t = reinterpret_cast<const float4*>(
                p.T1 + (((long long)blockIdx.y * W + o) * nx + ix0 + c) * M);
            float2 y[M];
#pragma unroll
            for (int a = 0; a < M; a += 2) {
                const float4 x = t[a / 2];
                y[a] = cmulc(p.twz[a * q + b], make_float2(x.x, x.y));
                y[a + 1] = cmulc(p.twz[(a + 1) * q + b], make_float2(x.z, x.w));
            }
            reg_dft<M, true>(y);
            float2* d = tile + o * ld + c * p.nz + b;
#pragma unroll
            for (int j = 0; j < M; ++j) d[q * j] = y[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int u = 0; u < 8; ++u)
                acc[j][u] = live && 8 * g + u < W ? tile[(8 * g + u) * ld + ct + CT * j] : make_float2(0.f, 0.f);
        __syncthreads();
        load_tile();
    } else {
        load_tile();
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = ct + CT * j;
                acc[j][u] = live && 8 * g + u < W && c < nc ? p.zin[base + (8 * g + u) * p.n + c] : make_float2(0.f, 0.f);
            }
    }
    cp_async_wait_all();
    __syncthreads();
    if (!live) return;
    for (int i = 0; i < W; ++i) {
        float2 x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = tile[i * ld + ct + CT * j];
        const float4* wr = reinterpret_cast<const float4*>(ws + i * 8 * og + 8 * g);
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const float4 w = wr[u / 2];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                cfma(acc[j][u], make_float2(w.x, w.y), x[j]);
                cfma(acc[j][u + 1], make_float2(w.z, w.w), x[j]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int o = 8 * g + u;
        if (o >= W) break;
        const float2 bo = p.bias ? p.bias[o] : make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = ct + CT * j;
            if (c >= nc) continue;
            const float2 t = make_float2(acc[j][u].x + bo.x, acc[j][u].y + bo.y);
            if (p.z) __stcs(p.z + base + o * p.n + c, t);
            p.out[base + o * p.n + c] = p.act ? make_float2(gelu_f(t.x), gelu_f(t.y)) : t;
        }
    }
}

// v[b][w] = P[w][0] x0 + P[w][1] x1 + p[w], every channel of 256 cells per CTA
__global__ void __launch_bounds__(256)
k_fno_lift(const float2* __restrict__ x, const float2* __restrict__ PT, const float2* __restrict__ bias,
           float2* __restrict__ v, long long n, int W) {
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i >= n) return;
    const float2 x0 = x[(long long)blockIdx.y * 2 * n + i], x1 = x[((long long)blockIdx.y * 2 + 1) * n + i];
    float2* o = v + (long long)blockIdx.y * W * n + i;
    for (int w = 0; w < W; ++w) {
        float2 a = make_float2(0.f, 0.f);
        cfma(a, x0, PT[2 * w]);
        cfma(a, x1, PT[2 * w + 1]);
        o[w * n] = cadd(a, bias[w]);
    }
}

// y[b] = x0[b] + sum_w Q[w] v[b][w] + q
__global__ void __launch_bounds__(256)
k_fno_project(const float2* __restrict__ x, const float2* __restrict__ v, const float2* __restrict__ Q,
              const float2* __restrict__ q, float2* __restrict__ y, long long n, int W) {
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i >= n) return;
    const float2* p = v + (long long)blockIdx.y * W * n + i;
    float2 a = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int w = 0; w < W; ++w) cfma(a, p[w * n], Q[w]);
    y[(long long)blockIdx.y * n + i] = cadd(cadd(x[(long long)blockIdx.y * 2 * n + i], a), q[0]);
}

// G[b][w] = conj(Q[w]) Gy[b]
__global__ void __launch_bounds__(256)
k_fno_project_grad(const float2* __restrict__ Gy, const float2* __restrict__ Q, float2* __restrict__ G, long long n,
                   int W) {
    const long long i = blockIdx.x * 256LL + threadIdx.x;
    if (i >= n) return;
    const float2 g = Gy[(long long)blockIdx.y * n + i];
    float2* o = G + (long long)blockIdx.y * W * n + i;
    for (int w = 0; w < W; ++w) o[w * n] = cmulc(Q[w], g);
}

// part[field chunk] = sum of g over chunk entries of a field, after
// g <- g sigma'(z) in place (z not NULL)
constexpr int kFnoSumChunk = 8192;
__global__ void __launch_bounds__(256)
k_fno_act_sum(float2* __restrict__ g, const float2* __restrict__ z, long long n, float2* __restrict__ part) {
    const long long f = blockIdx.y;
    const long long i0 = (long long)blockIdx.x * kFnoSumChunk, i1 = min(n, i0 + kFnoSumChunk);
    float sx = 0, sy = 0;
#pragma unroll 4
    for (long long i = i0 + threadIdx.x; i < i1; i += 256) {
        float2 a = g[f * n + i];
        if (z) {
            const float2 t = z[f * n + i];
            a.x *= gelu_g(t.x);
            a.y *= gelu_g(t.y);
            g[f * n + i] = a;
        }
        sx += a.x;
        sy += a.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    __shared__ float2 red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(sx, sy);
    __syncthreads();
    if (threadIdx.x == 0) {
        float2 a = make_float2(0.f, 0.f);
        for (int i = 0; i < 8; ++i) a = cadd(a, red[i]);
        part[f * gridDim.x + blockIdx.x] = a;
    }
}

// out[w] = sum over samples and chunks of part, a warp per channel
__global__ void k_fno_sum_channels(const float2* __restrict__ part, int chunks, int W, int B, float2* __restrict__ out) {
    const int w = blockIdx.x, lane = threadIdx.x;
    float sx = 0, sy = 0;
    for (int e = lane; e < B * chunks; e += 32) {
        const int b = e / chunks;
        const float2 a = part[((long long)b * W + w) * chunks + e - b * chunks];
        sx += a.x;
        sy += a.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    if (lane == 0) out[w] = make_float2(sx, sy);
}

}  // namespace lsw
