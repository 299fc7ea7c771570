// Shared-memory Stockham FFT over a set of lines held by one CTA.
//
// Each stage of radix R (4, or 8 for the first stage of an odd power of two,
// or 2 for P = 2) maps butterfly j (0 <= j < P/R) with k = j mod Ns:
//     v_r = x[j + r P/R] * w^(r k P / (Ns R)),   r = 0..R-1
//     V   = DFT_R(v)
//     x'[(j / Ns) Ns R + k + r Ns] = V_r
// (the self-sorting "autosort" formulation: no bit reversal).  Every thread
// loads all of its butterflies into registers before a barrier and stores
// after it, so the stage is done in place.  The host guarantees
// nlines * P / 4 <= NT * MB4 (at most MB4 radix-4 butterflies per thread).
#pragma once

#include "lsw_internal.cuh"

namespace lsw {

template <typename C>
__device__ __forceinline__ C twiddle(const C* __restrict__ tw, int m, bool inv) {
    C w = tw[m];
    if (inv) w.y = -w.y;
    return w;
}

// multiply by -i (forward) or +i (inverse)
template <typename C>
__device__ __forceinline__ C rot90(C a, bool inv) { return inv ? mk(-a.y, a.x) : mk(a.y, -a.x); }

template <typename C>
__device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3, bool inv) {
    C t0 = cadd(v0, v2), t1 = csub(v0, v2), t2 = cadd(v1, v3), t3 = rot90(csub(v1, v3), inv);
    v0 = cadd(t0, t2); v2 = csub(t0, t2); v1 = cadd(t1, t3); v3 = csub(t1, t3);
}

template <typename C>
__device__ __forceinline__ void dft8(C* v, bool inv) {
    // even / odd halves, then combine with w8^k
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4(e0, e1, e2, e3, inv);
    dft4(o0, o1, o2, o3, inv);
    typedef decltype(o0.x) R;
    const R s = (R)0.70710678118654752440;
    // w8^1 = (1 -+ i)/sqrt2, w8^2 = -+ i, w8^3 = (-1 -+ i)/sqrt2
    C w1o1 = inv ? mk((o1.x - o1.y) * s, (o1.x + o1.y) * s) : mk((o1.x + o1.y) * s, (o1.y - o1.x) * s);
    C w2o2 = rot90(o2, inv);
    C w3o3 = inv ? mk((-o3.x - o3.y) * s, (o3.x - o3.y) * s) : mk((o3.y - o3.x) * s, (-o3.x - o3.y) * s);
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, w1o1); v[5] = csub(e1, w1o1);
    v[2] = cadd(e2, w2o2); v[6] = csub(e2, w2o2);
    v[3] = cadd(e3, w3o3); v[7] = csub(e3, w3o3);
}

// One radix-R stage over nlines lines of length P (line l at s + l*lstride).
template <typename C, int R, int NT, int MB>
__device__ __forceinline__ void fft_stage(C* s, int lstride, int nlines, int P, int logP, int Ns,
                                          const C* __restrict__ tw, int twstep, bool inv) {
    const int nbl = P / R;            // butterflies per line
    const int total = nlines * nbl;
    const int lognb = logP - (R == 8 ? 3 : (R == 4 ? 2 : 1));
    C v[MB][R];
#pragma unroll
    for (int i = 0; i < MB; ++i) {
        const int b = threadIdx.x + i * NT;
        if (b < total) {
            const int line = b >> lognb, j = b & (nbl - 1);
            const C* x = s + line * lstride;
            const int k = j & (Ns - 1);
#pragma unroll
            for (int r = 0; r < R; ++r) v[i][r] = x[j + r * nbl];
            if (Ns > 1) {
                const int m = k * (P / (Ns * R)) * twstep;
#pragma unroll
                for (int r = 1; r < R; ++r) v[i][r] = cmul(v[i][r], twiddle(tw, r * m, inv));
            }
            if (R == 4) dft4(v[i][0], v[i][1], v[i][2], v[i][3], inv);
            else if (R == 8) dft8(v[i], inv);
            else { C a = v[i][0]; v[i][0] = cadd(a, v[i][1]); v[i][1] = csub(a, v[i][1]); }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MB; ++i) {
        const int b = threadIdx.x + i * NT;
        if (b < total) {
            const int line = b >> lognb, j = b & (nbl - 1);
            C* x = s + line * lstride;
            const int k = j & (Ns - 1);
            const int base = (j - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) x[base + r * Ns] = v[i][r];
        }
    }
    __syncthreads();
}

// Full transform of nlines lines of length P = 2^logP (P >= 2).
// Caller synchronises before (data in smem) -- this routine ends synchronised.
template <typename C, int NT, int MB4>
__device__ void smem_fft(C* s, int lstride, int nlines, int P, int logP,
                         const C* __restrict__ tw, int twstep, bool inv) {
    if (P == 1) return;
    if (P == 2) { fft_stage<C, 2, NT, (MB4 * 2 > 16 ? 16 : MB4 * 2)>(s, lstride, nlines, P, logP, 1, tw, twstep, inv); return; }
    int Ns = 1;
    if (logP & 1) {
        fft_stage<C, 8, NT, (MB4 / 2 > 0 ? MB4 / 2 : 1)>(s, lstride, nlines, P, logP, Ns, tw, twstep, inv);
        Ns = 8;
    }
    while (Ns < P) {
        fft_stage<C, 4, NT, MB4>(s, lstride, nlines, P, logP, Ns, tw, twstep, inv);
        Ns *= 4;
    }
}

// ------------------------------------------------------------------------
// Line FFTs of N = 2^LOGN points (4 <= N <= 1024) held by T threads of one
// warp, E = N / T entries each, T <= E: thread t owns v[a] = x[T a + t].  The
// transform is an E-point DFT in registers, one twiddle, one transpose
// through shared memory inside the warp (no block barrier) and E / T T-point
// DFTs in registers; the result has the input's layout, v[a] = X[T a + t].
// The transposed line is stored with T + 1 slots per row, which spreads both
// the writes (consecutive lanes) and the reads (stride T + 1) over the banks.
template <int LOGN> struct LineCfg {
    static constexpr int N = 1 << LOGN;
    static constexpr int E = LOGN >= 9 ? 32 : LOGN >= 7 ? 16 : LOGN >= 5 ? 8 : 4;
    static constexpr int T = N / E;
    static constexpr int XCH = E * (T + 1);       // entries of a line's transpose buffer
    static_assert(T <= E && T <= 32 && E % T == 0, "one transpose");
};

// tan(pi r / 64) and sin(pi r / 32), 1 <= r <= 8
__host__ __device__ constexpr double tan64(int r) {
    return r == 1 ? 0.04912684976946725411 : r == 2 ? 0.09849140335716425308 : r == 3 ? 0.14833598753834742875
         : r == 4 ? 0.19891236737965800691 : r == 5 ? 0.25048696019130546160 : r == 6 ? 0.30334668360734239168
         : r == 7 ? 0.35780572131452410467 : 0.41421356237309504880;
}
__host__ __device__ constexpr double sin32(int r) {
    return r == 1 ? 0.09801714032956060199 : r == 2 ? 0.19509032201612826785 : r == 3 ? 0.29028467725446236764
         : r == 4 ? 0.38268343236508977172 : r == 5 ? 0.47139673682599764856 : r == 6 ? 0.55557023301960222474
         : r == 7 ? 0.63439328416364549822 : 0.70710678118654752440;
}

// v times exp(-2 pi i K / 64) (forward) or its conjugate (inverse): an exact
// quarter turn and a turn of at most 45 degrees by three shears,
//   x += t y,  y -= s x,  x += t y,   t = tan(phi / 2), s = sin(phi).
// Three multiply-adds instead of the four operations of a product with
// (cos, sin), and a smaller error: the rounding of a cosine near one (3e-8 at
// cos(pi / 16)), which all entries share, was the largest part of a transform's.
template <int K, bool INV, typename C>
__device__ __forceinline__ C rot64(C v) {
    typedef decltype(v.x) R;
    constexpr int k = (INV ? 64 - (K % 64) : K) % 64;
    constexpr int quarter = (k + 8) / 16 % 4, r = k - (k + 8) / 16 * 16;       // -8 <= r < 8
    const C u = quarter == 0 ? v : quarter == 1 ? mk(v.y, -v.x) : quarter == 2 ? mk(-v.x, -v.y) : mk(-v.y, v.x);
    if constexpr (r == 0) {
        return u;
    } else {
        constexpr R t = (R)(r > 0 ? tan64(r) : -tan64(-r)), sn = (R)(r > 0 ? sin32(r) : -sin32(-r));
        const R x = fma(t, u.y, u.x), y = fma(-sn, x, u.y);
        return mk(fma(t, y, x), y);
    }
}

// Complex sums of the butterflies: for FP32 one packed instruction per
// complex entry instead of two.
template <typename C> __device__ __forceinline__ C vadd(C a, C b) { return cadd(a, b); }
template <typename C> __device__ __forceinline__ C vsub(C a, C b) { return csub(a, b); }
template <> __device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <> __device__ __forceinline__ float2 vsub(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
    return reinterpret_cast<const float2&>(r);
}

// The butterflies of the register transforms, their direction known at compile
// time (dft4 and dft8 above take it as an argument: with these sums and
// selections 2048-point lines took 5% longer).
template <bool INV, typename C>
__device__ __forceinline__ void reg_dft4(C& v0, C& v1, C& v2, C& v3) {
    const C t0 = vadd(v0, v2), t1 = vsub(v0, v2), t2 = vadd(v1, v3), t3 = vsub(v1, v3);
    v0 = vadd(t0, t2);
    v2 = vsub(t0, t2);
    // t1 +- (-i) t3 (forward) or (+i) t3
    const C a = mk(t1.x + t3.y, t1.y - t3.x), b = mk(t1.x - t3.y, t1.y + t3.x);
    v1 = INV ? b : a;
    v3 = INV ? a : b;
}

template <bool INV, typename C>
__device__ __forceinline__ void reg_dft8(C* v) {
    // even / odd halves, then combine with w8^k
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    reg_dft4<INV>(e0, e1, e2, e3);
    reg_dft4<INV>(o0, o1, o2, o3);
    typedef decltype(o0.x) R;
    const R s = (R)0.70710678118654752440;
    // w8^1 = (1 -+ i)/sqrt2, w8^2 = -+ i, w8^3 = (-1 -+ i)/sqrt2; the factor
    // 1/sqrt2 goes into the sums (one rounding less than a product and a sum)
    const C q1 = INV ? mk(o1.x - o1.y, o1.x + o1.y) : mk(o1.x + o1.y, o1.y - o1.x);
    const C q3 = INV ? mk(-o3.x - o3.y, o3.x - o3.y) : mk(o3.y - o3.x, -o3.x - o3.y);
    v[0] = vadd(e0, o0); v[4] = vsub(e0, o0);
    v[1] = mk(fma(s, q1.x, e1.x), fma(s, q1.y, e1.y));
    v[5] = mk(fma(-s, q1.x, e1.x), fma(-s, q1.y, e1.y));
    const C a = mk(e2.x + o2.y, e2.y - o2.x), b = mk(e2.x - o2.y, e2.y + o2.x);
    v[2] = INV ? b : a;
    v[6] = INV ? a : b;
    v[3] = mk(fma(s, q3.x, e3.x), fma(s, q3.y, e3.y));
    v[7] = mk(fma(-s, q3.x, e3.x), fma(-s, q3.y, e3.y));
}

// rows b = 1, 2, 3 of the M / 4 entries c times w_M^(b c)
template <int M, bool INV, int LEFT, typename C>
__device__ __forceinline__ void rot_rows(C* y1, C* y2, C* y3) {
    if constexpr (LEFT > 1) {
        constexpr int c = LEFT - 1, S = 64 / M;
        y1[c] = rot64<S * c, INV>(y1[c]);
        y2[c] = rot64<S * 2 * c, INV>(y2[c]);
        y3[c] = rot64<S * 3 * c, INV>(y3[c]);
        rot_rows<M, INV, LEFT - 1>(y1, y2, y3);
    }
}

// DFT of M entries (1, 2, 4, 8, 16, 32) of a register array, in natural order
template <int M, bool INV, typename C>
__device__ __forceinline__ void reg_dft(C* v) {
    if constexpr (M == 1) {
    } else if constexpr (M == 2) {
        const C a = v[0];
        v[0] = vadd(a, v[1]);
        v[1] = vsub(a, v[1]);
    } else if constexpr (M == 4) {
        reg_dft4<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (M == 8) {
        reg_dft8<INV>(v);
    } else {
        // n = 4 a + b: DFT over a, twiddle w_M^(b c), DFT over b -> X[c + (M / 4) d]
        constexpr int Q = M / 4;
        C y[4][Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            y[0][a] = v[4 * a];
            y[1][a] = v[4 * a + 1];
            y[2][a] = v[4 * a + 2];
            y[3][a] = v[4 * a + 3];
        }
        reg_dft<Q, INV>(y[0]);
        reg_dft<Q, INV>(y[1]);
        reg_dft<Q, INV>(y[2]);
        reg_dft<Q, INV>(y[3]);
        rot_rows<M, INV, Q>(y[1], y[2], y[3]);
#pragma unroll
        for (int c = 0; c < Q; ++c) {
            reg_dft4<INV>(y[0][c], y[1][c], y[2][c], y[3][c]);
            v[c] = y[0][c];
            v[c + Q] = y[1][c];
            v[c + 2 * Q] = y[2][c];
            v[c + 3 * Q] = y[3][c];
        }
    }
}

// v[a] times exp(-2 pi i a / (2 M)) (forward) or its conjugate, a < M <= 32
template <int M, bool INV, int LEFT = M, typename C>
__device__ __forceinline__ void half_shift(C* v) {
    if constexpr (LEFT > 1) {
        constexpr int a = LEFT - 1;
        v[a] = rot64<a * (32 / M), INV>(v[a]);
        half_shift<M, INV, LEFT - 1>(v);
    }
}

// The line transform.  buf: the line's transpose buffer (XCH entries, used by
// this line's threads alone, all in one warp).  Every lane of the warp calls
// it.  odd (the same for the whole warp): the input (forward) or the output
// (inverse) is also multiplied by the half-sample shift w_2N^n or its
// conjugate, n = T a + t.  Of that factor the part that depends on the
// register index is a constant, and the part that depends on the lane
// commutes with the register DFT next to it, so it is part of the twiddle
// table and costs no load.  lt (line_table): w_N^(c t), w_2N^((2c + 1) t) or
// w_2N^(c (2t + 1)) at c T + t.  Both parities run the same code but for the
// constants: with a copy for each, the passes' code outgrew the instruction
// cache.
template <int LOGN, bool INV, typename C>
__device__ __forceinline__ void line_fft(C (&v)[LineCfg<LOGN>::E], C* buf, int t, int odd, const C* __restrict__ lt) {
    constexpr int N = LineCfg<LOGN>::N, E = LineCfg<LOGN>::E, T = LineCfg<LOGN>::T, J = E / T;
    if (!INV && odd) half_shift<E, false>(v);
    reg_dft<E, INV>(v);
    const C* tw = lt + (odd ? (INV ? 2 * N : N) : 0) + t;
#pragma unroll
    for (int c = 0; c < E; ++c) {
        if (c || !INV) {
            C w = tw[c * T];
            if (INV) w.y = -w.y;
            v[c] = cmul(v[c], w);
        }
        buf[c * (T + 1) + t] = v[c];
    }
    __syncwarp();
    C x[E];
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int b = 0; b < T; ++b) x[j * T + b] = buf[(t + T * j) * (T + 1) + b];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < J; ++j) reg_dft<T, INV>(x + j * T);
    if (INV && odd) {
#pragma unroll
        for (int j = 0; j < J; ++j) half_shift<T, true>(x + j * T);
    }
    // X[(t + T j) + E d]: entry a = j + J d of the layout T a + t
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int d = 0; d < T; ++d) v[j + J * d] = x[j * T + d];
}

// Lines of both parities of `cols` columns (a power of two) over groups of T
// threads: group `line` takes column col of parity par, or none (false).  The
// odd ones start on a whole warp, as line_fft wants it.
__host__ __device__ constexpr int parity_lines(int cols, int T) { return 2 * (cols > 32 / T ? cols : 32 / T); }
__host__ __device__ inline bool parity_line(int line, int cols, int T, int& par, int& col) {
    const int half = parity_lines(cols, T) / 2;
    par = line >= half;
    col = line - par * half;
    return col < cols;
}

// Tables of the line transforms, N = 4 .. 1024: three of N entries each.
__host__ __device__ constexpr int line_table(int N) { return 3 * N - 12; }   // first entry of N's tables
constexpr int kLineTables = line_table(2048);                                // entries in all

}  // namespace lsw
