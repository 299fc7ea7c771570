// The Lippmann-Schwinger operator through zero-padded FFTs (Sec. 2.2, Eq. 4),
// and the Green table / spectra it multiplies by.
//
// A field on a (bz x bx) box is convolved with the Green table on the
// (2bz x 2bx) padded grid in three passes; the padded half of each axis is
// never stored:
//   pass A  (per column)  chi-multiply, zero-pad, FFT along z     -> T[kz][ix]
//   pass B  (per row kz)  zero-pad, FFT along x, multiply by the quarter
//                         spectrum, inverse FFT along x, crop      -> T[kz][ix]
//   pass C  (per column)  inverse FFT along z, crop, epilogue     -> y
// T holds 2bz x bx complex per field.  The spectrum carries the 1/(4 bz bx)
// of the inverse transform.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "fft.cuh"
#include "lsw_internal.cuh"

namespace lsw {

namespace {

template <typename R> struct FftCfg;
template <> struct FftCfg<float>  { static constexpr int NT = 256, MB4 = 8; };
template <> struct FftCfg<double> { static constexpr int NT = 256, MB4 = 4; };

// elements of one CTA's line set: nlines * P <= 4 * NT * MB4
template <typename R> constexpr int fft_capacity() { return 4 * FftCfg<R>::NT * FftCfg<R>::MB4; }


// 16-byte accesses: two complex64 entries or one complex128
template <typename C> struct Vec16;
template <> struct Vec16<float2> { typedef float4 T; };
template <> struct Vec16<double2> { typedef double2 T; };

struct DevGeom {
    int bz, bx, logbz;
    const double* chi;
    int chi_ld;
    const int2* origin;
    int vpb;
};

__device__ __forceinline__ int2 box_origin(const DevGeom& g, int b) {
    return g.origin ? g.origin[b / g.vpb] : make_int2(0, 0);
}

// ----------------------------------------------------------------- pass A
template <typename R, int NT, int MB4>
__global__ void __launch_bounds__(NT)
k_pass_a(const typename Cx<R>::T* __restrict__ u, DevGeom geo, int pz, int logpz, int cx, int logcx,
         int lstride, const typename Cx<R>::T* __restrict__ tw, int twstep, int adjoint,
         typename Cx<R>::T* __restrict__ T) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C* sm = reinterpret_cast<C*>(sm_raw);
    const int b = blockIdx.y;
    const int ix0 = blockIdx.x * cx;
    const int2 org = box_origin(geo, b);           // (z0, x0)
    const long long nbox = (long long)geo.bz * geo.bx;
    const C* ub = u + b * nbox;
    const int tot = cx * pz;
    for (int e = threadIdx.x; e < tot; e += NT) {
        const int c = e >> logpz, iz = e & (pz - 1);
        C v = czero<C>();
        if (iz < geo.bz) {
            const int ix = ix0 + c;
            v = ub[(long long)ix * geo.bz + iz];
            if (adjoint) {
                v.y = -v.y;
            } else {
                const R ch = (R)geo.chi[(long long)(org.y + ix) * geo.chi_ld + org.x + iz];
                v = cscale(v, ch);
            }
        }
        sm[c * lstride + iz] = v;
    }
    __syncthreads();
    smem_fft<C, NT, MB4>(sm, lstride, cx, pz, logpz, tw, twstep, false);
    C* Tb = T + (long long)b * pz * geo.bx;
    for (int e = threadIdx.x; e < tot; e += NT) {
        const int kz = e >> logcx, c = e & (cx - 1);
        Tb[(long long)kz * geo.bx + ix0 + c] = sm[c * lstride + kz];
    }
}

// ----------------------------------------------------------------- pass B
template <typename R, int NT, int MB4>
__global__ void __launch_bounds__(NT)
k_pass_b(typename Cx<R>::T* __restrict__ T, int bx, int pz, int px, int logpx, int rz, int logrz,
         int lstride, const typename Cx<R>::T* __restrict__ specq, int qz,
         const typename Cx<R>::T* __restrict__ tw, int twstep) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C* sm = reinterpret_cast<C*>(sm_raw);
    const int b = blockIdx.y;
    const int kz0 = blockIdx.x * rz;
    C* Tb = T + (long long)b * pz * bx;
    const int tot = rz * px;
    for (int e = threadIdx.x; e < tot; e += NT) {
        const int r = e >> logpx, ix = e & (px - 1);
        sm[r * lstride + ix] = ix < bx ? Tb[(long long)(kz0 + r) * bx + ix] : czero<C>();
    }
    __syncthreads();
    smem_fft<C, NT, MB4>(sm, lstride, rz, px, logpx, tw, twstep, false);
    for (int e = threadIdx.x; e < tot; e += NT) {
        const int r = e >> logpx, kx = e & (px - 1);
        const int kz = kz0 + r;
        const int qx = min(kx, px - kx), qzz = min(kz, pz - kz);
        sm[r * lstride + kx] = cmul(sm[r * lstride + kx], specq[qx * qz + qzz]);
    }
    __syncthreads();
    smem_fft<C, NT, MB4>(sm, lstride, rz, px, logpx, tw, twstep, true);
    const int totc = rz * bx;
    for (int e = threadIdx.x; e < totc; e += NT) {
        const int r = e / bx, ix = e - r * bx;
        Tb[(long long)(kz0 + r) * bx + ix] = sm[r * lstride + ix];
    }
}

// ----------------------------------------------------------------- pass C
template <typename R, int NT, int MB4>
__global__ void __launch_bounds__(NT)
k_pass_c(const typename Cx<R>::T* __restrict__ T, DevGeom geo, int pz, int logpz, int cx, int logcx,
         int lstride, const typename Cx<R>::T* __restrict__ tw, int twstep, int mode,
         const typename Cx<R>::T* __restrict__ u, const typename Cx<R>::T* __restrict__ u0,
         typename Cx<R>::T* __restrict__ y) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C* sm = reinterpret_cast<C*>(sm_raw);
    const int b = blockIdx.y;
    const int ix0 = blockIdx.x * cx;
    const C* Tb = T + (long long)b * pz * geo.bx;
    const int tot = cx * pz;
    for (int e = threadIdx.x; e < tot; e += NT) {
        const int kz = e >> logcx, c = e & (cx - 1);
        sm[c * lstride + kz] = Tb[(long long)kz * geo.bx + ix0 + c];
    }
    __syncthreads();
    smem_fft<C, NT, MB4>(sm, lstride, cx, pz, logpz, tw, twstep, true);
    const long long nbox = (long long)geo.bz * geo.bx;
    const int2 org = box_origin(geo, b);
    const int tote = cx * geo.bz;
    for (int e = threadIdx.x; e < tote; e += NT) {
        const int c = e >> geo.logbz, iz = e & (geo.bz - 1);
        const int ix = ix0 + c;
        const long long idx = b * nbox + (long long)ix * geo.bz + iz;
        C g = sm[c * lstride + iz];
        C out;
        switch (mode) {
            case LSW_OP_FORWARD:
                out = u0 ? cadd(u0[idx], g) : g;
                break;
            case LSW_OP_RESIDUAL:
                out = csub(u[idx], g);
                if (u0) out = csub(out, u0[idx]);
                break;
            case LSW_OP_ADJOINT: {
                const R ch = (R)geo.chi[(long long)(org.y + ix) * geo.chi_ld + org.x + iz];
                out = mk(g.x * ch, -g.y * ch);
                break;
            }
            default:
                out = g;
        }
        y[idx] = out;
    }
}

// ------------------------------------------------- register-FFT passes
// The same three passes with register-resident line FFTs, for box sides of
// 4 .. 1024 cells.  A line of N cells zero-padded to 2N has the spectrum
//   X[2k] = DFT_N(x)[k],   X[2k + 1] = DFT_N(x w_2N^n)[k],
// and the first N entries of an inverse transform of length 2N are
//   y[n] = IDFT_N(Y[even])[n] + conj(w_2N^n) IDFT_N(Y[odd])[n],
// so the padding costs no butterfly: the two halves (parities) of a line are
// N-point transforms, run by two thread groups of T threads (LineCfg) that
// meet only where their results are added.
//
// T holds, per field, the rows kz' = parity * bz + k (kz = 2k + parity) in
// blocks: kblk rows (64 bytes of one column) lie next to each other for
// ix = 0, 1, ..., bx - 1, and the blocks follow each other.  A column's write
// (pass A) and read (pass C) move whole 64-byte segments, and pass B reads
// and writes its rows of a block in runs of at least 32 bytes.
//
// What bounds them: shared-memory wavefronts (63% of peak in pass B) and FP32
// issue, at the 16 - 32 warps the registers leave; FP64 is bound by its pipe
// (85% busy).  A line's transform moves every entry twice through shared
// memory (one transpose, inside a warp) where the radix-8 passes these
// replaced moved it six times with two block barriers each.  RESIDUAL on one
// GB300, before -> now: 256^2, 32 fields 95 -> 56 us; 1024^2, 16 fields 1098 ->
// 536 us; ADJOINT 256 x 1024, 30 fields 487 -> 216 us; FP64 256^2, 32 fields
// 1401 -> 1272 us.  The complex64 results are nearer to FP64's at every size
// (256^2: 1.97e-7 -> 1.63e-7, 1024^2: 2.20e-7 -> 1.85e-7; rot64).
template <typename C> __host__ __device__ constexpr int kblk() { return 64 / (int)sizeof(C); }
template <typename C> __device__ __forceinline__ long long tile_index(int kz, int ix, int bx) {
    constexpr int KB = kblk<C>();
    return (long long)(kz / KB) * bx * KB + (long long)ix * KB + (kz % KB);
}
// entries between the buffers of two lines: the transpose buffer and, in pass
// B, a row, rounded so that the transposing stores of 2 (c64: pairs) or 1
// (c128) rows per lane fall into different banks
template <typename C, int LOGN, int ROWS> __host__ __device__ constexpr int line_stride() {
    constexpr int need = LineCfg<LOGN>::XCH > LineCfg<LOGN>::N ? LineCfg<LOGN>::XCH : LineCfg<LOGN>::N;
    constexpr int want = sizeof(C) == 16 ? 2 : ROWS >= kblk<C>() ? 10 : 4, mod = sizeof(C) == 16 ? 8 : 16;
    return need + ((want - need) % mod + mod) % mod;
}
// A line's two halves after the inverse transforms: group par keeps the
// entries a = par E / 2 .. of the sum (v[0 .. E / 2)), handing the others to
// its partner (buffer `other`) in its own buffer.  Called by the whole CTA.
template <int LOGN, typename C>
__device__ __forceinline__ void add_parities(C (&v)[LineCfg<LOGN>::E], C* buf, const C* other, int t, int par) {
    constexpr int E = LineCfg<LOGN>::E, T = LineCfg<LOGN>::T, EH = E / 2;
    if (par) {
#pragma unroll
        for (int a = 0; a < EH; ++a) buf[T * a + t] = v[a];
    } else {
#pragma unroll
        for (int a = EH; a < E; ++a) buf[T * a + t] = v[a];
    }
    __syncthreads();
    if (par) {
#pragma unroll
        for (int a = 0; a < EH; ++a) v[a] = cadd(other[T * (EH + a) + t], v[EH + a]);
    } else {
#pragma unroll
        for (int a = 0; a < EH; ++a) v[a] = cadd(v[a], other[T * a + t]);
    }
}
// T is read and written past L1 (every sector is used once per pass; L1 is
// left to the twiddles), u0 and y evict first from L2, where T is to stay.
// Threads of a CTA.  FP64 128: its pipe is the bound (2 lanes per SM and cycle),
// so that few fields want their lines on many SMs, and many fields gain by the
// finer tail (with 256: one field of 256 x 256 137 us instead of 78, 8 fields of 1024 x
// 256 1.49 ms instead of 1.37).
template <typename R> constexpr int fft_threads() { return sizeof(R) == 8 ? 128 : 256; }
// launch bounds: CTAs per SM the registers are to allow (E complex entries
// and about as many temporaries per thread, more in pass B)
template <typename R, int LOGN, bool PASS_B> constexpr int fft_ctas() {
    return sizeof(R) == 8 ? (LineCfg<LOGN>::E == 32 ? 2 : 4)
                          : (LineCfg<LOGN>::E == 32 ? 2 : LineCfg<LOGN>::E == 16 && PASS_B ? 3 : 4);
}

// Pass A: a CTA takes COLS columns of `per` consecutive fields.  chi is kept
// as R in shared memory for all of them: the FP64 -> FP32 conversion runs on
// the FP64 pipe (2 lanes per SM and cycle) and was 42% of its time when both
// parity groups converted every cell of every field.
// Programmatic dependent launch: the passes follow each other on one stream,
// and each is launched while its predecessor still runs.  A pass lets its
// successor's CTAs start as soon as all of its own have, and touches nothing
// an earlier kernel writes (or writes anything one reads) before
// pdl_wait(), which returns once the whole preceding grid has finished.
__device__ __forceinline__ void pdl_start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename R, int LOGN>
__global__ void __launch_bounds__(fft_threads<R>(), (fft_ctas<R, LOGN, false>()))
k_fa(const typename Cx<R>::T* __restrict__ u, DevGeom geo, const typename Cx<R>::T* __restrict__ lt, int adjoint,
     typename Cx<R>::T* __restrict__ T_, int nbatch, int per) {
    typedef typename Cx<R>::T C;
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, NT = fft_threads<R>(), COLS = NT / (2 * T);
    constexpr int LS = line_stride<C, LOGN, kblk<C>()>();
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int t = threadIdx.x % T, line = threadIdx.x / T;
    const int par = line / COLS, l = line - par * COLS;
    C* buf = reinterpret_cast<C*>(sm_raw) + line * LS;
    R* chs = reinterpret_cast<R*>(reinterpret_cast<C*>(sm_raw) + 2 * COLS * LS);    // COLS x N
    const int ix0 = blockIdx.x * COLS, ix = ix0 + l;
    const bool valid = ix < geo.bx;
    const int b0 = blockIdx.y * per, b1 = min(nbatch, b0 + per);
    pdl_start_next();
    pdl_wait();
    int box = -1;
    for (int b = b0; b < b1; ++b) {
        if (!adjoint && (geo.origin ? b / geo.vpb : 0) != box) {
            box = geo.origin ? b / geo.vpb : 0;
            const int2 org = box_origin(geo, b);
            if (b != b0) __syncthreads();
#pragma unroll 4
            for (int e = threadIdx.x; e < COLS * N; e += NT) {
                const int c = e / N, iz = e % N;
                if (ix0 + c < geo.bx) chs[e] = (R)geo.chi[(long long)(org.y + ix0 + c) * geo.chi_ld + org.x + iz];
            }
            __syncthreads();
        }
        const C* ub = u + ((long long)b * geo.bx + (valid ? ix : 0)) * N;
        C v[E];
#pragma unroll
        for (int a = 0; a < E; ++a) v[a] = ub[T * a + t];
        if (adjoint) {
#pragma unroll
            for (int a = 0; a < E; ++a) v[a].y = -v[a].y;
        } else {
#pragma unroll
            for (int a = 0; a < E; ++a) v[a] = cscale(v[a], chs[l * N + T * a + t]);
        }
        line_fft<LOGN, false>(v, buf, t, par, lt);
        if (valid) {
            C* Tb = T_ + (long long)b * 2 * N * geo.bx;
#pragma unroll
            for (int a = 0; a < E; ++a) __stcg(Tb + tile_index<C>(par * N + T * a + t, ix, geo.bx), v[a]);
        }
    }
}

// Pass B: a CTA takes ROWS consecutive rows kz' of one field, turns them into
// rows of a shared-memory tile, and two groups of T threads per row transform,
// multiply by the spectrum and transform back one parity each; the odd group
// hands its half over in shared memory.  The even group's transposes reuse the
// row itself, once both groups have read it.  Rows past the field's end are
// transformed as they lie in shared memory and not stored.
template <typename R, int LOGN, int NTB>
__global__ void __launch_bounds__(NTB, (NTB == fft_threads<R>() ? fft_ctas<R, LOGN, true>() : 1))
k_fb(typename Cx<R>::T* __restrict__ T_, int bz, const typename Cx<R>::T* __restrict__ spt,
     const typename Cx<R>::T* __restrict__ lt) {
    typedef typename Cx<R>::T C;
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, ROWS = NTB / (2 * T), KB = kblk<C>();
    constexpr int RB = ROWS < KB ? ROWS : KB;           // rows of one kz-block in this CTA
    constexpr int PK = sizeof(C) == 16 ? 1 : 2;         // rows per 16-byte access
    constexpr int LS = line_stride<C, LOGN, ROWS>();
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C* tile = reinterpret_cast<C*>(sm_raw);             // ROWS rows, then ROWS buffers of the odd groups
    C* spec = tile + 2 * ROWS * LS;                     // the rows' spectra, N + 1 entries each
    const int row0 = blockIdx.x * ROWS, pz = 2 * bz;
    const int nrun = (min(ROWS, pz - row0) / PK) * N;   // 16-byte accesses
    C* Tb = T_ + (long long)blockIdx.y * pz * N;
    // access e: rows r, r + 1 (c128: r) of kz-block blk at ix
    auto where = [&](int e, int& r, int& ix) -> C* {
        const int rp = e % (RB / PK), q = e / (RB / PK);
        const int blk = q / N;
        ix = q - blk * N;
        r = blk * KB + rp * PK;
        return Tb + ((long long)(row0 / KB + blk) * N + ix) * KB + (row0 % KB) + rp * PK;
    };
    pdl_start_next();
    pdl_wait();
    // the spectra arrive asynchronously behind the rows (after the wait: the
    // kernel that made them may be the one before pass A)
    for (int r = threadIdx.x >> 5; r < ROWS; r += NTB / 32) {
        // kz = 2k + (kz parity) of row kz'; the spectrum's row holds the even
        // qx (N / 2 + 1 entries) and then the odd ones
        const int kr = min(row0 + r, pz - 1);
        const int kz = kr < bz ? 2 * kr : 2 * (kr - bz) + 1;
        const C* sp = spt + (long long)min(kz, pz - kz) * (N + 1);
        for (int e = threadIdx.x & 31; e <= N; e += 32) cp_async<sizeof(C)>(spec + r * (N + 1) + e, sp + e);
    }
#pragma unroll 8
    for (int e = threadIdx.x; e < nrun; e += NTB) {
        int r, ix;
        const C* p = where(e, r, ix);
        const auto w = __ldcg(reinterpret_cast<const typename Vec16<C>::T*>(p));
        if constexpr (PK == 2) {
            tile[r * LS + ix] = mk(w.x, w.y);
            tile[(r + 1) * LS + ix] = mk(w.z, w.w);
        } else {
            tile[r * LS + ix] = w;
        }
    }
    __syncthreads();
    const int t = threadIdx.x % T, line = threadIdx.x / T;
    const int par = line / ROWS, row = line - par * ROWS;
    C* rowp = tile + row * LS;
    C* buf = tile + line * LS;
    C v[E];
#pragma unroll
    for (int a = 0; a < E; ++a) v[a] = rowp[T * a + t];
    cp_async_wait_all();
    __syncthreads();
    line_fft<LOGN, false>(v, buf, t, par, lt);
    const C* sp = spec + row * (N + 1) + par * (N / 2 + 1);
#pragma unroll
    for (int a = 0; a < E; ++a) v[a] = cmul(v[a], sp[min(T * a + t, N - par - (T * a + t))]);
    line_fft<LOGN, true>(v, buf, t, par, lt);
    add_parities<LOGN>(v, buf, buf + (par ? -ROWS * LS : ROWS * LS), t, par);
    // both groups' halves of the row
    constexpr int EH = E / 2;
#pragma unroll
    for (int a = 0; a < EH; ++a) rowp[T * (par * EH + a) + t] = v[a];
    __syncthreads();
#pragma unroll 8
    for (int e = threadIdx.x; e < nrun; e += NTB) {
        int r, ix;
        C* p = where(e, r, ix);
        typename Vec16<C>::T w;
        if constexpr (PK == 2) {
            const C w0 = tile[r * LS + ix], w1 = tile[(r + 1) * LS + ix];
            w.x = w0.x; w.y = w0.y; w.z = w1.x; w.w = w1.y;
        } else {
            w = tile[r * LS + ix];
        }
        __stcg(reinterpret_cast<typename Vec16<C>::T*>(p), w);
    }
}

// The epilogue of one group's half of a column: entry a of the EH in v lies
// at iz0 + T a of the column, which starts at col0 (chi's at ch); the fields
// it is combined with are all loaded before the first is used.
template <typename R, typename C, int E, int EH>
__device__ __forceinline__ void column_out(C (&v)[E], const C* __restrict__ u, const C* __restrict__ u0,
                                           C* __restrict__ y, const double* __restrict__ ch, long long col0, int iz0,
                                           int T, int mode, std::integral_constant<int, EH>) {
    const long long off = col0 + iz0;
    if (mode == LSW_OP_RESIDUAL) {
        C x[EH];
#pragma unroll
        for (int a = 0; a < EH; ++a) x[a] = __ldcs(u + off + T * a);
#pragma unroll
        for (int a = 0; a < EH; ++a) v[a] = csub(x[a], v[a]);
        if (u0) {
#pragma unroll
            for (int a = 0; a < EH; ++a) x[a] = __ldcs(u0 + off + T * a);
#pragma unroll
            for (int a = 0; a < EH; ++a) v[a] = csub(v[a], x[a]);
        }
    } else if (mode == LSW_OP_FORWARD) {
        if (u0) {
            C x[EH];
#pragma unroll
            for (int a = 0; a < EH; ++a) x[a] = __ldcs(u0 + off + T * a);
#pragma unroll
            for (int a = 0; a < EH; ++a) v[a] = cadd(x[a], v[a]);
        }
    } else if (mode == LSW_OP_ADJOINT) {
        R x[EH];
#pragma unroll
        for (int a = 0; a < EH; ++a) x[a] = (R)ch[iz0 + T * a];
#pragma unroll
        for (int a = 0; a < EH; ++a) v[a] = mk(v[a].x * x[a], -v[a].y * x[a]);
    }
#pragma unroll
    for (int a = 0; a < EH; ++a) __stcs(y + off + T * a, v[a]);
}

template <typename R, int LOGN>
__global__ void __launch_bounds__(fft_threads<R>(), (fft_ctas<R, LOGN, false>()))
k_fc(const typename Cx<R>::T* __restrict__ T_, DevGeom geo, const typename Cx<R>::T* __restrict__ lt, int mode,
     const typename Cx<R>::T* __restrict__ u, const typename Cx<R>::T* __restrict__ u0,
     typename Cx<R>::T* __restrict__ y) {
    typedef typename Cx<R>::T C;
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, NT = fft_threads<R>(), COLS = NT / (2 * T);
    constexpr int LS = line_stride<C, LOGN, kblk<C>()>();
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int t = threadIdx.x % T, line = threadIdx.x / T;
    const int par = line / COLS, l = line - par * COLS;
    C* buf = reinterpret_cast<C*>(sm_raw) + line * LS;
    const int b = blockIdx.y, ix = blockIdx.x * COLS + l;
    const bool valid = ix < geo.bx;
    const C* Tb = T_ + (long long)b * 2 * N * geo.bx;
    pdl_start_next();
    pdl_wait();
    if (valid && (mode == LSW_OP_RESIDUAL || mode == LSW_OP_FORWARD)) {
        // the fields this half of the column is combined with: into L2 while
        // the transform runs
        const long long lo = ((long long)b * geo.bx + ix) * N + par * (N / 2);
        for (int i = t * (128 / (int)sizeof(C)); i < N / 2; i += T * (128 / (int)sizeof(C))) {
            if (mode == LSW_OP_RESIDUAL) prefetch_l2(u + lo + i);
            if (u0) prefetch_l2(u0 + lo + i);
        }
    }
    C v[E];
#pragma unroll
    for (int a = 0; a < E; ++a) v[a] = __ldcg(Tb + tile_index<C>(par * N + T * a + t, valid ? ix : 0, geo.bx));
    line_fft<LOGN, true>(v, buf, t, par, lt);
    add_parities<LOGN>(v, buf, buf + (par ? -COLS * LS : COLS * LS), t, par);
    if (!valid) return;
    constexpr int EH = E / 2;
    const int2 org = box_origin(geo, b);
    column_out<R>(v, u, u0, y, geo.chi + (long long)(org.y + ix) * geo.chi_ld + org.x,
                  ((long long)b * geo.bx + ix) * N, par * EH * T + t, T, mode, std::integral_constant<int, EH>());
}

// --------------------------------------------- small fields: one launch
// Boxes of few cells finish in one launch: a cluster of CL thread blocks takes
// a field through all three passes, the intermediate T lying in the blocks'
// shared memory, each holding 2 bz / CL of its rows.  Pass A writes its
// columns into the owners' rows (distributed shared memory), pass B works on
// a block's own rows, pass C reads its columns back.  The line transforms and
// the epilogues are those of the three-pass kernels, so the results are the same
// bit for bit.  Bound by its chain of latencies (three line transforms, two
// cluster barriers): one 64 x 64 c64 field takes 8.2 us on the GPU (three
// launches: 7.6, overlapping their starts), but a call costs the host 13.9 us
// instead of 19.5, with one launch and no work array.
constexpr int kSmallThreads = 256;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// the address of this block's shared variable at p in block `rank`
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_load(uint32_t a, float2& v) {
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void cluster_load(uint32_t a, double2& v) {
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
}

// The block's share of a field: columns ix0 .. ix0 + cols, rows of T
// rank * rows ..; row r of T at rows + r * ls in shared memory.
template <typename C> struct SmallField {
    int logrows, cols, ix0, ls;
    C* rows;
    C* bufs;                                 // transpose buffers of the block's lines
    __device__ __forceinline__ uint32_t remote(int kz, int ix) const {
        return cluster_addr(rows + (kz & ((1 << logrows) - 1)) * ls + ix, (uint32_t)(kz >> logrows));
    }
};

template <typename R, int LOGN, typename C>
__device__ __forceinline__ void small_a(const SmallField<C>& f, const C* __restrict__ ub, const double* __restrict__ chb,
                                        int chi_ld, int adjoint, const C* __restrict__ lt) {
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, LINES = kSmallThreads / T, LS = line_stride<C, LOGN, kblk<C>()>();
    const int t = threadIdx.x % T;
    C* buf = f.bufs + (threadIdx.x / T) * LS;
    for (int l0 = 0; l0 < parity_lines(f.cols, T); l0 += LINES) {
        int par, col;
        const bool valid = parity_line(l0 + threadIdx.x / T, f.cols, T, par, col);
        const int ix = f.ix0 + (valid ? col : 0);
        const C* uc = ub + (long long)ix * N;
        const double* ch = chb + (long long)ix * chi_ld;
        C v[E];
#pragma unroll
        for (int a = 0; a < E; ++a) v[a] = uc[T * a + t];
        if (adjoint) {
#pragma unroll
            for (int a = 0; a < E; ++a) v[a].y = -v[a].y;
        } else {
            double c[E];
#pragma unroll
            for (int a = 0; a < E; ++a) c[a] = ch[T * a + t];
#pragma unroll
            for (int a = 0; a < E; ++a) v[a] = cscale(v[a], (R)c[a]);
        }
        line_fft<LOGN, false>(v, buf, t, par, lt);
        if (l0 == 0) cluster_wait();         // every block of the cluster has started
        if (valid) {
#pragma unroll
            for (int a = 0; a < E; ++a) cluster_store(f.remote(par * N + T * a + t, ix), v[a]);
        }
    }
}

// spec: the spectra of the block's rows, N + 1 entries each
template <int LOGN, typename C>
__device__ __forceinline__ void small_b(const SmallField<C>& f, const C* spec, const C* __restrict__ lt) {
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, HALF = kSmallThreads / T / 2, LS = line_stride<C, LOGN, kblk<C>()>();
    const int t = threadIdx.x % T, line = threadIdx.x / T, par = line / HALF, nrows = 1 << f.logrows;
    C* buf = f.bufs + line * LS;
    for (int r0 = 0; r0 < nrows; r0 += HALF) {
        const int row = r0 + line - par * HALF;
        const bool valid = row < nrows;
        C* rowp = f.rows + (valid ? row : 0) * f.ls;
        if (r0) __syncthreads();
        C v[E];
#pragma unroll
        for (int a = 0; a < E; ++a) v[a] = rowp[T * a + t];
        line_fft<LOGN, false>(v, buf, t, par, lt);
        const C* sp = spec + (valid ? row : 0) * (N + 1) + par * (N / 2 + 1);
#pragma unroll
        for (int a = 0; a < E; ++a) v[a] = cmul(v[a], sp[min(T * a + t, N - par - (T * a + t))]);
        line_fft<LOGN, true>(v, buf, t, par, lt);
        add_parities<LOGN>(v, buf, buf + (par ? -HALF * LS : HALF * LS), t, par);
        constexpr int EH = E / 2;
        if (valid) {
#pragma unroll
            for (int a = 0; a < EH; ++a) rowp[T * (par * EH + a) + t] = v[a];
        }
    }
}

template <typename R, int LOGN, typename C>
__device__ __forceinline__ void small_c(const SmallField<C>& f, const C* __restrict__ ub, const C* __restrict__ u0b,
                                        C* __restrict__ yb, const double* __restrict__ chb, int chi_ld, int mode,
                                        const C* __restrict__ lt) {
    typedef LineCfg<LOGN> L;
    constexpr int N = L::N, E = L::E, T = L::T, HALF = kSmallThreads / T / 2, LS = line_stride<C, LOGN, kblk<C>()>();
    const int t = threadIdx.x % T, line = threadIdx.x / T, par = line / HALF;
    C* buf = f.bufs + line * LS;
    for (int c0 = 0; c0 < f.cols; c0 += HALF) {
        const int col = c0 + line - par * HALF;
        const bool valid = col < f.cols;
        const int ix = f.ix0 + (valid ? col : 0);
        if (c0) __syncthreads();
        C v[E];
#pragma unroll
        for (int a = 0; a < E; ++a) cluster_load(f.remote(par * N + T * a + t, ix), v[a]);
        if (c0 + HALF >= f.cols) cluster_arrive();
        line_fft<LOGN, true>(v, buf, t, par, lt);
        add_parities<LOGN>(v, buf, buf + (par ? -HALF * LS : HALF * LS), t, par);
        if (valid) {
            constexpr int EH = E / 2;
            column_out<R>(v, ub, u0b, yb, chb + (long long)ix * chi_ld, (long long)ix * N, par * EH * T + t, T, mode,
                          std::integral_constant<int, EH>());
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(kSmallThreads, sizeof(R) == 8 ? 1 : 2)
k_small(const typename Cx<R>::T* __restrict__ u, DevGeom geo, int logrows, const typename Cx<R>::T* __restrict__ spt,
        const typename Cx<R>::T* __restrict__ tab, int mode, const typename Cx<R>::T* __restrict__ u0,
        typename Cx<R>::T* __restrict__ y, int cl) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int b = blockIdx.x / cl, rank = (int)cluster_rank(), nrows = 1 << logrows, bz = geo.bz, bx = geo.bx;
    SmallField<C> f;
    f.logrows = logrows;
    f.cols = bx / cl;
    f.ix0 = rank * f.cols;
    f.ls = bx + 1;
    f.rows = reinterpret_cast<C*>(sm_raw);
    cluster_arrive();
    C* spec = f.rows + nrows * f.ls;
    f.bufs = spec + nrows * f.ls;
    for (int r = threadIdx.x >> 5; r < nrows; r += kSmallThreads / 32) {
        const int kr = rank * nrows + r, kz = kr < bz ? 2 * kr : 2 * (kr - bz) + 1;
        const C* sp = spt + (long long)min(kz, 2 * bz - kz) * (bx + 1);
        for (int e = threadIdx.x & 31; e <= bx; e += 32) cp_async<sizeof(C)>(spec + r * (bx + 1) + e, sp + e);
    }
    const int2 org = box_origin(geo, b);
    const double* chb = geo.chi + (long long)org.y * geo.chi_ld + org.x;
    const long long off = (long long)b * bz * bx;
    const C* ub = u + off;
    const C* u0b = u0 ? u0 + off : nullptr;
    const C* ltz = tab + line_table(bz);
#define LSW_SMALL_SWITCH(n, ...)                                  \
    switch (n) {                                                  \
        case 4: { constexpr int L_ = 2; __VA_ARGS__; break; }     \
        case 8: { constexpr int L_ = 3; __VA_ARGS__; break; }     \
        case 16: { constexpr int L_ = 4; __VA_ARGS__; break; }    \
        case 32: { constexpr int L_ = 5; __VA_ARGS__; break; }    \
        case 64: { constexpr int L_ = 6; __VA_ARGS__; break; }    \
        default: { constexpr int L_ = 7; __VA_ARGS__; break; }    \
    }
    LSW_SMALL_SWITCH(bz, small_a<R, L_>(f, ub, chb, geo.chi_ld, mode == LSW_OP_ADJOINT, ltz))
    cp_async_wait_all();
    cluster_arrive();
    cluster_wait();
    LSW_SMALL_SWITCH(bx, small_b<L_>(f, spec, tab + line_table(bx)))
    cluster_arrive();
    cluster_wait();
    LSW_SMALL_SWITCH(bz, small_c<R, L_>(f, ub, u0b, y + off, chb, geo.chi_ld, mode, ltz))
#undef LSW_SMALL_SWITCH
    cluster_wait();                          // no block leaves while its rows may be read
}

// ------------------------------------------------ generic strided 1D FFTs
// nlines lines of length P: element i of line l at data[l * lstep + i * estep].
template <int NT>
__global__ void __launch_bounds__(NT)
k_fft_strided64(double2* data, int P, int logP, int nlines, int lpc, long long lstep, long long estep,
                const double2* __restrict__ tw, int twstep, int inv) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double2* sm = reinterpret_cast<double2*>(sm_raw);
    const int l0 = blockIdx.x * lpc;
    const int nl = min(lpc, nlines - l0);
    for (int e = threadIdx.x; e < nl * P; e += NT) {
        const int l = e >> logP, i = e & (P - 1);
        sm[l * P + i] = data[(l0 + l) * lstep + i * estep];
    }
    __syncthreads();
    smem_fft<double2, NT, 4>(sm, P, nl, P, logP, tw, twstep, inv != 0);
    for (int e = threadIdx.x; e < nl * P; e += NT) {
        const int l = e >> logP, i = e & (P - 1);
        data[(l0 + l) * lstep + i * estep] = sm[l * P + i];
    }
}

// ------------------------------------------------------------ Green table
// Cell-integrated Green's function (disk of equal area, radius a):
//   r > 0:  (i pi a / (2k)) J1(ka) H0(kr)
//   r = 0:  (i pi a / (2k)) H1(ka) - 1/k^2
__global__ void k_green_table(double2* table, int nz, int nx, double h, double k) {
    const int n = (nz + 1) * (nx + 1);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int dx = e / (nz + 1), dz = e - dx * (nz + 1);
        const double a = h * rsqrt(M_PI);
        const double ka = k * a;
        const double pre = M_PI * a / (2.0 * k);        // prefactor is i * pre
        double2 g;
        if (dx == 0 && dz == 0) {
            // i pre (J1 + i Y1) - 1/k^2
            g = make_double2(-pre * y1(ka) - 1.0 / (k * k), pre * j1(ka));
        } else {
            const double kr = k * h * sqrt((double)dz * dz + (double)dx * dx);
            const double s = pre * j1(ka);
            // i s (J0 + i Y0)
            g = make_double2(-s * y0(kr), s * j0(kr));
        }
        table[e] = g;
    }
}

// even extension of the table to (2bz x 2bx), column-major (2bx columns)
__global__ void k_extend(const double2* __restrict__ table, int nz, int bz, int bx, double2* ext) {
    const int pz = 2 * bz, px = 2 * bx;
    const long long n = (long long)pz * px;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(e / pz), iz = (int)(e - (long long)ix * pz);
        const int dx = min(ix, px - ix), dz = min(iz, pz - iz);
        ext[e] = table[dx * (nz + 1) + dz];
    }
}

__global__ void k_quarter(const double2* __restrict__ F, int bz, int bx, double2* q64, float2* q32, double2* t64,
                          float2* t32) {
    const int pz = 2 * bz;
    const int n = (bz + 1) * (bx + 1);
    const double sc = 1.0 / (4.0 * bz * bx);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int qx = e / (bz + 1), qz = e - qx * (bz + 1);
        const double2 v = F[(long long)qx * pz + qz];
        const double2 w = make_double2(v.x * sc, v.y * sc);
        const float2 f = make_float2((float)w.x, (float)w.y);
        q64[e] = w;
        q32[e] = f;
        // kz-major rows: the even qx, then the odd ones
        const int p = qz * (bx + 1) + ((qx & 1) ? bx / 2 + 1 : 0) + (qx >> 1);
        t64[p] = w;
        t32[p] = f;
    }
}

// exp(-2 pi i m / P), m < P, then the line twiddles and half-sample shifts of
// every line length (line_table), in one launch
__global__ void k_twiddles(double2* tw64, float2* tw32, int P) {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < P + kLineTables; m += gridDim.x * blockDim.x) {
        double turn;                    // in half turns
        if (m < P) {
            turn = -2.0 * m / P;
        } else {
            const int e = m - P;
            int N = 4;
            while (line_table(2 * N) <= e) N *= 2;
            const int E = N >= 512 ? 32 : N >= 128 ? 16 : N >= 32 ? 8 : 4, T = N / E;      // LineCfg
            const int i = e - line_table(N), which = i / N, c = (i - which * N) / T, t = i % T;
            turn = -(double)(which == 0 ? 2 * c * t : which == 1 ? (2 * c + 1) * t : c * (2 * t + 1)) / N;
        }
        double s, c;
        sincospi(turn, &s, &c);
        tw64[m] = make_double2(c, s);
        tw32[m] = make_float2((float)c, (float)s);
    }
}

__global__ void k_contrast(const double* __restrict__ vel, double* chi, long long n, double w2, double ic02) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const double c = vel[e];
        chi[e] = w2 * (1.0 / (c * c) - ic02);
    }
}

template <typename C>
__global__ void k_point_sources(const double2* __restrict__ table, int nz, int nx, const int2* __restrict__ pos,
                                int nsrc, double ih2, C* u0) {
    const long long n = (long long)nz * nx;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * nsrc; e += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(e / n);
        const long long i = e - s * n;
        const int ix = (int)(i / nz), iz = (int)(i - (long long)ix * nz);
        const int dz = abs(iz - pos[s].x), dx = abs(ix - pos[s].y);
        const double2 g = table[dx * (nz + 1) + dz];
        C v;
        v.x = g.x * ih2;
        v.y = g.y * ih2;
        u0[e] = v;
    }
}

// Algorithmic bytes of one batched apply: per field read u (and u0) and
// write y; chi (FP64) and the quarter spectrum once per batch.
double op_bytes(size_t elem, int bz, int bx, int nb, bool has_u0, int) {
    const double cells = (double)bz * bx;
    return (double)elem * cells * (2.0 + (has_u0 ? 1.0 : 0.0)) * nb + 8.0 * cells + (double)elem * (bz + 1) * (bx + 1);
}
// 5 N log2 N per complex FFT: nx columns of 2nz, 2nz rows forward and back
// of 2nx, nx columns back; 6 per spectrum product.
double op_flops(int bz, int bx, int nb) {
    const double pz = 2.0 * bz, px = 2.0 * bx;
    const double fz = 5.0 * pz * std::log2(pz), fx = 5.0 * px * std::log2(px);
    return nb * (2.0 * bx * fz + 2.0 * pz * fx + 6.0 * pz * px);
}

int grid_for(long long n, int bs = 256) {
    long long g = (n + bs - 1) / bs;
    return (int)std::max<long long>(1, std::min<long long>(g, 152LL * 16));
}

}  // namespace

// Launch the register-FFT passes for a runtime log2 size (2..10).
template <typename K>
lsw_status set_smem(K k, std::atomic<bool>& done) {
    if (!done) {
        LSW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
        done = true;
    }
    return LSW_OK;
}

#define LSW_LOG_SWITCH(lg, ...)                  \
    switch (lg) {                                \
        case 2: { constexpr int L_ = 2; __VA_ARGS__; break; }   \
        case 3: { constexpr int L_ = 3; __VA_ARGS__; break; }   \
        case 4: { constexpr int L_ = 4; __VA_ARGS__; break; }   \
        case 5: { constexpr int L_ = 5; __VA_ARGS__; break; }   \
        case 6: { constexpr int L_ = 6; __VA_ARGS__; break; }   \
        case 7: { constexpr int L_ = 7; __VA_ARGS__; break; }   \
        case 8: { constexpr int L_ = 8; __VA_ARGS__; break; }   \
        case 9: { constexpr int L_ = 9; __VA_ARGS__; break; }   \
        case 10: { constexpr int L_ = 10; __VA_ARGS__; break; } \
        default: return LSW_ERR_UNSUPPORTED_SIZE;        \
    }

// pdl: let the kernel start while its predecessor runs (pdl_wait)
template <typename K, typename... A>
lsw_status launch_pass(K k, bool pdl, dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = pdl ? 1 : 0;
    LSW_CUDA(cudaLaunchKernelEx(&cfg, k, args...));
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

// log2 box sides lz, lx: 2 .. 10
template <typename R>
lsw_status launch_fa(int lz, bool pdl, int nbatch, cudaStream_t st, const typename Cx<R>::T* u, const DevGeom& dg,
                     const typename Cx<R>::T* tab, int adj, typename Cx<R>::T* work) {
    typedef typename Cx<R>::T C;
    static std::atomic<bool> done[11];
    LSW_LOG_SWITCH(lz, {
        constexpr int NT = fft_threads<R>(), lines = NT / LineCfg<L_>::T, cols = lines / 2;
        LSW_TRY(set_smem(k_fa<R, L_>, done[L_]));
        // fields per CTA: up to 4 while 2048 threads per SM remain
        const int gx = (dg.bx + cols - 1) / cols;
        const int per = std::max(1, std::min(4, (int)((long long)gx * nbatch * NT / (152 * 2048))));
        LSW_TRY(launch_pass(k_fa<R, L_>, pdl, dim3(gx, (nbatch + per - 1) / per), NT,
                            sizeof(C) * lines * line_stride<C, L_, kblk<C>()>() + sizeof(R) * cols * LineCfg<L_>::N, st,
                            u, dg, tab + line_table(1 << L_), adj, work, nbatch, per));
    })
    return LSW_OK;
}

// 512 threads: twice the rows (FP64: four times), where they fit in shared memory and registers
template <typename R, int LOGN> constexpr bool fb_wide() { return sizeof(R) == 4 || LineCfg<LOGN>::E < 32; }

template <typename R, int NTB>
lsw_status launch_fb(int lx, bool pdl, int bz, int nbatch, cudaStream_t st, typename Cx<R>::T* work,
                     const typename Cx<R>::T* spt, const typename Cx<R>::T* tab) {
    typedef typename Cx<R>::T C;
    static std::atomic<bool> done[11];
    LSW_LOG_SWITCH(lx, {
        constexpr int NT = fb_wide<R, L_>() ? NTB : fft_threads<R>(), rows = NT / (2 * LineCfg<L_>::T);
        LSW_TRY(set_smem(k_fb<R, L_, NT>, done[L_]));
        LSW_TRY(launch_pass(k_fb<R, L_, NT>, pdl, dim3((2 * bz + rows - 1) / rows, nbatch), NT,
                            sizeof(C) * rows * (2 * line_stride<C, L_, rows>() + LineCfg<L_>::N + 1), st, work, bz, spt,
                            tab + line_table(1 << L_)));
    })
    return LSW_OK;
}

template <typename R>
lsw_status launch_fc(int lz, bool pdl, int nbatch, cudaStream_t st, const typename Cx<R>::T* work, const DevGeom& dg,
                     const typename Cx<R>::T* tab, int mode, const typename Cx<R>::T* u, const typename Cx<R>::T* u0,
                     typename Cx<R>::T* y) {
    typedef typename Cx<R>::T C;
    static std::atomic<bool> done[11];
    LSW_LOG_SWITCH(lz, {
        constexpr int NT = fft_threads<R>(), lines = NT / LineCfg<L_>::T, cols = lines / 2;
        LSW_TRY(set_smem(k_fc<R, L_>, done[L_]));
        LSW_TRY(launch_pass(k_fc<R, L_>, pdl, dim3((dg.bx + cols - 1) / cols, nbatch), NT,
                            sizeof(C) * lines * line_stride<C, L_, kblk<C>()>(), st, work, dg, tab + line_table(1 << L_),
                            mode, u, u0, y));
    })
    return LSW_OK;
}

// Whether the passes start while their predecessors run.  It hides 2 to 3 us per
// pass, but a pass that starts early lands on the SMs that its predecessor has
// left free, and stays there: with CTAs for part of the SMs only, two and more of a
// pass share an SM while others idle.  FP64, whose pipe is the bound, then loses
// far more than it gains (8 fields of 128 x 128: 201 us against 100; one of 512 x 512 290
// against 231; 16 x 1024, 8 fields 202 against 111), so it starts early only where
// either kind of line has CTAs for four fifths of the SMs' slots (from there on
// 7 to 10 us are gained: 128 x 128, 32 fields 307 against 315; 512 x 512, 2 fields 425 against
// 433).  FP32 always does.
template <typename R>
bool start_early(int bz, int bx, int nbatch) {
    if (sizeof(R) == 4) return true;
    auto filled = [&](int side, long long lines) {      // lines of `side` cells, both parities
        const int e = side >= 512 ? 32 : side >= 128 ? 16 : side >= 32 ? 8 : 4;                         // LineCfg
        return lines * 2 * (side / e) / fft_threads<R>() * 5 >= 4LL * 152 * (e == 32 ? 2 : 4);          // fft_ctas
    };
    return filled(bz, (long long)bx * nbatch) && filled(bx, 2LL * bz * nbatch);
}

// The one-launch kernel's cluster: blocks per field, as many (at most 8) as
// give every block a full set of row lines in pass B, and its shared memory.
template <typename R>
size_t small_cfg(int bz, int bx, int& cl) {
    typedef typename Cx<R>::T C;
    auto line_t = [](int n) { return n >= 512 ? n / 32 : n >= 128 ? n / 16 : n >= 32 ? n / 8 : n / 4; };   // LineCfg::T
    cl = 1;
    while (cl < 8 && 4 * bz * line_t(bx) > kSmallThreads * cl && bx / cl > 1) cl *= 2;
    size_t bufs = 0;
    auto lines = [&](auto lg) {
        constexpr int L = decltype(lg)::value;
        if (bz == 1 << L || bx == 1 << L)
            bufs = std::max(bufs, (size_t)(kSmallThreads / LineCfg<L>::T) * line_stride<C, L, kblk<C>()>());
    };
    lines(std::integral_constant<int, 2>());
    lines(std::integral_constant<int, 3>());
    lines(std::integral_constant<int, 4>());
    lines(std::integral_constant<int, 5>());
    lines(std::integral_constant<int, 6>());
    lines(std::integral_constant<int, 7>());
    return sizeof(C) * (2 * (size_t)(2 * bz / cl) * (bx + 1) + bufs);
}

// ---------------------------------------------------------- pass tuning
// Variant of the operator passes per (2bz, 2bx, precision): 0 register FFT
// with row CTAs of fft_threads in pass B, 1 the same with 512-thread row CTAs,
// 2 the shared-memory Stockham passes.  Chosen by lsw_autotune.
namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int>, int> g_tune;
thread_local int g_force_variant = -1;
}  // namespace

int op_variant(int pz, int px, int rsize) {
    if (g_force_variant >= 0) return g_force_variant;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune.find(std::make_tuple(pz, px, rsize));
    return it == g_tune.end() ? 0 : it->second;
}

void op_force_variant(int v) { g_force_variant = v; }

void op_set_variant(int pz, int px, int rsize, int v) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[std::make_tuple(pz, px, rsize)] = v;
}

// One launch (k_small) for this product?  Where a call's time is the host's,
// which takes longer to launch three kernels and fetch a work array (19.5 us a
// call of one 64 x 64 field) than to launch one (13.9).  The GPU alone is a little
// slower with it.  One launch against three, c64: 64 x 64 cells, 1
// field 8.2 / 7.6 us, 8 fields 8.3 / 7.7, 16 fields 11.6 / 8.0; 64 x 128, 1
// field 10.2 / 9.5; 128 x 128, 1 field 17.4 / 11.9.  c128: 32 x 32 46.6 / 47.2,
// 64 x 64, 8 fields 53.5 / 54.2, 16 fields 103 / 54.5.  So fields of up to 8192
// cells, 32768 cells in all.  Solvers keep a work array and replay their steps as
// graphs; there the two are even: FGMRES in c64, 4 sources, 32 x 32 1.96 / 1.99 ms,
// 64 x 64 5.34 / 5.29, 64 x 128 7.20 / 7.10; mixed with H 1.74 / 1.78, 2.85 / 2.87,
// 2.74 / 2.69.  A field has a block of its own however small it is, so at most 512
// fields: 2048 fields of 4 x 4 cells take 37 us in one launch, 23 in three.  u and y
// must not overlap: one field's blocks may write y before another's read u.
bool op_small(const lsw_green* g, const Spectrum& sp, const OpGeom& geo, int rsize, int nbatch, const void* u,
              const void* y) {
    const int bz = geo.bz, bx = geo.bx;
    if (!is_pow2(bz) || !is_pow2(bx) || bz < 4 || bx < 4 || bz > 128 || bx > 128 || bz * bx > 8192) return false;
    const long long cells = (long long)bz * bx * nbatch;
    if (cells > (1 << 15) || nbatch > 512 || !sp.t32 || !sp.t64 || op_variant(2 * bz, 2 * bx, rsize) == 2) return false;
    const char *pu = static_cast<const char*>(u), *py = static_cast<const char*>(y);
    return py + 2 * rsize * cells <= pu || pu + 2 * rsize * cells <= py;
}

// ------------------------------------------------------------ op_apply
template <typename R>
lsw_status op_apply(const lsw_green* g, const Spectrum& sp, const OpGeom& geo, int mode,
                    const typename Cx<R>::T* u, const typename Cx<R>::T* u0, typename Cx<R>::T* y,
                    int nbatch, typename Cx<R>::T* work, cudaStream_t st) {
    typedef typename Cx<R>::T C;
    constexpr int NT = FftCfg<R>::NT, MB4 = FftCfg<R>::MB4, CAP = fft_capacity<R>();
    if (nbatch <= 0) return LSW_OK;
    const int bz = geo.bz, bx = geo.bx;
    const int pz = 2 * bz, px = 2 * bx;
    if (!is_pow2(bz) || !is_pow2(bx) || pz > CAP || px > CAP) return LSW_ERR_UNSUPPORTED_SIZE;
    if (sp.bz != bz || sp.bx != bx) return LSW_ERR_INVALID_ARG;
    const C* tw = reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)g->tw64 : (const void*)g->tw32);
    const C* specq = reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)sp.q64 : (const void*)sp.q32);

    DevGeom dg{bz, bx, ilog2(bz), geo.chi, geo.chi_ld, geo.origin, geo.vpb > 0 ? geo.vpb : 1};
    const int logpz = ilog2(pz), logpx = ilog2(px);
    const int variant = op_variant(pz, px, (int)sizeof(R));
    // no work array: the caller has asked op_small (the variant may change meanwhile)
    if (!work || op_small(g, sp, geo, (int)sizeof(R), nbatch, u, y)) {
        int cl = 1;
        const size_t smem = small_cfg<R>(bz, bx, cl);
        static std::atomic<bool> done{false};
        LSW_TRY(set_smem(k_small<R>, done));
        KTimer kt(sizeof(R) == 8 ? "operator_c128" : "operator_c64", st,
                  op_bytes(sizeof(C), bz, bx, nbatch, u0 != nullptr, mode), op_flops(bz, bx, nbatch));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cl * nbatch);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = cl;
        at.val.clusterDim.y = 1;
        at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        LSW_CUDA(cudaLaunchKernelEx(&cfg, k_small<R>, u, dg, ilog2(2 * bz / cl),
                                    reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)sp.t64 : (const void*)sp.t32),
                                    reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)g->lt64 : (const void*)g->lt32),
                                    mode, u0, y, cl));
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    }
    if (variant != 2 && bz >= 4 && bx >= 4 && bz <= 1024 && bx <= 1024 && sp.t32 && sp.t64) {
        const C* spt = reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)sp.t64 : (const void*)sp.t32);
        const C* tab = reinterpret_cast<const C*>(sizeof(R) == 8 ? (const void*)g->lt64 : (const void*)g->lt32);
        KTimer kt(sizeof(R) == 8 ? "operator_c128" : "operator_c64", st, op_bytes(sizeof(C), bz, bx, nbatch, u0 != nullptr, mode),
                  op_flops(bz, bx, nbatch));
        const int lz = logpz - 1, lx = logpx - 1;
        const bool pdl = start_early<R>(bz, bx, nbatch);
        LSW_TRY(launch_fa<R>(lz, pdl, nbatch, st, u, dg, tab, mode == LSW_OP_ADJOINT, work));
        if (variant == 1) LSW_TRY((launch_fb<R, 512>(lx, pdl, bz, nbatch, st, work, spt, tab)));
        else LSW_TRY((launch_fb<R, fft_threads<R>()>(lx, pdl, bz, nbatch, st, work, spt, tab)));
        LSW_TRY(launch_fc<R>(lz, pdl, nbatch, st, work, dg, tab, mode, u, u0, y));
        return LSW_OK;
    }
    // columns per CTA for passes A and C, rows per CTA for pass B
    int cx = std::min(bx, std::max(1, CAP / pz));
    cx = std::min(cx, 16);
    int rz = std::min(pz, std::max(1, CAP / px));
    rz = std::min(rz, 16);
    const int lsa = pz + 1, lsb = px + 1;
    const size_t smA = (size_t)cx * lsa * sizeof(C), smB = (size_t)rz * lsb * sizeof(C);
    auto ka = k_pass_a<R, NT, MB4>;
    auto kb = k_pass_b<R, NT, MB4>;
    auto kc = k_pass_c<R, NT, MB4>;
    static std::atomic<bool> attr_done[2];
    if (!attr_done[sizeof(R) == 8]) {
        const int maxsm = 200 * 1024;
        LSW_CUDA(cudaFuncSetAttribute(ka, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        LSW_CUDA(cudaFuncSetAttribute(kb, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        LSW_CUDA(cudaFuncSetAttribute(kc, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        attr_done[sizeof(R) == 8] = true;
    }
    const int twz = g->twP / pz, twx = g->twP / px;
    dim3 gA(bx / cx, nbatch), gB(pz / rz, nbatch);
    ka<<<gA, NT, smA, st>>>(u, dg, pz, logpz, cx, ilog2(cx), lsa, tw, twz, mode == LSW_OP_ADJOINT, work);
    LSW_LAUNCH_CHECK();
    kb<<<gB, NT, smB, st>>>(work, bx, pz, px, logpx, rz, ilog2(rz), lsb, specq, bz + 1, tw, twx);
    LSW_LAUNCH_CHECK();
    kc<<<gA, NT, smA, st>>>(work, dg, pz, logpz, cx, ilog2(cx), lsa, tw, twz, mode, u, u0, y);
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

template lsw_status op_apply<float>(const lsw_green*, const Spectrum&, const OpGeom&, int, const float2*,
                                    const float2*, float2*, int, float2*, cudaStream_t);
template lsw_status op_apply<double>(const lsw_green*, const Spectrum&, const OpGeom&, int, const double2*,
                                     const double2*, double2*, int, double2*, cudaStream_t);

// ------------------------------------------------------- spectra and table
lsw_status build_spectrum(const lsw_green* g, int bz, int bx, Spectrum* out, cudaStream_t st) {
    if (bz > g->nz || bx > g->nx || !is_pow2(bz) || !is_pow2(bx)) return LSW_ERR_INVALID_ARG;
    const int pz = 2 * bz, px = 2 * bx;
    constexpr int NT = 256;
    const int cap = 4 * NT * 4;
    if (pz > cap || px > cap) return LSW_ERR_UNSUPPORTED_SIZE;
    DevBuf ext;
    LSW_TRY(ext.alloc(sizeof(double2) * (size_t)pz * px, st));
    double2* E = ext.as<double2>();
    k_extend<<<grid_for((long long)pz * px), 256, 0, st>>>(g->table, g->nz, bz, bx, E);
    LSW_LAUNCH_CHECK();
    auto kf = k_fft_strided64<NT>;
    LSW_CUDA(cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    // along z: px lines of length pz, contiguous
    {
        const int lpc = std::max(1, std::min(px, cap / pz));
        kf<<<(px + lpc - 1) / lpc, NT, sizeof(double2) * lpc * pz, st>>>(E, pz, ilog2(pz), px, lpc, pz, 1,
                                                                         g->tw64, g->twP / pz, 0);
        LSW_LAUNCH_CHECK();
    }
    // along x: pz lines of length px, stride pz
    {
        const int lpc = std::max(1, std::min(pz, cap / px));
        kf<<<(pz + lpc - 1) / lpc, NT, sizeof(double2) * lpc * px, st>>>(E, px, ilog2(px), pz, lpc, 1, pz,
                                                                         g->tw64, g->twP / px, 0);
        LSW_LAUNCH_CHECK();
    }
    Spectrum s;
    s.bz = bz;
    s.bx = bx;
    const size_t nq = (size_t)(bz + 1) * (bx + 1);
    if (cudaMalloc(&s.q64, 2 * nq * sizeof(double2)) != cudaSuccess ||
        cudaMalloc(&s.q32, 2 * nq * sizeof(float2)) != cudaSuccess) {
        free_spectrum(&s);
        return LSW_ERR_OOM;
    }
    s.t64 = s.q64 + nq;
    s.t32 = s.q32 + nq;
    k_quarter<<<grid_for((long long)nq), 256, 0, st>>>(E, bz, bx, s.q64, s.q32, s.t64, s.t32);
    LSW_LAUNCH_CHECK();
    *out = s;
    return LSW_OK;
}

void free_spectrum(Spectrum* s) {
    if (s->q64) device_free(s->q64);
    if (s->q32) device_free(s->q32);
    s->q64 = nullptr;
    s->q32 = nullptr;
    s->t64 = nullptr;
    s->t32 = nullptr;
}

lsw_status green_init(lsw_green* g, cudaStream_t st) {
    const size_t nt = (size_t)(g->nz + 1) * (g->nx + 1);
    LSW_CUDA(cudaMalloc(&g->table, nt * sizeof(double2)));
    k_green_table<<<grid_for((long long)nt), 256, 0, st>>>(g->table, g->nz, g->nx, g->h, g->k);
    LSW_LAUNCH_CHECK();
    g->twP = 2 * std::max(g->nz, g->nx);
    LSW_CUDA(cudaMalloc(&g->tw64, (g->twP + kLineTables) * sizeof(double2)));
    LSW_CUDA(cudaMalloc(&g->tw32, (g->twP + kLineTables) * sizeof(float2)));
    g->lt64 = g->tw64 + g->twP;
    g->lt32 = g->tw32 + g->twP;
    k_twiddles<<<grid_for(g->twP + kLineTables), 256, 0, st>>>(g->tw64, g->tw32, g->twP);
    LSW_LAUNCH_CHECK();
    LSW_TRY(build_spectrum(g, g->nz, g->nx, &g->full, st));
    LSW_CUDA(cudaStreamSynchronize(st));
    return LSW_OK;
}

lsw_status contrast(const lsw_green* g, const double* vel, double* chi, cudaStream_t st) {
    const long long n = (long long)g->nz * g->nx;
    const double w = 2.0 * M_PI * g->freq;
    k_contrast<<<grid_for(n), 256, 0, st>>>(vel, chi, n, w * w, 1.0 / (g->c0 * g->c0));
    LSW_LAUNCH_CHECK();
    return LSW_OK;
}

lsw_status point_sources(const lsw_green* g, const int32_t* pos_host, int nsrc, int prec, void* u0,
                         cudaStream_t st) {
    for (int s = 0; s < nsrc; ++s) {
        if (pos_host[2 * s] < 0 || pos_host[2 * s] >= g->nz || pos_host[2 * s + 1] < 0 ||
            pos_host[2 * s + 1] >= g->nx)
            return LSW_ERR_INVALID_ARG;
    }
    DevBuf pos;
    LSW_TRY(pos.alloc(sizeof(int2) * nsrc, st));
    LSW_CUDA(cudaMemcpyAsync(pos.p, pos_host, sizeof(int2) * nsrc, cudaMemcpyHostToDevice, st));
    const long long n = (long long)g->nz * g->nx * nsrc;
    const double ih2 = 1.0 / (g->h * g->h);
    if (prec == LSW_C128)
        k_point_sources<double2><<<grid_for(n), 256, 0, st>>>(g->table, g->nz, g->nx, pos.as<int2>(), nsrc, ih2,
                                                              (double2*)u0);
    else
        k_point_sources<float2><<<grid_for(n), 256, 0, st>>>(g->table, g->nz, g->nx, pos.as<int2>(), nsrc, ih2,
                                                             (float2*)u0);
    LSW_LAUNCH_CHECK();
    // the host array is read by an async copy: wait before returning
    LSW_CUDA(cudaStreamSynchronize(st));
    return LSW_OK;
}

}  // namespace lsw
