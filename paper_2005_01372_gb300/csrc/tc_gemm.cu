// Batched complex FP32 GEMM on the 5th-generation tensor cores (tcgen05),
// for the products of the HODLR dense leaves with a block of vectors:
//     C_b = alpha A_b B_b,   A_b: M x K, B_b: K x N (N <= 32), column-major.
//
// Complex as real: with A'' (M x 2K) = [Re a_ik, Im a_ik] interleaved along
// K and B'' (2K x 64) whose columns 0..31 are [Re b_kj; -Im b_kj] and
// 32..63 are [Im b_kj; Re b_kj], the real product A'' B'' holds Re C in its
// first 32 columns and Im C in the last 32.
//
// FP32 accuracy from TF32 inputs ("3xTF32"): x = hi + lo with hi = x rounded
// to TF32 and lo = x - hi (exact in FP32); A B ~ Ahi Bhi + Ahi Blo + Alo Bhi,
// the dropped Alo Blo being ~2^-22 relative.  The accumulator stays in TMEM
// (FP32) for the whole K loop.
//
// One CTA of 128 threads owns 128 rows of one matrix.  Per stage of 8 complex
// K (16 real): every thread loads its row of A and a slice of B into registers
// two stages ahead and splits them.  A's hi/lo go straight into tensor memory
// (a thread's row is its TMEM lane, a K index a column), B's into shared memory in
// the canonical K-major layout without swizzle (8-row x 16-byte core matrices,
// 128 B apart along K, 512 B apart along rows); one thread issues 3 x 2
// tcgen05.mma of 128 x 64 x 8 and commits them to the stage's mbarrier, which the
// producer waits on (bounded) before reusing that buffer.  128 TMEM columns and
// 16 KB of shared memory: four CTAs per SM.  With few matrices K is split over
// blockIdx.z into parts sP apart, added afterwards.
//
// Bound by reading A.  64 leaves of 1024 x 1024 (0.54 GB) times 32 vectors:
// 135 us (4 TB/s); with A's hi/lo in shared memory 197 us (two CTAs of 16-deep
// stages per SM, whose writes and the MMAs' reads took most of that memory's
// bandwidth, and 512 CTAs in 1.7 waves).
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "lsw_internal.cuh"
#include "tc_ptx.cuh"

namespace lsw {
namespace {

constexpr int TC_M = 128;                       // rows per CTA (TMEM lanes)
constexpr int TC_KC = 8;                        // complex K per stage
constexpr int TC_NN = 64;                       // real output columns
constexpr int B_TILE = TC_NN * 2 * TC_KC * 4;   // 4 KB: 64 rows x 16 TF32
constexpr int B_SBO = 8 * 2 * TC_KC * 4;        // bytes between 8-row groups
// TMEM columns: the accumulator, then per stage buffer A hi and A lo
constexpr uint32_t TC_TMEM_COLS = 128;
constexpr uint32_t TC_ACOL = 64, TC_ASTAGE = 4 * TC_KC;
// D F32 (bits 4-5 = 1), A and B TF32 (bits 7-9, 10-12 = 2), both K-major,
// N / 8 at bits 17-22, M / 16 at bits 24-28.
constexpr uint32_t TC_IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(TC_NN >> 3) << 17) |
                              ((uint32_t)(TC_M >> 4) << 24);
__device__ int g_tc_timeouts = 0;

using namespace tcx;

__global__ void __launch_bounds__(128, 4)
k_cgemm_tc(const float2* __restrict__ A, int lda, long long sA, const float2* __restrict__ B, int ldb, long long sB,
           float2* __restrict__ Cm, int ldc, long long sC, long long sP, int N, int Kper, float2 alpha) {
    __shared__ __align__(1024) unsigned char sm[4 * B_TILE];
    __shared__ uint64_t mbar[2];
    __shared__ uint32_t tslot;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.y, i0 = blockIdx.x * TC_M;
    const float2* Ab = A + b * sA + i0 + (long long)blockIdx.z * Kper * lda;     // part z of K
    const float2* Bb = B + b * sB + (long long)blockIdx.z * Kper;
    float2* Cb = Cm + blockIdx.z * sP + b * sC + i0;
    const uint32_t mb0 = smem_u32(&mbar[0]), mb1 = smem_u32(&mbar[1]);
    if (tid == 0) {
        mbar_init(mb0, 1);
        mbar_init(mb1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        *abort_flag = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);      // this warp's lanes

    const int S = Kper / TC_KC;
    const int jb = lane, gb = warp;              // B slice: column jb, complex k 2 gb, 2 gb + 1 (kgroup gb)
    // two register sets, each loaded two stages ahead of its use
    float2 ra0[TC_KC], rb0[2], ra1[TC_KC], rb1[2];
    auto gload = [&](int s, float2 (&ra)[TC_KC], float2 (&rb)[2]) {
        const int k0 = s * TC_KC;
#pragma unroll
        for (int kk = 0; kk < TC_KC; ++kk) ra[kk] = Ab[(long long)(k0 + kk) * lda + tid];
#pragma unroll
        for (int q = 0; q < 2; ++q)
            rb[q] = jb < N ? Bb[(long long)jb * ldb + k0 + 2 * gb + q] : make_float2(0.f, 0.f);
    };
    int committed = 0;
    // one stage: wait for the buffer, split and store, refill the register
    // set for stage s + 2, issue the MMAs; false when a wait gave up
    auto stage = [&](int s, float2 (&ra)[TC_KC], float2 (&rb)[2]) -> bool {
        const int buf = s & 1;
        unsigned char* Bhi = sm + buf * 2 * B_TILE;
        unsigned char* Blo = Bhi + B_TILE;
        const uint32_t acol = TC_ACOL + buf * TC_ASTAGE;
        if (tid == 0 && s >= 2 && !mbar_wait(buf ? mb1 : mb0, ((s - 2) >> 1) & 1)) *abort_flag = 1;
        __syncthreads();
        if (*abort_flag) return false;
        asm volatile("tcgen05.fence::after_thread_sync;");
        // A'' row tid: Re a(0), Im a(0), Re a(1), ...
        {
            float h[2 * TC_KC], l[2 * TC_KC];
#pragma unroll
            for (int kk = 0; kk < TC_KC; ++kk) {
                split_tf32(ra[kk].x, h[2 * kk], l[2 * kk]);
                split_tf32(ra[kk].y, h[2 * kk + 1], l[2 * kk + 1]);
            }
            tmem_st16(trow + acol, h);
            tmem_st16(trow + acol + 2 * TC_KC, l);
        }
        // B'' rows jb (real part) and jb + 32 (imaginary part), kgroup gb
        {
            const float2 x0 = rb[0], x1 = rb[1];
            float r0h, r0l, i0h, i0l, r1h, r1l, i1h, i1l;
            split_tf32(x0.x, r0h, r0l);
            split_tf32(x0.y, i0h, i0l);
            split_tf32(x1.x, r1h, r1l);
            split_tf32(x1.y, i1h, i1l);
            const int o = (jb >> 3) * B_SBO + gb * 128 + (jb & 7) * 16, oi = o + 4 * B_SBO;
            *reinterpret_cast<float4*>(Bhi + o) = make_float4(r0h, -i0h, r1h, -i1h);
            *reinterpret_cast<float4*>(Blo + o) = make_float4(r0l, -i0l, r1l, -i1l);
            *reinterpret_cast<float4*>(Bhi + oi) = make_float4(i0h, r0h, i1h, r1h);
            *reinterpret_cast<float4*>(Blo + oi) = make_float4(i0l, r0l, i1l, r1l);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        if (s + 2 < S) gload(s + 2, ra, rb);    // two stages of loads stay in flight
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t ah = tmem + acol, al = ah + 2 * TC_KC, bh = smem_u32(Bhi), bl = smem_u32(Blo);
#pragma unroll
            for (int ks = 0; ks < TC_KC / 4; ++ks) {
                const uint32_t o = ks * 256;    // 8 real K = two core matrices, eight columns of A
                mma_tf32_ta(tmem, ah + 8 * ks, sdesc_sbo(bh + o, B_SBO), TC_IDESC, (s > 0 || ks > 0) ? 1u : 0u);
                mma_tf32_ta(tmem, ah + 8 * ks, sdesc_sbo(bl + o, B_SBO), TC_IDESC, 1u);
                mma_tf32_ta(tmem, al + 8 * ks, sdesc_sbo(bh + o, B_SBO), TC_IDESC, 1u);
            }
            mma_commit(buf ? mb1 : mb0);
        }
        committed = s + 1;
        return true;
    };
    gload(0, ra0, rb0);
    if (S > 1) gload(1, ra1, rb1);
    for (int s = 0; s < S; s += 2) {
        if (!stage(s, ra0, rb0)) break;
        if (s + 1 < S && !stage(s + 1, ra1, rb1)) break;
    }
    // the last commit covers every MMA issued before it
    if (tid == 0 && committed > 0) {
        const int s = committed - 1;
        if (!mbar_wait((s & 1) ? mb1 : mb0, (s >> 1) & 1)) *abort_flag = 1;
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const bool bad = *abort_flag != 0 || committed != S;
    // TMEM -> registers: warp w reads lanes 32 w .. 32 w + 31 (its rows)
    float d[TC_NN];
#pragma unroll
    for (int c = 0; c < TC_NN; c += 16) tmem_ld16(trow + c, d + c);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int row = warp * 32 + lane;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        if (j >= N) break;
        float2 o;
        if (bad) {
            o = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
        } else {
            const float re = d[j], im = d[32 + j];
            o = make_float2(alpha.x * re - alpha.y * im, alpha.x * im + alpha.y * re);
        }
        Cb[(long long)j * ldc + row] = o;
    }
    if (bad && tid == 0) atomicAdd(&g_tc_timeouts, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS));
}

std::atomic<int> g_tc_enabled{1};

}  // namespace

bool tc_gemm_enabled() { return g_tc_enabled.load() != 0; }
void tc_gemm_enable(bool on) { g_tc_enabled.store(on ? 1 : 0); }

bool tc_gemm_fits(int M, int N, int K) { return M > 0 && M % TC_M == 0 && K > 0 && K % (2 * TC_KC) == 0 && N >= 1 && N <= 32; }

lsw_status cgemm_tc(const float2* A, int lda, long long sA, const float2* B, int ldb, long long sB, float2* C, int ldc,
                    long long sC, int M, int N, int K, float2 alpha, int batch, cudaStream_t st) {
    if (!tc_gemm_fits(M, N, K) || batch <= 0 || batch > 65535) return LSW_ERR_INVALID_ARG;
    KTimer kt("leaf_tc", st, 8.0 * ((double)batch * M * K + (double)batch * K * N + (double)batch * M * N),
              8.0 * (double)batch * M * N * K);
    // A CTA takes the same time per stage however few there are, so one leaf of
    // 1024 on 8 CTAs cost as much as 30 leaves.  K is split until two CTAs per
    // SM are busy, with at least 8 stages each (8 CTAs of 128 stages become 128
    // of 8): the inversion's products with 1 to 32 leaves take 18 us on average
    // instead of 73 (256^2 build, one GB300).
    int ksplit = 1;
    while ((long long)(M / TC_M) * batch * ksplit * 2 <= 304 && K % (ksplit * 4 * TC_KC) == 0 &&
           K / (ksplit * 2) >= 8 * TC_KC)
        ksplit *= 2;
    if (ksplit == 1) {
        k_cgemm_tc<<<dim3(M / TC_M, batch), 128, 0, st>>>(A, lda, sA, B, ldb, sB, C, ldc, sC, 0, N, K, alpha);
        LSW_LAUNCH_CHECK();
        return LSW_OK;
    }
    DevBuf part;
    const long long mn = (long long)M * N;
    LSW_TRY(part.alloc(sizeof(float2) * (size_t)(ksplit * batch * mn), st));
    k_cgemm_tc<<<dim3(M / TC_M, batch, ksplit), 128, 0, st>>>(A, lda, sA, B, ldb, sB, part.as<float2>(), M, mn,
                                                                    batch * mn, N, K / ksplit, make_float2(1.f, 0.f));
    LSW_LAUNCH_CHECK();
    return gemm_reduce_parts<float>(M, N, batch, ksplit, part.as<float2>(), alpha, make_float2(0.f, 0.f), C, ldc, sC, st);
}

}  // namespace lsw

extern "C" lsw_status lsw_set_tensor_cores(int enable) {
    lsw::tc_gemm_enable(enable != 0);
    return LSW_OK;
}
