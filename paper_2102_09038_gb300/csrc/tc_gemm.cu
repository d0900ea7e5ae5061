// Tensor-core GEMM for sm_103a (tcgen05 + TMA) for the dense angular
// contractions of the hot path: the scattering apply U S^+ (eq. bKebKo) and
// the two eigenbasis contractions of (M^- - K^-)^{-1} (Lemma
// apply_high_order_pre taken over the full eigenbasis).
//
//   C[M x N] = epi(A[M x K] * B^T)   with A row-major (K contiguous) and the
//   second operand given K-major as Bt[N x K] (K contiguous)
//
// Operands are BF16 (tcgen05.mma kind::f16) or FP32 read as TF32
// (kind::tf32); accumulation is FP32 in tensor memory.  Tiles of 128 x BN:
// warp 0 issues TMA loads into a 4-stage shared-memory ring (128-byte
// swizzle), warp 1 the MMAs, warps 2 to 9 drain the accumulators with
// tcgen05.ld and apply the epilogue.  Blocks are persistent and the
// accumulator is double-buffered, so the loads and MMAs of a tile run under
// the epilogue of the one before: at the solver's sizes (K = 768) a
// tile's epilogue (a division per element, 64 to 128 KB of stores) takes about
// as long as its MMAs, and one tile per block exposed both.  Measured in a
// solve, 32768 x 768 x 768 BF16: with the shifted inverse in the epilogue 152
// -> 79 us, the plain product to FP32 81 -> 57 us.  Calls of at most one tile
// an SM gain nothing from it and lose nothing (a whole rte_gemm_lowp call, one
// tile per block of 128 threads before and now: 128 x 256 x 768 BF16 48 and 46
// us, 1000 x 100 x 128 TF32 47 and 46).  Every wait on an mbarrier is bounded:
// on timeout the kernel records an error flag and leaves instead of hanging.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "device.h"
#include "rte_internal.h"
#include "tc_gemm.h"
#include "tcgen05.cuh"

namespace rte {

namespace {

using namespace tc;

constexpr int kBM = 128;
constexpr int kStages = 4;

constexpr int kEpiWarps = 8;
constexpr int kTcThreads = 64 + 32 * kEpiWarps;

template <int BN, bool TF32, typename TOut>
__global__ void __launch_bounds__(kTcThreads, 1)
k_tc_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
          int M, int N, int K, TOut* __restrict__ C, int ldc, int epi,
          const float* __restrict__ at, const float* __restrict__ as,
          const float* __restrict__ lam, int rows, float beta) {
    constexpr uint32_t kABytes = kBM * kRowBytes;
    constexpr uint32_t kBBytes = BN * kRowBytes;
    constexpr uint32_t kTmemCols = 2 * BN;   // two FP32 accumulators, one column per N
    constexpr int kKB = TF32 ? 32 : 64;      // values of K per stage
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1024-byte alignment of the operand ring (swizzle atoms)
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sB = smem + kStages * kABytes;
    __shared__ __align__(8) uint64_t bars[2 * kStages + 4];
    __shared__ uint32_t tmem_slot;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntn = (N + BN - 1) / BN, tiles = ntn * ((M + kBM - 1) / kBM);
    const int kblocks = (K + kKB - 1) / kKB;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kStages,
                   accf0 = full0 + 16 * kStages, acce0 = accf0 + 16;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf0 + 8 * b, 1);
            mbar_init(acce0 + 8 * b, kEpiWarps);   // one arrival per epilogue warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    bool ok = true;

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------ TMA producer
        int st = 0;
        uint32_t ph = 1, loaded = 0;
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
            const int m0 = tile / ntn * kBM, n0 = tile % ntn * BN;
            for (int kb = 0; kb < kblocks; ++kb) {
                if (!mbar_wait(empty0 + 8 * st, ph)) { ok = false; break; }
                mbar_expect_tx(full0 + 8 * st, kABytes + kBBytes);
                tma_load_2d(smem_u32(sA + st * kABytes), &mapA, full0 + 8 * st, kb * kKB, m0);
                tma_load_2d(smem_u32(sB + st * kBBytes), &mapB, full0 + 8 * st, kb * kKB, n0);
                loaded |= 1u << st;
                if (++st == kStages) { st = 0; ph ^= 1; }
            }
        }
        // after a timeout: the copies still in flight land before the block
        // leaves (stages before st hold one of this round)
        if (!ok)
            for (int i = 0; i < kStages; ++i)
                if (loaded >> i & 1u) mbar_wait(full0 + 8 * i, i < st ? ph ^ 1u : ph);
    } else if (warp == 1) {
        // ------------------------------------------------- MMA issuer
        // the whole warp keeps warp-uniform values; one lane issues
        constexpr uint32_t idesc = (1u << 4)                                   // D: FP32
                                   | ((TF32 ? 2u : 1u) << 7)                   // A: TF32 / BF16
                                   | ((TF32 ? 2u : 1u) << 10)                  // B: TF32 / BF16
                                   | ((uint32_t)(BN >> 3) << 17)               // N
                                   | ((uint32_t)(kBM >> 4) << 24);             // M
        const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        int st = 0;
        uint32_t ph = 0, used = 0;
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++used) {
            const uint32_t buf = used & 1u;
            if (!mbar_wait_warp(acce0 + 8 * buf, (used >> 1 & 1u) ^ 1u)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t d = tm + buf * BN;
            for (int kb = 0; kb < kblocks; ++kb) {
                if (!mbar_wait_warp(full0 + 8 * st, ph)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t da = da0 + (uint64_t)(st * (kABytes >> 4)),
                               db = db0 + (uint64_t)(st * (kBBytes >> 4));
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)   // 4 MMAs of 32 bytes of K each
                        mma_issue(TF32, d, da + 2 * kk, db + 2 * kk, idesc,
                                  (kb > 0 || kk > 0) ? 1u : 0u);
                    mma_commit(empty0 + 8 * st);   // frees the stage once these MMAs have read it
                }
                if (++st == kStages) { st = 0; ph ^= 1; }
            }
            if (ok && elect_one()) mma_commit(accf0 + 8 * buf);
        }
    } else if (warp >= 2) {
        // ---------------------------------------------------------- epilogue
        const int wq = warp & 3, half = (warp - 2) >> 2;
        uint32_t used = 0;
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++used) {
            const uint32_t buf = used & 1u;
            const int m0 = tile / ntn * kBM, n0 = tile % ntn * BN;
            const int row = m0 + wq * 32 + lane;
            float fat = 0.f, fas = 0.f;
            if (epi != 0 && row < M) {
                const int rr = row % rows;
                fat = at[rr];
                fas = as[rr];
            }
            if (ok) {
                int got = 1;
                if (lane == 0) got = mbar_wait(accf0 + 8 * buf, used >> 1 & 1u);
                ok = __shfl_sync(0xffffffffu, got, 0) != 0;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int c0 = half * (BN / 2); c0 < (half + 1) * (BN / 2); c0 += 16) {
                float v[16];
                // every lane of the warp takes part in the load, whatever its row
                tmem_ld16(tmem + ((uint32_t)(wq * 32) << 16) + buf * BN + (uint32_t)c0, v);
                if (c0 + 16 == (half + 1) * (BN / 2)) {
                    // the buffer is free once every warp has read its part
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce0 + 8 * buf);
                }
                if (!ok || row >= M || n0 + c0 >= N) continue;
                TOut* dst = C + (size_t)row * ldc + n0 + c0;
                const bool full = n0 + c0 + 16 <= N && beta == 0.f &&
                                  ((reinterpret_cast<uintptr_t>(dst) & 15) == 0);
                if (full) {
                    if (epi == 1) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            v[i] = v[i] / (fat - __ldg(lam + n0 + c0 + i) * fas);
                    }
                    if constexpr (sizeof(TOut) == 4) {
                        float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            d4[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    } else {
                        uint32_t w[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                            w[i] = *reinterpret_cast<uint32_t*>(&h);
                        }
                        uint4* d4 = reinterpret_cast<uint4*>(dst);
                        d4[0] = make_uint4(w[0], w[1], w[2], w[3]);
                        d4[1] = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                    continue;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int col = n0 + c0 + i;
                    if (col >= N) break;
                    float x = v[i];
                    if (epi == 1) x = x / (fat - lam[col] * fas);
                    if (beta != 0.f) x += beta * static_cast<float>(dst[i]);
                    dst[i] = static_cast<TOut>(x);
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols));
}

// A wait for an arrival that never comes: it runs out and sets the pipelines'
// flag, as a wait in the kernels above would.
__global__ void k_wait_alone() {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(smem_u32(&bar), 1);
    mbar_wait(smem_u32(&bar), 0);
}

template <int BN>
constexpr size_t smem_bytes() {
    return 1024 + (size_t)kStages * (kBM + BN) * kRowBytes;   // 1024: alignment
}

template <int BN, bool TF32, typename TOut>
int launch(cudaStream_t s, const TcGemmArgs& g) {
    CUtensorMap ma, mb;
    RTE_TRY(make_map(&ma, g.A, TF32, g.M, g.K, kBM));
    RTE_TRY(make_map(&mb, g.Bt, TF32, g.N, g.K, BN));
    auto kern = k_tc_gemm<BN, TF32, TOut>;
    const size_t sm = smem_bytes<BN>();
    // set on every call: the attribute is per device, and cheap to set
    RTE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const long long tiles = (long long)((g.N + BN - 1) / BN) * ((g.M + kBM - 1) / kBM);
    count_launches(1);
    kern<<<(unsigned)std::min<long long>(tiles, device_sm_count()), kTcThreads, sm, s>>>(
        ma, mb, g.M, g.N, g.K, static_cast<TOut*>(g.C), g.ldc, g.epi, g.at, g.as, g.lam, g.rows,
        g.beta);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

}  // namespace

int tc_gemm(cudaStream_t s, const TcGemmArgs& g) {
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return RTE_OK;
    if (g.bn != 0 && g.bn != 128 && g.bn != 256) return fail(RTE_ERR_ARG, "tile width 128 or 256");
    const bool wide = g.bn ? g.bn == 256 : g.N > 128;
    if (g.tf32) {
        if (g.out_bf16) return fail(RTE_ERR_ARG, "TF32 GEMM writes FP32");
        return wide ? launch<256, true, float>(s, g) : launch<128, true, float>(s, g);
    }
    if (g.out_bf16)
        return wide ? launch<256, false, __nv_bfloat16>(s, g)
                    : launch<128, false, __nv_bfloat16>(s, g);
    return wide ? launch<256, false, float>(s, g) : launch<128, false, float>(s, g);
}

int tc_set_wait_cycles(long long cycles) {
    RTE_CUDA_TRY(cudaMemcpyToSymbol(g_tc_wait_cycles, &cycles, sizeof(cycles)));
    return RTE_OK;
}

int tc_gemm_flag(const int** flag) {
    RTE_CUDA_TRY(cudaGetSymbolAddress((void**)flag, g_tc_error));
    return RTE_OK;
}

int tc_gemm_error_check(cudaStream_t s, int flag) {
    if (!flag) return RTE_OK;
    const int zero = 0;
    cudaMemcpyToSymbolAsync(g_tc_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
    return fail(RTE_ERR_TIMEOUT, "a tensor-core GEMM pipeline wait timed out");
}

int tc_gemm_error(cudaStream_t s) {
    int e = 0;
    RTE_CUDA_TRY(cudaMemcpyFromSymbolAsync(&e, g_tc_error, sizeof(int), 0,
                                           cudaMemcpyDeviceToHost, s));
    RTE_CUDA_TRY(cudaStreamSynchronize(s));
    return tc_gemm_error_check(s, e);
}

int tc_wait_selftest(cudaStream_t s) {
    count_launches(1);
    k_wait_alone<<<1, 32, 0, s>>>();
    RTE_CUDA_TRY(cudaGetLastError());
    RTE_CUDA_TRY(cudaStreamSynchronize(s));
    return RTE_OK;
}

}  // namespace rte

// ======================================================================
// FP64-accurate GEMM from exact BF16 tensor-core products (error-free
// splitting of the operands, after Ozaki, Ogita, Oishi and Rump).
//
// Every row of A (and of the K-major second operand Bt) is scaled by a power
// of two 2^e so that its entries lie in (-1, 1), then cut into S digit
// slices: r <- r * 2^7, d = rint(r), r <- r - d.  The digits are integers
// with |d| <= 128, exact in BF16, and A = 2^e sum_s d_s 2^{-7(s+1)} up to a
// remainder below 2^{-7S-1}.  A product of two digit slices summed over at
// most 1024 terms is an integer below 2^24, so the tensor cores' FP32
// accumulation of it is exact.  The kernel accumulates the slice pairs
// (s, t) with s + t <= S - 1 (the others lie below the truncation level)
// in groups of one weight 2^{-7(s+t+2)} each: a group owns a tensor-memory
// accumulator over 512 terms of K, and holds pairs whose digit bounds add up
// to at most 2^15 per term (|d_0 d_0| <= 2^14, |d_0 d_t| <= 2^13, |d_s d_t|
// <= 2^12 for s, t > 0), so its sum stays an integer of magnitude at most
// 2^15 * 512 = 2^24 and the FP32 accumulation is exact in any order (the
// tensor cores truncate when they add, so only exact sums are safe).  A
// weight with more pairs than that takes two groups.  Each accumulator is
// folded into double-float registers with its weight; the row and column
// scales come last.
//
// What bounds it: the tensor pipe and the L2 -> SM path.  One slice pair of a
// 128 x 128 x 64 block is 2.1 MFLOP for 32 KB of operands, so loading a tile
// per pair (the earlier design) needs more L2 bandwidth than there is
// (11 TB/s at a third of the tensor rate).  Here every accumulator of a tile
// is resident at once (groups x BN columns of the 512 of tensor memory), so
// a K step of 16 loads each of the S + S slices once and uses them for all
// S(S+1)/2 pairs; BN is the widest that fits (96 for S = 5, 80 for 6, 64 for
// 7) unless a narrower one fills the GPU better.  The B slices of a step lie
// one after the other in shared memory and the accumulators of successive
// weights in tensor memory, so A_s times B_t, B_t+1, ... is one MMA of up to
// 256 columns, which reads A_s once.  Measured (S slices, BF16 products of the
// S(S+1)/2 pairs, kernel time by ncu): 9216 x 3072 x 1024, S = 6: 0.77 ms,
// 1.58 PFLOP/s, 0.83 of the measured BF16 peak; 18432 x 768 x 768, S = 5:
// 0.24 ms, 1.35 PFLOP/s (0.62 ms before), S = 7: 0.47 ms.  What is left is the
// chunk boundaries and the shared-memory traffic of operands and copies.
// ======================================================================
namespace rte {

namespace {

using namespace tc;

constexpr int kOzBM = 128;
constexpr int kOzChunk = 32;         // K steps of 16 per exact chunk (512)
constexpr int kOzMaxStages = 6;
constexpr int kOzSmemMax = 224 * 1024;   // dynamic; the barriers are static

__host__ __device__ constexpr int oz_stage_bytes(int BN, int S) { return S * 32 * (kOzBM + BN); }
__host__ __device__ constexpr int oz_stages(int BN, int S) {
    return kOzSmemMax / oz_stage_bytes(BN, S) < kOzMaxStages ? kOzSmemMax / oz_stage_bytes(BN, S)
                                                              : kOzMaxStages;
}
// Groups of slice pairs, by the digit bounds above: weights 0 to 5 take one
// group, 6 and more take two (2 * 8192 + 5 * 4096 > 2^15 at weight 6); the
// second one holds the pairs whose A slice is 6 (weight 6) or at least 7.
__host__ __device__ constexpr int oz_groups(int S) { return S <= 6 ? S : 2 * S - 6; }
__host__ __device__ constexpr int oz_weight(int g) { return g < 6 ? g : 6 + (g - 6) / 2; }
__host__ __device__ constexpr int oz_group(int a, int b) {
    return a + b < 6 ? a + b : 2 * (a + b) - 6 + (a >= (a + b == 6 ? 6 : 7) ? 1 : 0);
}
// B slices b, b + 1, ... one MMA takes with A slice a: successive weights in
// successive groups (so in neighbouring accumulators), at most 256 columns
__host__ __device__ constexpr int oz_run(int S, int BN, int a, int b) {
    int len = 1;
    while (a + b + len < S && oz_group(a, b + len) == oz_group(a, b) + len && (len + 1) * BN <= 256)
        ++len;
    return len;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand without swizzle:
// core matrices of 8 rows x 16 bytes are contiguous, the next 8 rows follow
// 128 bytes later (stride offset) and the next 8 values of K `lead` bytes
// later (leading offset).
__device__ __forceinline__ uint64_t plain_desc(uint32_t addr, uint32_t lead) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(lead >> 4) << 16) |
           ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}

// CW columns (a multiple of 4, at most 28) of this warp's 32 accumulator rows
template <int CW>
__device__ __forceinline__ void tmem_ld_cols(uint32_t t, float (&v)[CW]) {
    uint32_t r[CW];
    if constexpr (CW >= 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
              "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
              "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(t));
    }
    if constexpr (CW % 16 >= 8) {
        constexpr int o = CW / 16 * 16;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]),
              "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
            : "r"(t + o));
    }
    if constexpr (CW % 8 == 4) {
        constexpr int o = CW / 8 * 8;
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3])
                     : "r"(t + o));
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    // tie the registers to the wait, so that no use moves above it
#pragma unroll
    for (int i = 0; i < CW; ++i) asm volatile("" : "+r"(r[i]));
#pragma unroll
    for (int i = 0; i < CW; ++i) v[i] = __uint_as_float(r[i]);
}

// 18 warps: warp 0 issues TMA loads, warp 1 issues MMAs, warps 2..17 drain
// the accumulators (warp w reads TMEM lanes 32 (w % 4) .. + 31 and the
// quarter (w - 2) / 4 of the columns), so the producer and the MMA issuer
// never wait on the epilogue's own arrivals.
constexpr int kOzThreads = 576;
constexpr int kOzEpiWarps = 16;

// f 2^E as an FP64 bit pattern built with integer operations (sign, the
// exponent rebased and shifted by E, the 23 mantissa bits moved up): exact,
// and no FP64 instruction, which this GPU issues at a small fraction of its
// FP32 and integer rates.  False where f is subnormal, infinite or NaN or
// f 2^E leaves the normal FP64 range.
__device__ __forceinline__ bool f32_scaled_to_f64(float f, int E, double* out) {
    const uint32_t b = __float_as_uint(f);
    const uint32_t mag = b & 0x7FFFFFFFu;
    if (mag == 0) {
        *out = __longlong_as_double((long long)(b & 0x80000000u) << 32);
        return true;
    }
    const int e8 = (int)(mag >> 23);
    const int e11 = e8 + (1023 - 127) + E;
    if (e8 == 0 || e8 == 255 || e11 < 1 || e11 > 2046) return false;
    const uint64_t bits = ((uint64_t)(b & 0x80000000u) << 32) | ((uint64_t)e11 << 52) |
                          ((uint64_t)(mag & 0x7FFFFFu) << 29);
    *out = __longlong_as_double((long long)bits);
    return true;
}

// (hi + lo) 2^E rounded once to FP64: both parts widened and scaled exactly,
// then one FP64 add; out-of-range cases take the FP64 route
__device__ __forceinline__ double df_scaled_to_f64(float hi, float lo, int E) {
    double a, b;
    if (f32_scaled_to_f64(hi, E, &a) && f32_scaled_to_f64(lo, E, &b)) return a + b;
    return ldexp((double)hi + (double)lo, E);
}

// four consecutive doubles at a 32-byte aligned address
__device__ __forceinline__ void ld_f64x4(const double* p, double (&v)[4]) {
    asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p));
}
__device__ __forceinline__ void st_f64x4(double* p, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
                 "d"(v[2]), "d"(v[3])
                 : "memory");
}

// Every MMA of one K step, A_a against runs of B slices, from (a, b) on; da,
// db: the stage's descriptors, tm: tensor memory base.  All offsets are
// compile-time constants (kOzIdesc: FP32 accumulator, BF16 operands, M = 128).
constexpr uint32_t kOzIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kOzBM >> 4) << 24);
template <int S, int BN, int a, int b>
__device__ __forceinline__ void oz_issue_wide(uint32_t tm, uint64_t da, uint64_t db) {
    if constexpr (a < S && a + b >= S) {
        oz_issue_wide<S, BN, a + 1, 0>(tm, da, db);
    } else if constexpr (a < S) {
        constexpr int len = oz_run(S, BN, a, b);
        mma_issue(false, tm + (uint32_t)(oz_group(a, b) * BN), da + (uint64_t)(a * kOzBM),
                  db + (uint64_t)(b * BN), kOzIdesc | ((uint32_t)(len * BN / 8) << 17), 1u);
        oz_issue_wide<S, BN, a, b + len>(tm, da, db);
    }
}
// The pairs of group g alone, from A slice a on; fresh: the first one
// overwrites the accumulator.
template <int S, int BN, int g, int a>
__device__ __forceinline__ void oz_issue_group(uint32_t tm, uint64_t da, uint64_t db, bool fresh) {
    constexpr int b = oz_weight(g) - a;
    if constexpr (b >= 0) {
        constexpr bool mine = oz_group(a, b) == g;
        if constexpr (mine)
            mma_issue(false, tm + (uint32_t)(g * BN), da + (uint64_t)(a * kOzBM),
                      db + (uint64_t)(b * BN), kOzIdesc | ((uint32_t)(BN / 8) << 17),
                      fresh ? 0u : 1u);
        oz_issue_group<S, BN, g, a + 1>(tm, da, db, mine ? false : fresh);
    }
}

// f(g) for g = 0 .. n - 1 as compile-time constants while it returns true
template <int n, int g = 0, typename F>
__device__ __forceinline__ bool oz_each_group(F&& f) {
    if constexpr (g < n) {
        if (!f(std::integral_constant<int, g>{})) return false;
        return oz_each_group<n, g + 1>(f);
    }
    return true;
}

// Persistent: block b computes the tiles b, b + gridDim.x, ... (column tiles
// fastest, so the blocks running together share A slices in L2), and the
// epilogue of one tile overlaps the MMAs of the next.  With every group's
// accumulator in use there is no second buffer to drain from; instead the
// last `tail` K steps of a chunk and the first of the next one run group by
// group, so that a group is complete, drained and free again while the MMAs
// of the other groups run.
template <int BN, int S>
__global__ void __launch_bounds__(kOzThreads, 1)
k_ozaki(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
        int M, int N, int K, const int* __restrict__ ea, const int* __restrict__ eb,
        double* __restrict__ C, int ldc, int epi, const double* __restrict__ rinv, int rows,
        int vec) {
    constexpr int CW = BN / 4;   // columns per epilogue thread
    extern __shared__ __align__(128) uint8_t smem_raw[];
    constexpr int groups = oz_groups(S), stages = oz_stages(BN, S);
    constexpr uint32_t abytes = S * 2 * kOzBM * 16, bbytes = S * 2 * BN * 16;
    uint8_t* sA = smem_raw;
    uint8_t* sB = sA + (size_t)stages * abytes;
    __shared__ __align__(8) uint64_t bars[2 * stages + 2 * groups];
    __shared__ uint32_t tmem_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntn = (N + BN - 1) / BN, tiles = ntn * ((M + kOzBM - 1) / kOzBM);
    const int ksteps = (K + 15) / 16;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * stages,
                   accf0 = full0 + 16 * stages, acce0 = accf0 + 8 * groups;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int g = 0; g < groups; ++g) {
            mbar_init(accf0 + 8 * g, 1);
            mbar_init(acce0 + 8 * g, kOzEpiWarps);   // one arrival per epilogue warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    bool ok = true;

    if (warp == 0 && lane == 0) {
        // --------------------------------------------- TMA producer
        int st = 0;
        uint32_t ph = 1;   // a fresh barrier passes a wait for the phase before
        uint32_t loaded = 0;   // stages with a copy not known to be complete
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
            const int m0 = tile / ntn * kOzBM, n0 = tile % ntn * BN;
            for (int k = 0; k < ksteps; ++k) {
                if (!mbar_wait(empty0 + 8 * st, ph)) { ok = false; break; }
                mbar_expect_tx(full0 + 8 * st, abytes + bbytes);
                tma_load_3d(smem_u32(sA + (size_t)st * abytes), &mapA, full0 + 8 * st, 2 * m0, 0,
                            2 * k);
                tma_load_3d(smem_u32(sB + (size_t)st * bbytes), &mapB, full0 + 8 * st, 2 * n0, 0,
                            2 * k);
                loaded |= 1u << st;
                if (++st == stages) { st = 0; ph ^= 1; }
            }
        }
        // every copy has arrived before the block leaves: the MMAs consumed
        // them all, or (after a timeout) wait for the last one of each stage
        if (!ok)
            for (int i = 0; i < stages; ++i) {
                // stages before st hold a copy of this round, the others of
                // the previous one
                const uint32_t par = i < st ? ph ^ 1u : ph;
                if (loaded >> i & 1u) mbar_wait(full0 + 8 * i, par);
            }
    } else if (warp == 1) {
        // ---------------------------------------------- MMA issuer
        // One lane issues every MMA, so what it does per MMA must stay below
        // the MMA's own time (32 to 128 cycles): the slice count and width
        // are compile-time, so every offset and instruction descriptor is an
        // immediate, and the whole warp runs this loop with warp-uniform
        // values (the MMAs take them from uniform registers; descriptors
        // built in a one-lane branch are moved there one by one).  Measured
        // on 18432 x 768 x 768, S = 5: 620 us with the offsets in a table in
        // shared memory and a one-lane branch, 407 us uniform with the table
        // in the kernel's parameters, 241 us this way.
        const uint64_t da0 = plain_desc(smem_u32(sA), S * kOzBM * 16);
        const uint64_t db0 = plain_desc(smem_u32(sB), S * BN * 16);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        constexpr int tail_max = stages > 3 ? stages - 2 : 1;
        int st = 0;
        uint32_t ph = 0;
        uint32_t used = 0;   // chunks done: phase of the accumulators
        auto next = [&](int& s, uint32_t& p) {
            if (++s == stages) { s = 0; p ^= 1; }
        };
        auto wait_full = [&](int s, uint32_t p) {
            const bool got = mbar_wait_warp(full0 + 8 * s, p);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            return got;
        };
        auto adesc = [&](int s) { return da0 + (uint64_t)((uint32_t)s * abytes >> 4); };
        auto bdesc = [&](int s) { return db0 + (uint64_t)((uint32_t)s * bbytes >> 4); };
        // group g on a stage once its accumulator has been drained
        auto first_of = [&](auto gc, int s, uint32_t eph) {
            constexpr int g = decltype(gc)::value;
            if (!mbar_wait_warp(acce0 + 8 * g, eph)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) oz_issue_group<S, BN, g, 0>(tm, adesc(s), bdesc(s), true);
            return true;
        };
        // group g on the last `tail` stages of a chunk (from stage s on);
        // begun: earlier stages of the chunk have been accumulated
        auto last_of = [&](auto gc, int s, uint32_t p, int tail, bool begun, uint32_t eph) {
            constexpr int g = decltype(gc)::value;
            for (int i = 0; i < tail; ++i) {
                if (g == 0 && !wait_full(s, p)) return false;
                if (i == 0 && !begun) {
                    if (!first_of(gc, s, eph)) return false;
                } else if (elect_one()) {
                    oz_issue_group<S, BN, g, 0>(tm, adesc(s), bdesc(s), false);
                }
                next(s, p);
            }
            if (elect_one()) mma_commit(accf0 + 8 * g);
            return true;
        };
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x)
            for (int k0 = 0; k0 < ksteps && ok; k0 += kOzChunk, ++used) {
                const int ns = min(kOzChunk, ksteps - k0);
                const int tail = min(tail_max, ns), head = ns - tail;
                const uint32_t eph = (used & 1u) ^ 1u;
                for (int i = 0; i < head; ++i) {
                    if (!wait_full(st, ph)) { ok = false; break; }
                    if (i == 0) {
                        ok = oz_each_group<groups>([&](auto gc) { return first_of(gc, st, eph); });
                        if (!ok) break;
                    } else if (elect_one()) {
                        oz_issue_wide<S, BN, 0, 0>(tm, adesc(st), bdesc(st));
                    }
                    if (elect_one()) mma_commit(empty0 + 8 * st);
                    next(st, ph);
                }
                if (!ok) break;
                ok = oz_each_group<groups>(
                    [&](auto gc) { return last_of(gc, st, ph, tail, head > 0, eph); });
                for (int i = 0; i < tail; ++i) {
                    if (elect_one()) mma_commit(empty0 + 8 * st);
                    next(st, ph);
                }
            }
    } else if (warp >= 2) {
        // -------------------------------------------------------- epilogue
        const int wq = warp & 3, quarter = (warp - 2) >> 2;
        uint32_t used = 0;
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int m0 = tile / ntn * kOzBM, n0 = tile % ntn * BN;
            // Double-float accumulators (hi + lo, about 48 significant bits):
            // every drain adds v 2^-7(s+t+2) with v an integer below 2^24,
            // exact in FP32; the two-sum keeps the rounding error of each
            // addition in lo.  FP32 runs at many times the FP64 rate.
            float hi[CW], lo[CW];
#pragma unroll
            for (int i = 0; i < CW; ++i) hi[i] = lo[i] = 0.f;
            for (int k0 = 0; k0 < ksteps; k0 += kOzChunk, ++used) {
                for (int g = 0; g < groups; ++g) {
                    // lane 0 polls for its warp: 512 polling threads would take
                    // issue slots from the MMA warp
                    if (ok) {
                        int got = 1;
                        if (lane == 0) got = mbar_wait(accf0 + 8 * g, used & 1u);
                        ok = __shfl_sync(0xffffffffu, got, 0) != 0;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const float w = __int_as_float((127 - 7 * (oz_weight(g) + 2)) << 23);
                    float v[CW];
                    tmem_ld_cols<CW>(tmem + ((uint32_t)(wq * 32) << 16) +
                                         (uint32_t)(g * BN + quarter * CW),
                                     v);
                    // the accumulator is free once every warp has read it
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce0 + 8 * g);
#pragma unroll
                    for (int i = 0; i < CW; ++i) {
                        const float x = v[i] * w;                 // exact
                        const float sum = __fadd_rn(hi[i], x);
                        const float bb = __fsub_rn(sum, hi[i]);
                        const float err = __fadd_rn(__fsub_rn(hi[i], __fsub_rn(sum, bb)),
                                                    __fsub_rn(x, bb));
                        hi[i] = sum;
                        lo[i] = __fadd_rn(lo[i], err);
                    }
                }
            }
            // a thread finishes its row's CW columns: whole 32-byte sectors
            // where the rows are aligned (vec)
            const int row = m0 + wq * 32 + lane, c0 = n0 + quarter * CW;
            if (!ok || row >= M) continue;
            const int er = __ldg(ea + row);
            const double* rr = epi == 1 ? rinv + (size_t)(row % rows) * N : nullptr;
            double* dst = C + (size_t)row * ldc;
#pragma unroll
            for (int i = 0; i < CW; i += 4) {
                const int col = c0 + i;
                if (col >= N) break;
                double x[4], f[4];
                if (vec) {   // N is a multiple of 4: the four columns exist
                    if (epi == 1) ld_f64x4(rr + col, f);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        x[j] = df_scaled_to_f64(hi[i + j], lo[i + j], er + __ldg(eb + col + j));
                        if (epi == 1) x[j] *= f[j];
                    }
                    st_f64x4(dst + col, x);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (col + j < N) {
                            double y = df_scaled_to_f64(hi[i + j], lo[i + j],
                                                        er + __ldg(eb + col + j));
                            if (epi == 1) y *= rr[col + j];
                            dst[col + j] = y;
                        }
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// 1 / (at[r] - lam[c] as[r]) for r < rows, c < N, row-major: the diagonal of
// (M^- - K^-)^{-1} in the eigenbasis per cell, built once so that the split
// GEMM's epilogue multiplies instead of dividing in FP64
__global__ void k_oz_recip(int rows, int N, const double* __restrict__ at,
                           const double* __restrict__ as, const double* __restrict__ lam,
                           double* __restrict__ out) {
    const size_t total = (size_t)rows * N;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / N), c = (int)(e % N);
        out[e] = 1.0 / (at[r] - lam[c] * as[r]);
    }
}

// x's integer X = round(x 2^(7S - ex)) for the row exponent ex (emax its
// biased form): the FP64 mantissa shifted once to the row's fixed point
__device__ __forceinline__ long long oz_fixed(double x, int S, int emax) {
    const long long bits = __double_as_longlong(x);
    const int be = (int)((bits >> 52) & 0x7FF);
    if (be == 0 || emax == 0) return 0;
    const long long mant = (bits & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
    // x 2^(7S - ex) = mant 2^(be - 1075 + 7S - ex)
    const int sh = be - 1075 + 7 * S - (emax - 1022);
    long long v = 0;
    if (sh >= 0)
        v = sh <= 10 ? (mant << sh) : 0;   // S = 8, 9 (|v| < 2^(7S) <= 2^63)
    else if (sh > -60)
        v = (mant + (1ll << (-sh - 1))) >> (-sh);
    return bits < 0 ? -v : v;
}

// Digit slices of the rows of X (rows x K FP64, K a multiple of 8), in the
// layout the GEMM's shared-memory tiles have: out[k / 8][s][row][k % 8], so
// that the S slices of 8 columns of a row tile are S contiguous pieces.
// Exponent ex of the row maximum (|x| < 2^ex), then the S balanced base-128
// digits of X in integer arithmetic, peeled from the least significant end,
// d = ((X + 64) mod 128) - 64, X <- (X - d) / 128; the leading digit keeps
// the rest (|d_0| <= 128).  x 2^-ex = sum_s d_s 2^{-7(s+1)} + r with |r| <=
// 2^{-7S-1}.  A block takes R = 32, 16 or 8 rows: its warps find their maxima
// (one row per warp and trip), then lane l cuts 8 columns of row l % R and
// stores 16 bytes per slice next to its neighbours', so the stores are runs
// of 16 R bytes and the second read of the rows comes from L2.  The digits
// are peeled four at a time in 32-bit registers and turned into BF16 by an
// exact FP32 add of 1.5 2^23 and byte moves: integer-to-float conversions
// and 64-bit shifts run at a quarter or less of the 32-bit rate.
// VEC: rows start on 32 bytes.
template <bool VEC>
__global__ void __launch_bounds__(1024)
k_oz_split(const double* __restrict__ X, int rows, int K, int S, int R,
           __nv_bfloat16* __restrict__ out, int* __restrict__ e) {
    __shared__ int s_emax[32];
    const int r0 = blockIdx.x * R, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int warps = blockDim.x >> 5;
    for (int rl = warp; rl < R; rl += warps) {
        const int row = r0 + rl;
        int emax = 0;
        if (row < rows) {
            const double* x = X + (size_t)row * K;
            if constexpr (VEC) {
                for (int k = 4 * lane; k < K; k += 128) {
                    double v[4];
                    ld_f64x4(x + k, v);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        emax = max(emax, __double2hiint(v[j]) >> 20 & 0x7FF);
                }
            } else {
                for (int k = lane; k < K; k += 32) emax = max(emax, __double2hiint(x[k]) >> 20 & 0x7FF);
            }
        }
        emax = __reduce_max_sync(0xffffffffu, emax);
        if (lane == 0) {
            s_emax[rl] = emax;
            if (row < rows) e[row] = emax == 0 ? 0 : emax - 1022;
        }
    }
    __syncthreads();
    const int rl = lane & (R - 1), row = r0 + rl;
    if (row >= rows) return;
    const int emax = s_emax[rl], per = 32 / R;   // groups of 8 columns per warp and trip
    const double* x = X + (size_t)row * K;
    uint4* o = reinterpret_cast<uint4*>(out);
    for (int k8 = warp * per + lane / R; k8 < K / 8; k8 += warps * per) {
        double v[8];
        if constexpr (VEC) {
            double a[4], b[4];
            ld_f64x4(x + 8 * k8, a);
            ld_f64x4(x + 8 * k8 + 4, b);
#pragma unroll
            for (int j = 0; j < 4; ++j) { v[j] = a[j]; v[4 + j] = b[j]; }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = x[8 * k8 + j];
        }
        long long q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) q[j] = oz_fixed(v[j], S, emax);
        auto store = [&](int s, const int (&d)[8]) {
            uint32_t f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                f[j] = __float_as_uint(__int_as_float(0x4B400000 + d[j]) - 12582912.f);
            o[((size_t)k8 * S + s) * rows + row] =
                make_uint4(__byte_perm(f[0], f[1], 0x7632), __byte_perm(f[2], f[3], 0x7632),
                           __byte_perm(f[4], f[5], 0x7632), __byte_perm(f[6], f[7], 0x7632));
        };
        int s = S - 1;
        while (s > 0) {
            // four digits from the low 28 bits, or the last up to three of a
            // rest that fits 32 bits
            const int cnt = min(s, 4);
            int t[8], d[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] = cnt == 4 ? (int)(q[j] & 0xFFFFFFFll) : (int)q[j];
            for (int c = 0; c < cnt; ++c) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = (t[j] + 64) >> 7;
                    d[j] = t[j] - (n << 7);
                    t[j] = n;
                }
                store(s - c, d);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) q[j] = cnt == 4 ? (q[j] >> 28) + t[j] : (long long)t[j];
            s -= cnt;
        }
        int lead[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) lead[j] = (int)q[j];
        store(0, lead);
    }
}

// Tensor map of digit slices [K / 8][SB][rows][8] BF16 as 8-byte words (a
// tile of up to 128 rows is then one box row of 256 words): box = tile_rows x
// S slices x 16 columns, zero fill out of bounds.
int make_slice_map(CUtensorMap* map, const void* base, int rows, int K, int SB, int S,
                   int tile_rows) {
    auto fn = encode_fn();
    if (!fn) return fail(RTE_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
    if ((reinterpret_cast<uintptr_t>(base) & 15) || K % 8)
        return fail(RTE_ERR_ARG, "tensor-core GEMM operand is not 16-byte aligned");
    cuuint64_t dims[3] = {(cuuint64_t)rows * 2, (cuuint64_t)SB, (cuuint64_t)K / 8};
    cuuint64_t strides[2] = {(cuuint64_t)rows * 16, (cuuint64_t)rows * 16 * SB};
    cuuint32_t box[3] = {(cuuint32_t)tile_rows * 2, (cuuint32_t)S, 2};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<void*>(base), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(RTE_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    return RTE_OK;
}

struct OzArgs {
    const void *A, *B;
    const int *ea, *eb;
    int M, N, K, SB;
    double* C;
    int ldc, epi;
    const double* rinv;
    int rows;
};

template <int BN, int S>
int oz_launch(cudaStream_t s, const OzArgs& g) {
    CUtensorMap ma, mb;
    RTE_TRY(make_slice_map(&ma, g.A, g.M, g.K, S, S, kOzBM));
    RTE_TRY(make_slice_map(&mb, g.B, g.N, g.K, g.SB, S, BN));
    constexpr int sm = oz_stages(BN, S) * oz_stage_bytes(BN, S);
    auto kern = k_ozaki<BN, S>;
    // set on every call: the attribute is per device, and cheap to set
    RTE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    const long long tiles = (long long)((g.N + BN - 1) / BN) * ((g.M + kOzBM - 1) / kOzBM);
    const int vec = g.N % 4 == 0 && g.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(g.C) & 31) == 0 &&
                    (g.epi == 0 || (reinterpret_cast<uintptr_t>(g.rinv) & 31) == 0);
    count_launches(1);
    kern<<<(unsigned)std::min<long long>(tiles, device_sm_count()), kOzThreads, sm, s>>>(
        ma, mb, g.M, g.N, g.K, g.ea, g.eb, g.C, g.ldc, g.epi, g.rinv, g.rows, vec);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

// Tile width: the one with the least estimated time among those built: waves
// of tiles, each of K / 16 steps of BN / 2 cycles a pair plus 480 for what a
// step costs whatever its width (A slices read from shared memory, barriers,
// issue), plus 5000 cycles for a tile's drains and finish.  The constants fit
// the times measured on 18432 x 768 x 768 (S = 5: 241, 307, 494 us at widths
// 96, 64, 32; S = 7: 474, 550, 726 us at 64, 48, 32) and 9216 x 3072 x 1024
// (S = 6: 772, 885, 1388 us at 80, 64, 32) to about 15 %: the widest tile
// wins wherever there are tiles for every SM, narrower ones below.
int oz_width(int M, int N, int K, int S, const int* widths, int n) {
    const int pairs = S * (S + 1) / 2, sms = device_sm_count();
    int best = widths[0];
    double best_cost = 1e300;
    for (int i = 0; i < n; ++i) {
        const int bn = widths[i];
        const double tiles = std::ceil((double)N / bn) * std::ceil((double)M / kOzBM);
        const double cost =
            std::ceil(tiles / sms) * (std::ceil(K / 16.0) * (pairs * bn * 0.5 + 480.0) + 5000.0);
        if (cost < best_cost) {
            best_cost = cost;
            best = bn;
        }
    }
    return best;
}

// The widest tile whose accumulators fit, and narrower ones for problems of
// few tiles.
template <int S, int W0, int W1, int W2>
int oz_run_width(cudaStream_t s, const OzArgs& g) {
    static_assert(oz_groups(S) * W0 <= 512, "accumulators must fit in tensor memory");
    const int widths[3] = {W0, W1, W2};
    const int w = oz_width(g.M, g.N, g.K, S, widths, 3);
    if (w == W0) return oz_launch<W0, S>(s, g);
    if (w == W1) return oz_launch<W1, S>(s, g);
    return oz_launch<W2, S>(s, g);
}

}  // namespace

size_t ozaki_slice_bytes(int rows, int K, int S) {
    return (size_t)S * rows * K * sizeof(__nv_bfloat16) + (size_t)rows * sizeof(int) + 512;
}

int ozaki_split(cudaStream_t s, const double* X, int rows, int K, int S, void* out, int** e) {
    char* p = static_cast<char*>(out);
    __nv_bfloat16* sl = reinterpret_cast<__nv_bfloat16*>(p);
    int* ex = reinterpret_cast<int*>(p + (((size_t)S * rows * K * 2 + 255) / 256) * 256);
    if (e) *e = ex;
    if (rows <= 0 || K % 8) return RTE_OK;   // the GEMM refuses such a K
    // 32 rows a block of 256 threads where that gives every SM two blocks,
    // else 16, or 8, rows of 512 or 1024: a short operand is then cut by as
    // many warps as a long one (1500 x 384 x 3072 at seven slices, the whole
    // product: 279 -> 229 us).  1500 x 384 in the static scratch, 256, 512 and
    // 1024 threads: K = 768 93, 86, 86 us; up to K = 512 all within 1 us.
    const int sms = device_sm_count();
    const int R = rows >= 64 * sms ? 32 : rows >= 16 * sms ? 16 : 8;
    const int threads = R == 32 ? 256 : K >= 512 ? 1024 : 512;
    const unsigned blocks = (unsigned)((rows + R - 1) / R);
    count_launches(1);
    if ((reinterpret_cast<uintptr_t>(X) & 31) == 0)
        k_oz_split<true><<<blocks, threads, 0, s>>>(X, rows, K, S, R, sl, ex);
    else
        k_oz_split<false><<<blocks, threads, 0, s>>>(X, rows, K, S, R, sl, ex);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

int ozaki_recip_table(cudaStream_t s, const double* at, const double* as, const double* lam,
                      int rows, int N, double* out) {
    if (rows <= 0 || N <= 0) return RTE_OK;
    count_launches(1);
    const size_t total = (size_t)rows * N;
    const unsigned blocks =
        (unsigned)std::min<size_t>((total + 255) / 256, (size_t)device_sm_count() * 8);
    k_oz_recip<<<blocks, 256, 0, s>>>(rows, N, at, as, lam, out);
    RTE_CUDA_TRY(cudaGetLastError());
    return RTE_OK;
}

int ozaki_gemm(cudaStream_t s, const void* Aslices, const int* ea, int M, const void* Bslices,
               const int* eb, int N, int K, int S, double* C, int ldc, int epi,
               const double* rinv, int rows, int SB) {
    if (M <= 0 || N <= 0 || K <= 0) return RTE_OK;
    if (epi == 1 && (!rinv || rows <= 0)) return fail(RTE_ERR_ARG, "epilogue 1 needs its table");
    if (S < 1 || S > 9) return fail(RTE_ERR_ARG, "bad slice count");
    if (SB == 0) SB = S;
    if (SB < S) return fail(RTE_ERR_ARG, "second operand has fewer slices than used");
    const OzArgs g{Aslices, Bslices, ea, eb, M, N, K, SB, C, ldc, epi, rinv, rows};
    switch (S) {
        case 1: return oz_run_width<1, 96, 32, 32>(s, g);
        case 2: return oz_run_width<2, 96, 32, 32>(s, g);
        case 3: return oz_run_width<3, 96, 32, 32>(s, g);
        case 4: return oz_run_width<4, 96, 32, 32>(s, g);
        case 5: return oz_run_width<5, 96, 64, 32>(s, g);
        case 6: return oz_run_width<6, 80, 64, 32>(s, g);
        case 7: return oz_run_width<7, 64, 48, 32>(s, g);
        case 8: return oz_run_width<8, 48, 32, 32>(s, g);
        default: return oz_run_width<9, 32, 32, 32>(s, g);
    }
}

}  // namespace rte
