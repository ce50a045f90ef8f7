// BF16 GEMM on the 5th-generation tensor cores (tcgen05) of sm_103a:
//   C[M x N] (fp32) = A[M x K] (bf16, row-major) * B[N x K]^T (bf16, row-major)
// Both operands are K-major.  One CTA of 128 threads computes a 128 x NT tile
// with an fp32 accumulator of NT columns in TMEM (tcgen05.mma, M = 128, N = NT,
// K = 16 per instruction); the operand tiles arrive by TMA through a ring of
// shared-memory stages; the 4 warps read their 32 TMEM lanes (rows) with
// tcgen05.ld for the epilogue.  Every wait is bounded; on a timeout the kernel
// records it in the status word, frees its TMEM and leaves.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "mpm_internal.cuh"

namespace mpm {

constexpr int kUmmaM = 128;
constexpr int kUmmaKC = 64;                       // K per staged chunk
constexpr int kUmmaThreads = 128;

__device__ __forceinline__ uint32_t umma_smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}


// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator, bf16 A and
// B, both K-major, shape M x N.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4)                  // D format: f32
           | (1u << 7)                // A format: bf16
           | (1u << 10)               // B format: bf16
           | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}


// Pipeline: the operand tiles are brought in by TMA (cp.async.bulk.tensor,
// 128-byte swizzle: a K-chunk of 64 bf16 is one 128-byte swizzle row per M/N
// row) through a ring of shared-memory stages.  Thread 0 produces
// (waits for a free stage, arms its mbarrier with the byte count, issues the
// two tile loads); thread 32 consumes (waits for a full stage, issues the four
// K = 16 MMAs, commits them to the stage's "empty" mbarrier so the producer can
// refill it).  A final commit signals the epilogue, which reads TMEM and either
// stores C or applies bias + GELU (bf16 copy for the next layer) or bias +
// scaled sigmoid.  All waits are bounded.
// Tile choice (umma_gemm_tma): 128 x 256 tiles when they alone fill every SM (half the
// operand traffic per FLOP), else 128 x 128, and narrower ones where 128 x 128 would
// leave most SMs idle.
#ifndef MPM_UMMA_STAGES
#define MPM_UMMA_STAGES 4
#endif
#ifndef MPM_UMMA_WIDE_STAGES
#define MPM_UMMA_WIDE_STAGES 4
#endif
enum UmmaEpilogue {
    kEpiStore = 0, kEpiBiasGelu = 1, kEpiBiasSigmoid = 2, kEpiBiasRelu = 3, kEpiBiasLinear = 4,
    kEpiGeluBack = 5, kEpiReluBack = 6
};

struct UmmaEpi {
    int mode = kEpiStore;
    const float *bias = nullptr;      // N
    // kEpiBiasGelu / kEpiBiasRelu: bf16 GELU(z) / max(z, 0), ld = ldc; kEpiGeluBack /
    // kEpiReluBack: the stored value in bf16.  xnextT: its transpose (N x M) when set.
    __nv_bfloat16 *xnext = nullptr, *xnextT = nullptr;
    float *y = nullptr;               // kEpiBiasSigmoid: lo + (hi - lo) sigmoid(z); kEpiBiasLinear: z; ld = ldc
    const float *zprev = nullptr;     // kEpiGeluBack / kEpiReluBack: C = acc GELU'(zprev) / acc [zprev > 0], ld = ldc
    float lo = 0.f, hi = 1.f;
};

// One GEMM of a launch: operands, output and its number of tiles (M fastest).
struct alignas(64) UmmaJob {
    CUtensorMap tmA, tmB;
    float *C;
    int M, N, K, ldc, tiles_m, tiles;
    UmmaEpi epi;
};
// Up to two independent GEMMs in one launch: a small product fills a fraction of the
// SMs, and the two of a network layer's backward pass need nothing from each other.
struct UmmaJobs {
    UmmaJob j[2];
};

// Shared-memory descriptor of a K-major tile written by TMA with 128-byte
// swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte
// offset), layout type SWIZZLE_128B.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                      // leading byte offset (unused within a swizzle row)
    d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset: 8 rows x 128 bytes
    d |= (uint64_t)1 << 46;                      // version
    d |= (uint64_t)2 << 61;                      // layout: 128-byte swizzle
    return d;
}

__device__ __forceinline__ bool umma_wait_parity(uint64_t *bar, uint32_t parity)
{
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok)
                     : "r"(umma_smem_u32(bar)), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ float umma_gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

__device__ __forceinline__ float umma_gelu_grad(float z)
{
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Eight consecutive fp32 values (16-byte aligned when whole; else the first `left`).
__device__ __forceinline__ void umma_row8(const float *src, bool whole, int left, float v[8])
{
    if (whole) {
        const float4 a = reinterpret_cast<const float4 *>(src)[0], b = reinterpret_cast<const float4 *>(src)[1];
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        return;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = e < left ? src[e] : 0.f;
}

// Epilogue of one 8-column chunk of a row (this lane's): C and the fused outputs, in
// 16-byte accesses where the chunk is whole and C's rows are 16-byte aligned.
__device__ __forceinline__ void umma_store8(const uint32_t r[8], int row, int M, int col0, int N, float *Cout, int ldc,
                                            const UmmaEpi &epi)
{
    const int64_t o0 = (int64_t)row * ldc + col0;
    const bool whole = col0 + 8 <= N && (ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(Cout) & 15) == 0;
    float z[8], x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) z[e] = __uint_as_float(r[e]);
    if (epi.mode == kEpiGeluBack || epi.mode == kEpiReluBack) {
        float zv[8];
        umma_row8(epi.zprev + o0, whole, N - col0, zv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float zp = zv[e];
            z[e] = epi.mode == kEpiReluBack ? (zp > 0.0f ? z[e] : 0.0f) : z[e] * umma_gelu_grad(zp);
            x[e] = z[e];
        }
    } else if (epi.mode != kEpiStore) {
        float bv[8];
        umma_row8(epi.bias + col0, whole, N - col0, bv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            z[e] += bv[e];
            x[e] = epi.mode == kEpiBiasGelu      ? umma_gelu(z[e])
                   : epi.mode == kEpiBiasRelu    ? fmaxf(z[e], 0.0f)
                   : epi.mode == kEpiBiasSigmoid ? epi.lo + (epi.hi - epi.lo) / (1.0f + expf(-z[e]))
                                                 : z[e];
        }
    }
    if (whole) {
        float4 *d = reinterpret_cast<float4 *>(Cout + o0);
        d[0] = make_float4(z[0], z[1], z[2], z[3]);
        d[1] = make_float4(z[4], z[5], z[6], z[7]);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (col0 + e < N) Cout[o0 + e] = z[e];
    }
    if (epi.mode == kEpiStore) return;
    if (epi.y != nullptr) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (col0 + e < N) epi.y[o0 + e] = x[e];
    }
    if (epi.xnext != nullptr) {
        __align__(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) h[e] = __float2bfloat16_rn(x[e]);
        if (whole && (ldc & 7) == 0) {
            *reinterpret_cast<uint4 *>(epi.xnext + o0) = *reinterpret_cast<const uint4 *>(h);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (col0 + e < N) epi.xnext[o0 + e] = h[e];
        }
        if (epi.xnextT != nullptr) {                 // 32 lanes: 32 consecutive rows of one column
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (col0 + e < N) epi.xnextT[(int64_t)(col0 + e) * M + row] = h[e];
        }
    }
}

// 16 accumulator columns of this warp's 32 TMEM lanes, without waiting for them.
__device__ __forceinline__ void umma_ld16(uint32_t taddr, uint32_t r[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void umma_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

template <int NT, int STAGES>
__global__ void __launch_bounds__(kUmmaThreads, 1)
    k_umma_gemm_tma(const __grid_constant__ UmmaJobs jobs, int32_t *__restrict__ status)
{
    static_assert(NT % 16 == 0 && NT >= 32 && NT <= 256, "tile width");
    constexpr int TMEM_COLS = NT <= 32 ? 32 : (NT <= 64 ? 64 : (NT <= 128 ? 128 : 256));
    constexpr uint32_t A_BYTES = kUmmaM * kUmmaKC * 2, B_BYTES = NT * kUmmaKC * 2;
    constexpr uint32_t STAGE = A_BYTES + B_BYTES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *sbase = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                             ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int second = (int)blockIdx.x >= jobs.j[0].tiles ? 1 : 0;
    const UmmaJob &jb = jobs.j[second];
    const int tile = (int)blockIdx.x - (second ? jobs.j[0].tiles : 0);
    const int M = jb.M, N = jb.N;
    const int m0 = tile % jb.tiles_m * kUmmaM, n0 = tile / jb.tiles_m * NT;
    const int nk = (jb.K + kUmmaKC - 1) / kUmmaKC;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         umma_smem_u32(&tmem_base)),
                     "r"((uint32_t)TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        failed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    pdl_enter();

    if (tid == 0) {                                        // producer
        for (int kc = 0; kc < nk; ++kc) {
            const int s = kc % STAGES;
            const uint32_t ph = (uint32_t)(kc / STAGES) & 1u;
            if (!umma_wait_parity(&empty[s], ph ^ 1u)) {
                failed = 1;
                break;
            }
            const uint32_t sa = umma_smem_u32(sbase + s * STAGE), sb = sa + A_BYTES;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(umma_smem_u32(&full[s])),
                         "r"(STAGE)
                         : "memory");
            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                         " [%0], [%1, {%2, %3}], [%4];" ::"r"(sa),
                         "l"(reinterpret_cast<uint64_t>(&jb.tmA)), "r"(kc * kUmmaKC), "r"(m0),
                         "r"(umma_smem_u32(&full[s]))
                         : "memory");
            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                         " [%0], [%1, {%2, %3}], [%4];" ::"r"(sb),
                         "l"(reinterpret_cast<uint64_t>(&jb.tmB)), "r"(kc * kUmmaKC), "r"(n0),
                         "r"(umma_smem_u32(&full[s]))
                         : "memory");
        }
    } else if (tid == 32) {                                // MMA issuer
        const uint32_t idesc = umma_idesc_bf16(kUmmaM, NT);
        bool ok = true;
        for (int kc = 0; kc < nk; ++kc) {
            const int s = kc % STAGES;
            const uint32_t ph = (uint32_t)(kc / STAGES) & 1u;
            if (!umma_wait_parity(&full[s], ph)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa = umma_smem_u32(sbase + s * STAGE), sb = sa + A_BYTES;
#pragma unroll
            for (int kk = 0; kk < kUmmaKC / 16; ++kk) {
                const uint64_t da = umma_desc_sw128(sa + kk * 32), db = umma_desc_sw128(sb + kk * 32);
                const uint32_t acc = (kc > 0 || kk > 0) ? 1u : 0u;
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                             "l"(da), "l"(db), "r"(idesc), "r"(acc)
                             : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             umma_smem_u32(&empty[s]))
                         : "memory");
        }
        if (!ok) failed = 1;
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         umma_smem_u32(&done))
                     : "memory");
    }
    __syncwarp();
    const bool fin = umma_wait_parity(&done, 0u);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool ok = __syncthreads_and(fin) && !failed;
    if (ok) {
        const int row = m0 + warp * 32 + lane;
        const UmmaEpi epi = jb.epi;
        for (int c0 = 0; c0 < NT && n0 + c0 < N; c0 += 16) {
            uint32_t r[16];
            umma_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
            umma_wait_ld();
            if (row < M) {
                umma_store8(r, row, M, n0 + c0, N, jb.C, jb.ldc, epi);
                if (n0 + c0 + 8 < N) umma_store8(r + 8, row, M, n0 + c0 + 8, N, jb.C, jb.ldc, epi);
            }
        }
    } else if (tid == 0) {
        atomicOr(status, (int32_t)kStatusTimeout);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)TMEM_COLS)
                     : "memory");
}

// Persistent, warp-specialised form for large problems: one CTA per SM walks the
// 128 x 256 tiles (M fastest within bands of 8 N-tiles, so that consecutive
// tiles of the SMs share their B tiles in L2).  Warp 0 produces (TMA into the
// ring of stages), warp 1 issues the MMAs, warps 2-5 run the epilogue; the fp32
// accumulator is double-buffered in TMEM (2 x 256 of the 512 columns), so the
// epilogue of one tile overlaps the main loop of the next.  Every wait is
// bounded; a timeout sets the status word and every role leaves.  The tiles of a last,
// partial wave are cut into `split` tiles of 256 / split columns where those still fit one
// wave, so that it takes half or a quarter of a full one (8192 x 2048 x 2048: 512 tiles
// on 152 SMs, 56 in the fourth wave: 61.2 us, 59.1 so).
constexpr int kUmmaPersistThreads = 192;
template <int STAGES>
__global__ void __launch_bounds__(kUmmaPersistThreads, 1)
    k_umma_gemm_persist(int M, int N, int K, const __grid_constant__ CUtensorMap tmA,
                        const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmBs, int n_full,
                        int split, float *__restrict__ Cout, int ldc, UmmaEpi epi, int32_t *__restrict__ status)
{
    constexpr int NT = 256;
    constexpr uint32_t A_BYTES = kUmmaM * kUmmaKC * 2, B_BYTES = NT * kUmmaKC * 2;
    constexpr uint32_t STAGE = A_BYTES + B_BYTES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *sbase = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                             ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], acc_full[2], acc_empty[2], done;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nk = (K + kUmmaKC - 1) / kUmmaKC;
    const int tm = (M + kUmmaM - 1) / kUmmaM, tn = (N + NT - 1) / NT;
    // work units: n_full tiles, then the remaining tiles in split parts each
    const int n_units = n_full + (tm * tn - n_full) * split;
    constexpr int BAND = 8;                              // N-tiles per band
    auto tile_coords = [&](int u, int &m0, int &n0, int &width) {
        const int v = u - n_full, t = v < 0 ? u : n_full + v / split;
        width = v < 0 ? NT : NT / split;
        const int band = t / (BAND * tm);
        const int r = t - band * BAND * tm;
        const int bw = min(BAND, tn - band * BAND);
        m0 = (r / bw) * kUmmaM;
        n0 = (band * BAND + r % bw) * NT + (v < 0 ? 0 : v % split * width);
    };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         umma_smem_u32(&tmem_base)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&empty[s])) : "memory");
        }
        for (int b = 0; b < 2; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&acc_full[b])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(umma_smem_u32(&acc_empty[b])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(umma_smem_u32(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        failed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    pdl_enter();

    if (warp == 0) {                                     // producer
        if (lane == 0) {
            int it = 0;
            for (int t = blockIdx.x; t < n_units && !failed; t += gridDim.x) {
                int m0, n0, width;
                tile_coords(t, m0, n0, width);
                const CUtensorMap *mapB = width == NT ? &tmB : &tmBs;
                for (int kc = 0; kc < nk; ++kc, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                    if (!umma_wait_parity(&empty[s], ph ^ 1u)) {
                        failed = 1;
                        break;
                    }
                    const uint32_t sa = umma_smem_u32(sbase + s * STAGE), sb = sa + A_BYTES;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                                     umma_smem_u32(&full[s])),
                                 "r"(A_BYTES + (uint32_t)width * kUmmaKC * 2)
                                 : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                                 " [%0], [%1, {%2, %3}], [%4];" ::"r"(sa),
                                 "l"(reinterpret_cast<uint64_t>(&tmA)), "r"(kc * kUmmaKC), "r"(m0),
                                 "r"(umma_smem_u32(&full[s]))
                                 : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                                 " [%0], [%1, {%2, %3}], [%4];" ::"r"(sb),
                                 "l"(reinterpret_cast<uint64_t>(mapB)), "r"(kc * kUmmaKC), "r"(n0),
                                 "r"(umma_smem_u32(&full[s]))
                                 : "memory");
                }
            }
        }
    } else if (warp == 1) {                              // MMA issuer
        if (lane == 0) {
            int it = 0, lt = 0;
            for (int t = blockIdx.x; t < n_units && !failed; t += gridDim.x, ++lt) {
                const int b = lt & 1;
                if (!umma_wait_parity(&acc_empty[b], ((uint32_t)(lt >> 1) & 1u) ^ 1u)) {
                    failed = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc_addr = tmem + (uint32_t)(b * NT);
                const uint32_t idesc = umma_idesc_bf16(kUmmaM, t < n_full ? NT : NT / split);
                bool ok = true;
                for (int kc = 0; kc < nk; ++kc, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
                    if (!umma_wait_parity(&full[s], ph)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = umma_smem_u32(sbase + s * STAGE), sb = sa + A_BYTES;
#pragma unroll
                    for (int kk = 0; kk < kUmmaKC / 16; ++kk) {
                        const uint64_t da = umma_desc_sw128(sa + kk * 32), db = umma_desc_sw128(sb + kk * 32);
                        const uint32_t acc = (kc > 0 || kk > 0) ? 1u : 0u;
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_addr),
                                     "l"(da), "l"(db), "r"(idesc), "r"(acc)
                                     : "memory");
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     umma_smem_u32(&empty[s]))
                                 : "memory");
                }
                if (!ok) {
                    failed = 1;
                    break;
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 umma_smem_u32(&acc_full[b]))
                             : "memory");
            }
            // every MMA this thread issued has completed before TMEM is released
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             umma_smem_u32(&done))
                         : "memory");
            if (!umma_wait_parity(&done, 0u)) failed = 1;
        }
    } else {                                             // epilogue: warps 2-5, TMEM lane quarter warp % 4
        const int q = warp & 3;
        int lt = 0;
        for (int t = blockIdx.x; t < n_units; t += gridDim.x, ++lt) {
            const int b = lt & 1;
            bool ok = false;
            if (lane == 0) ok = umma_wait_parity(&acc_full[b], (uint32_t)(lt >> 1) & 1u);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) {
                if (lane == 0) failed = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            int m0, n0, width;
            tile_coords(t, m0, n0, width);
            const int row = m0 + q * 32 + lane;
            for (int c0 = 0; c0 < width; c0 += 8) {
                uint32_t r[8];
                const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * NT + c0);
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                               "=r"(r[6]), "=r"(r[7])
                             : "r"(taddr)
                             : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (row < M && n0 + c0 < N) umma_store8(r, row, M, n0 + c0, N, Cout, ldc, epi);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)                               // this quarter of the accumulator is free again
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(umma_smem_u32(&acc_empty[b]))
                             : "memory");
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (failed && tid == 0) atomicOr(status, (int32_t)kStatusTimeout);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

template <int NT, int STAGES> constexpr size_t umma_tma_smem_bytes()
{
    return (size_t)STAGES * (kUmmaM + NT) * kUmmaKC * 2 + 1024;
}

// 2D tensor map of a row-major bf16 matrix (rows x cols, leading dimension ld
// elements) for boxes of box_rows x 64 with 128-byte swizzle.
inline bool umma_tensor_map(CUtensorMap *tm, const __nv_bfloat16 *ptr, int rows, int cols, int ld, int box_rows)
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kUmmaKC, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(ptr), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline int umma_num_sms()
{
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    }
    return sms;
}

// Tiles of 128 x nt of an M x N product.
inline int64_t umma_tiles(int M, int N, int nt)
{
    return (int64_t)((M + kUmmaM - 1) / kUmmaM) * ((N + nt - 1) / nt);
}

// Whether the 128 x 256 tiles of a product alone fill every SM: the persistent kernel's range.
inline bool umma_wide(int M, int N, int sms) { return N >= 256 && umma_tiles(M, N, 256) >= sms; }

// One GEMM C = A B^T of umma_gemm_tiles.
struct UmmaGemm {
    int M, N, K;
    const __nv_bfloat16 *A;
    int lda;
    const __nv_bfloat16 *B;
    int ldb;
    float *C;
    int ldc;
    UmmaEpi epi;
};

template <int NT, int STAGES>
inline cudaError_t umma_launch(const UmmaGemm *g, int n, int32_t *status, cudaStream_t stream)
{
    constexpr size_t smem = umma_tma_smem_bytes<NT, STAGES>();
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(k_umma_gemm_tma<NT, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        attr = true;
    }
    UmmaJobs jobs;
    int blocks = 0;
    for (int i = 0; i < n; ++i) {
        UmmaJob &j = jobs.j[i];
        if (!umma_tensor_map(&j.tmA, g[i].A, g[i].M, g[i].K, g[i].lda, kUmmaM) ||
            !umma_tensor_map(&j.tmB, g[i].B, g[i].N, g[i].K, g[i].ldb, NT))
            return cudaErrorInvalidValue;
        j.C = g[i].C;
        j.M = g[i].M;
        j.N = g[i].N;
        j.K = g[i].K;
        j.ldc = g[i].ldc;
        j.epi = g[i].epi;
        j.tiles_m = (j.M + kUmmaM - 1) / kUmmaM;
        j.tiles = j.tiles_m * ((j.N + NT - 1) / NT);
        blocks += j.tiles;
    }
    if (n == 1) jobs.j[1] = jobs.j[0];
    launch_after(k_umma_gemm_tma<NT, STAGES>, blocks, kUmmaThreads, smem, stream, jobs, status);
    return cudaGetLastError();
}

// One or two GEMMs in tiles of the width that suits them: 32 or 64 columns where 128
// would leave at least three quarters or half of the SMs without a tile (a tile's
// epilogue, erff on every value, and its operand stream are then spread over more
// SMs; the deeper ring covers the L2 latency of the short tiles: one row through
// 640-256-256-32 with its copies 84 -> 60 us, its first GEMM alone was 17 us on two SMs).
// Up to 32 columns in more tiles than SMs: a ring of 4 stages, so that two CTAs share an SM
// and one's loads run under the other's start and epilogue (us with 8 | 4 stages, N = 24:
// 153 tiles, K = 640: 11.96 | 7.05, 512 tiles: 26.30 | 19.28, K = 2048: 55.84 | 47.22;
// 152 tiles, one wave: K = 640: 7.36 | 7.15, K = 2048: 16.47 | 17.18).
inline cudaError_t umma_gemm_tiles(const UmmaGemm *g, int n, int32_t *status, cudaStream_t stream)
{
    int64_t tiles = 0;
    int widest = 0;
    for (int i = 0; i < n; ++i) {
        tiles += umma_tiles(g[i].M, g[i].N, 128);
        widest = g[i].N > widest ? g[i].N : widest;
    }
    const int sms = umma_num_sms();
    if (widest <= 32 && tiles > sms) return umma_launch<32, 4>(g, n, status, stream);
    if (widest <= 32 || 4 * tiles <= sms) return umma_launch<32, 8>(g, n, status, stream);
    if (2 * tiles <= sms) return umma_launch<64, 8>(g, n, status, stream);
    return umma_launch<128, MPM_UMMA_STAGES>(g, n, status, stream);
}

// C = A B^T through the pipelined TMA kernels, with an optional fused epilogue.
inline cudaError_t umma_gemm_tma(int M, int N, int K, const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B,
                                 int ldb, float *C, int ldc, const UmmaEpi &epi, int32_t *status, cudaStream_t stream)
{
    const int sms = umma_num_sms();
    if (umma_wide(M, N, sms)) {
        CUtensorMap tmA, tmB;
        if (!umma_tensor_map(&tmA, A, M, K, lda, kUmmaM) || !umma_tensor_map(&tmB, B, N, K, ldb, 256))
            return cudaErrorInvalidValue;
        constexpr size_t smem = umma_tma_smem_bytes<256, MPM_UMMA_WIDE_STAGES>();
        static bool attr = false;
        if (!attr) {
            cudaFuncSetAttribute(k_umma_gemm_persist<MPM_UMMA_WIDE_STAGES>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            attr = true;
        }
        const int tiles = ((M + kUmmaM - 1) / kUmmaM) * ((N + 255) / 256);
        const int rest = tiles % sms;                  // tiles of the last, partial wave
        const int split = rest == 0 ? 1 : 4 * rest <= sms ? 4 : 2 * rest <= sms ? 2 : 1;
        CUtensorMap tmBs = tmB;
        if (split > 1 && !umma_tensor_map(&tmBs, B, N, K, ldb, 256 / split)) return cudaErrorInvalidValue;
        launch_after(k_umma_gemm_persist<MPM_UMMA_WIDE_STAGES>, std::min(sms, tiles), kUmmaPersistThreads, smem, stream,
                     M, N, K, tmA, tmB, tmBs, split > 1 ? tiles - rest : tiles, split, C, ldc, epi, status);
        return cudaGetLastError();
    }
    const UmmaGemm g{M, N, K, A, lda, B, ldb, C, ldc, epi};
    return umma_gemm_tiles(&g, 1, status, stream);
}

// Whether two products share a launch of narrow tiles, or go one after the other so that
// a wide one (umma_wide) takes the persistent kernel.  They share it where neither is wide,
// and where the narrow one has tiles for less than a quarter of the SMs that take longer
// than twice the wide one, by K-chunks of a CTA with 16 for a wide tile's epilogue: the
// weight gradient of a small layer contracts over a large batch (256 x 256 over 65,536 rows:
// 292 us on 16 SMs) and costs nothing beside the other product.  Two training steps, one
// launch | one after the other: 4096-4096-4096-4096 at batch 4096 4.50 | 3.61 ms, 640-4096-32
// at 19,456 3.62 | 3.35, 8192-8192-8192 at 512 3.67 | 3.42, 768-768-768-768 at 16,384
// 2.80 | 2.89, 640-256-256-32 at 65,536 4.42 | 4.76.
inline bool umma_share_launch(const UmmaGemm &a, const UmmaGemm &b, int sms)
{
    const bool wa = umma_wide(a.M, a.N, sms), wb = umma_wide(b.M, b.N, sms);
    if (!wa && !wb) return true;
    if (wa && wb) return false;
    const UmmaGemm &w = wa ? a : b, &n = wa ? b : a;
    const int64_t waves = (umma_tiles(w.M, w.N, 256) + sms - 1) / sms;
    return 4 * umma_tiles(n.M, n.N, 128) <= sms && n.K / kUmmaKC >= 2 * waves * (w.K / kUmmaKC + 16);
}

// One or two independent GEMMs.
inline cudaError_t umma_gemms(const UmmaGemm *g, int n, int32_t *status, cudaStream_t stream)
{
    if (n == 2 && umma_share_launch(g[0], g[1], umma_num_sms())) return umma_gemm_tiles(g, 2, status, stream);
    for (int i = 0; i < n; ++i) {
        const cudaError_t e = umma_gemm_tma(g[i].M, g[i].N, g[i].K, g[i].A, g[i].lda, g[i].B, g[i].ldb, g[i].C,
                                            g[i].ldc, g[i].epi, status, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace mpm
