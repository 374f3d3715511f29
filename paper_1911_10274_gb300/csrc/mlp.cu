// mlp.cu -- a small fitness-surrogate MLP trained and run on the 5th-generation
// tensor cores (tcgen05) with BF16 operands and FP32 accumulation.
//
// The surrogate predicts a robot's 1 s centroid displacement from its voxel
// occupancy and per-voxel actuation phases; it pre-screens mutants in a
// morphology search whose survivors the simulator then scores (the paper's
// Sec. III-F topology and actuation optimisation, with a learned filter).
// Network: in -> hidden -> hidden -> hidden -> 1, GELU after each hidden layer.
//
// GEMM kernel (k_gemm_tn): C[M, N] = A[M, K] * B[N, K]^T with A and B row-major
// BF16 (K contiguous; either operand may also be stored with K as its slow
// dimension, which is how back-propagation multiplies by transposes).  One CTA
// per 128 x BN output tile (BN = 64, 128 or 256), 512 threads:
//   warp 0         - TMA producer: 2-D tiled loads (128-byte swizzle) of the
//                    A and B K-blocks (64 wide) into a ring of 3 or 4 stages;
//   warp 1         - MMA issuer: tcgen05.mma.kind::f16 (M = 128, N = BN,
//                    K = 16) into an FP32 accumulator in TMEM, releasing each
//                    stage with tcgen05.commit;
//   all 16 warps   - epilogue, a row per lane: FP32 output, fused bias + GELU,
//                    or the GELU-derivative product of back-propagation with
//                    its bias-gradient column sums.
// Every mbarrier wait is bounded (spin_limit polls); on expiry the kernel sets
// *err, waits (bounded) for its own copies and products in flight, skips the
// epilogue, frees its TMEM and returns.  No CTA leaves, after an expired wait or
// not, before every copy and every commit that targets it has landed (gemm_ring.h).
//
// Training step: nine launches on one stream, each a programmatic dependent of
// the one before: a copy of the batch, three forward products, the head (output
// layer, loss, first step back), two input gradients, the three weight gradients,
// and Adam (which adds the K slices and column sums up itself).  The learning rate
// and the Adam step counter live in device memory.  Large products of a caller's own
// (titan_gemm_bf16_tn) go to persistent CTA pairs, k_gemm_pair, where gemm_rule.h says.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <random>
#include <string>
#include <vector>

#include "gemm_ring.h"
#include "gemm_rule.h"
#include "mlp_layout.h"
#include "ptx.cuh"
#include "titan.h"

namespace titan {
void set_thread_error(const std::string &msg);   // runtime.cu
}

namespace {

// BM x BN output tile per CTA; BN = 64, 128 or 256 (wide tiles for large
// products: each A tile then feeds twice the columns, halving the A traffic
// from L2 per FLOP).
constexpr int BM = 128, BN = 128, BK = 64;
// 16 warps: warps 0 and 1 issue the loads and the products; after the
// mainloop all 16 run the epilogue, warp w on TMEM lanes 32 (w mod 4) ..
// + 31 (the lanes its quarter may read) and on quarter w / 4 of the columns,
// 16 at a time (the GELU's arithmetic needs the warps: with 8, each epilogue
// waited on its own instructions)
constexpr int kGemmThreads = 512;
constexpr uint32_t kStageA = BM * BK * 2;
template <int BN_> constexpr uint32_t stage_b() { return (uint32_t)BN_ * BK * 2; }
// Ring stages and resident CTAs per SM: two CTAs of the 64- and 128-wide tiles share
// an SM (97 KB each), so that one's epilogue runs beside the other's products.
template <int BN_> constexpr int stages() { return BN_ == 128 ? 3 : 4; }
template <int BN_> constexpr int resident() { return BN_ == 256 ? 1 : 2; }
template <int BN_> constexpr size_t gemm_smem() { return (size_t)stages<BN_>() * (kStageA + stage_b<BN_>()) + 1024; }

// Polls of a wait for what is already under way and completes by itself.
constexpr uint32_t kDrainPolls = 1u << 22;

enum Epi { EPI_F32 = 0, EPI_BIAS_GELU = 1, EPI_GELU_GRAD = 2 };

struct EpiArgs {
    int mode;
    int ldc;                      // row stride of the outputs (elements)
    const float *bias;            // [N]            (BIAS_GELU)
    float *out_f32;               // [M, ldc]       (F32: C; BIAS_GELU: pre-activation Z, if wanted)
    __nv_bfloat16 *out_bf16;      // [M, ldc]       (BIAS_GELU: GELU(Z); GELU_GRAD: dZ)
    const float *z;               // [M, ldc]       (GELU_GRAD: the forward pre-activation)
    float *colsum = nullptr;      // [M / 32, ldc] GELU_GRAD: per 32 rows, the column sums of out_bf16
};

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Instruction descriptor of tcgen05.mma.kind::f16: FP32 accumulator, BF16 A
// and B, each K-major or (MN) with K as the slow dimension, N = BN_, M = BM.
template <int BN_, bool AMN, bool BMN>
constexpr uint32_t idesc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((AMN ? 1u : 0u) << 15) | ((BMN ? 1u : 0u) << 16) |
           ((uint32_t)(BN_ >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// 16 consecutive values of one row (one lane of an epilogue warp) as whole
// 32-byte sectors; the row start is 32-byte aligned.
__device__ __forceinline__ void store_row16(float *o, const float *v) {
#pragma unroll
    for (int x = 0; x < 16; x += 8)
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o + x), "f"(v[x]), "f"(v[x + 1]),
                     "f"(v[x + 2]), "f"(v[x + 3]), "f"(v[x + 4]), "f"(v[x + 5]), "f"(v[x + 6]), "f"(v[x + 7])
                     : "memory");
}
__device__ __forceinline__ void store_row16(__nv_bfloat16 *o, const uint32_t *v) {      // 8 pairs
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
// Through L2: the row was written by an earlier kernel of the same chain.
__device__ __forceinline__ void load_row16(const float *o, float *v) {
#pragma unroll
    for (int x = 0; x < 16; x += 8)
        asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[x]), "=f"(v[x + 1]), "=f"(v[x + 2]), "=f"(v[x + 3]), "=f"(v[x + 4]), "=f"(v[x + 5]),
                       "=f"(v[x + 6]), "=f"(v[x + 7])
                     : "l"(o + x)
                     : "memory");
}
__device__ __forceinline__ uint32_t bf16_bits(__nv_bfloat16 lo, __nv_bfloat16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// One 128 x BN_ tile of C = A B^T over num_kb k-blocks from k0: the whole CTA.
// AMN / BMN: the operand is stored with K as its slow dimension (A[K][M],
// B[K][N]); its tiles are staged as 64 x 64 boxes, one per 64 rows of the tile
// (8 KB each, rows of K 128 bytes apart), which the tensor cores read directly:
// back-propagation multiplies by transposes that are never formed.
// zoff: offset of this tile's block of out_f32 (split K).
//
// The accumulator leaves TMEM one row per lane, 16 columns at a time, and every
// global access of the epilogue is a lane's own whole 32-byte sectors (3 stores a
// row of 16 instead of one per column through shared memory; no staging but for the
// column sums).
template <int BN_, bool AMN, bool BMN>
__device__ __forceinline__ void gemm_tile(const CUtensorMap *tma_a, const CUtensorMap *tma_b, int m0, int n0, int k0,
                                          int num_kb, const EpiArgs &ep, size_t zoff, uint32_t spin_limit, int *err) {
    constexpr int STAGES = stages<BN_>();
    extern __shared__ uint8_t gsm_raw[];
    __shared__ uint64_t full[STAGES], empty[STAGES], accf;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    __shared__ int n_issued, n_mma;                   // k-blocks whose loads, whose products were issued
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // known to be the same in every lane
    titan::ptx::grid_dep_launch();                    // the next kernel's prologue may overlap this one
    // 1024-byte aligned tiles (the 128-byte swizzle pattern repeats every 1024 bytes)
    const uint32_t raw = titan::ptx::smem_u32(gsm_raw);
    uint8_t *gsm = gsm_raw + (((raw + 1023u) & ~1023u) - raw);
    constexpr uint32_t kStageB = stage_b<BN_>();
    constexpr uint32_t kTmemCols = (uint32_t)BN_;      // one FP32 column per output column
    constexpr uint32_t kBox = 64 * 128;                // bytes of a 64 x 64 box
    auto tileA = [&](int s) { return gsm + (size_t)s * (kStageA + kStageB); };
    auto tileB = [&](int s) { return gsm + (size_t)s * (kStageA + kStageB) + kStageA; };

    if (warp == 0) titan::ptx::tmem_alloc(&tmem_base, kTmemCols);
    if (tid == 32) {
        for (int s = 0; s < STAGES; ++s) {
            titan::ptx::mbar_init(&full[s], 1);
            titan::ptx::mbar_init(&empty[s], 1);
        }
        titan::ptx::mbar_init(&accf, 1);
        titan::ptx::fence_mbar_init();
        failed = 0;
        n_issued = n_mma = 0;
    }
    titan::ptx::tc_fence_before();
    __syncthreads();
    titan::ptx::tc_fence_after();
    const uint32_t taddr = tmem_base;
    if (tid == 0) {
        titan::ptx::prefetch_tensormap(tma_a);
        titan::ptx::prefetch_tensormap(tma_b);
    }
    titan::ptx::grid_dep_wait();                      // the operands are in place

    // Both issuing warps run their loops whole, on values the same in every lane, and
    // one elected lane issues: loops of a single lane moved every descriptor, address
    // and barrier through vector registers and were the bound themselves (528 cycles a
    // k-block, whatever the tile).
    if (warp == 0) {                                   // TMA producer
        const bool leader = titan::ptx::elect_one();
        uint32_t s = 0, parity = 1;
        int issued = 0;
        for (int kb = 0, k = k0; kb < num_kb; ++kb, k += BK) {
            if (kb >= STAGES && !titan::ptx::mbar_wait_warp(&empty[s], parity, spin_limit)) {
                if (leader) atomicExch(&failed, 1);
                break;
            }
            if (leader) {
                titan::ptx::mbar_arrive_expect_tx(&full[s], kStageA + kStageB);
                if (AMN) {
#pragma unroll
                    for (int j = 0; j < BM / 64; ++j)
                        titan::ptx::tma_load_2d(tileA(s) + j * kBox, tma_a, m0 + 64 * j, k, &full[s]);
                } else {
                    titan::ptx::tma_load_2d(tileA(s), tma_a, k, m0, &full[s]);
                }
                if (BMN) {
#pragma unroll
                    for (int j = 0; j < BN_ / 64; ++j)
                        titan::ptx::tma_load_2d(tileB(s) + j * kBox, tma_b, n0 + 64 * j, k, &full[s]);
                } else {
                    titan::ptx::tma_load_2d(tileB(s), tma_b, k, n0, &full[s]);
                }
            }
            __syncwarp();
            issued = kb + 1;
            if (++s == STAGES) {
                s = 0;
                parity ^= 1;
            }
        }
        if (leader) n_issued = issued;
    } else if (warp == 1) {                            // MMA issuer
        const bool leader = titan::ptx::elect_one();
        // the descriptors of stage 0, moved by an addition (a stage, or 16 of K, in units of 16 bytes)
        uint64_t a = AMN ? titan::ptx::smem_desc_mn_sw128(titan::ptx::smem_u32(tileA(0)), kBox)
                         : titan::ptx::smem_desc_sw128(titan::ptx::smem_u32(tileA(0)));
        uint64_t b = BMN ? titan::ptx::smem_desc_mn_sw128(titan::ptx::smem_u32(tileB(0)), kBox)
                         : titan::ptx::smem_desc_sw128(titan::ptx::smem_u32(tileB(0)));
        constexpr uint32_t kStep = (kStageA + kStageB) >> 4, kStepA = (AMN ? 2048 : 32) >> 4, kStepB = (BMN ? 2048 : 32) >> 4;
        uint32_t s = 0, parity = 0;
        int kb = 0;
        bool ready = false;                            // this k-block was seen to have arrived
        for (; kb < num_kb; ++kb) {
            if (!ready && !titan::ptx::mbar_wait_warp(&full[s], parity, spin_limit)) {
                if (leader) atomicExch(&failed, 1);
                break;
            }
            titan::ptx::tc_fence_after();
            const uint32_t s1 = s + 1 == STAGES ? 0 : s + 1, parity1 = parity ^ (s1 == 0);
            ready = kb + 1 < num_kb && __all_sync(0xffffffffu, titan::ptx::mbar_test(&full[s1], parity1));
            if (leader) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    titan::ptx::tc_mma_bf16(taddr, a + kStepA * k, b + kStepB * k, idesc<BN_, AMN, BMN>(), (kb | k) != 0);
                titan::ptx::tc_commit(&empty[s]);
            }
            __syncwarp();
            a += s1 ? (int64_t)kStep : (int64_t)kStep - STAGES * (int64_t)kStep;
            b += s1 ? (int64_t)kStep : (int64_t)kStep - STAGES * (int64_t)kStep;
            s = s1;
            parity = parity1;
        }
        if (leader) {
            titan::ptx::tc_commit(&accf);              // fires when every issued MMA is done
            n_mma = kb;
        }
    }
    __syncwarp();
    // epilogue: every thread owns one output row (its TMEM lane); what its first
    // columns need from memory is requested while the products run
    constexpr int W = 16;                              // columns at a time
    const int quarter = (int)(warp & 3), group = (int)(warp >> 2);
    const int row = m0 + quarter * 32 + (int)lane;
    float z[W];
    auto request = [&](int col) {
        if (ep.mode == EPI_GELU_GRAD) {
            load_row16(ep.z + (size_t)row * ep.ldc + col, z);
        } else if (ep.mode == EPI_BIAS_GELU) {
#pragma unroll
            for (int k = 0; k < W; k += 4) {
                const float4 b = __ldcg(reinterpret_cast<const float4 *>(ep.bias + col + k));
                z[k] = b.x;
                z[k + 1] = b.y;
                z[k + 2] = b.z;
                z[k + 3] = b.w;
            }
        }
    };
    request(n0 + group * (BN_ / 4));
    // one warp polls; the others sleep at the barrier.  Beside it the producer waits for the
    // last releases of its ring, which land with the accumulator
    bool acc_ok = true;
    if (warp == 0) {
        if (n_issued == num_kb)
            for (int j = titan::ring_tail(num_kb, STAGES); j < num_kb; ++j)
                if (!titan::ptx::mbar_wait_warp(&empty[titan::ring_slot(j, STAGES)], titan::ring_parity(j, STAGES),
                                                spin_limit)) {
                    atomicExch(&failed, 1);
                    break;
                }
    } else if (warp == 1) {
        acc_ok = titan::ptx::mbar_wait_bounded(&accf, 0, spin_limit);
        if (!acc_ok) atomicExch(&failed, 1);
    }
    __syncthreads();
    titan::ptx::tc_fence_after();
    if (failed) {
        // a bounded wait expired: record it, then wait (bounded again) for
        // this CTA's own copies and products still in flight - the last TMA
        // load issued on each stage and every committed MMA - before the
        // tensor memory is freed and the CTA exits
        if (tid == 32) {
            // a plain store: the flag may live in pinned host memory
            *reinterpret_cast<volatile int *>(err) = 1;
            __threadfence_system();
            for (int j = titan::ring_tail(n_issued, STAGES); j < n_issued; ++j)
                titan::ptx::mbar_wait_bounded(&full[titan::ring_slot(j, STAGES)], titan::ring_parity(j, STAGES), kDrainPolls);
            if (!acc_ok) titan::ptx::mbar_wait_bounded(&accf, 0, kDrainPolls);
            for (int j = titan::ring_tail(n_mma, STAGES); j < n_mma; ++j)
                titan::ptx::mbar_wait_bounded(&empty[titan::ring_slot(j, STAGES)], titan::ring_parity(j, STAGES), kDrainPolls);
        }
        __syncthreads();
    } else {
        const bool sectors = !(reinterpret_cast<uintptr_t>(ep.out_f32) & 31);
        // this warp's scratch in the idle stage buffers, rows 17 (values) or 9 (pairs) words apart
        float *scr = reinterpret_cast<float *>(gsm) + warp * (32 * (W + 1));
#pragma unroll 1
        for (int c0 = group * (BN_ / 4); c0 < (group + 1) * (BN_ / 4); c0 += W) {
            float v[W];
            titan::ptx::tmem_ld16(taddr + (((uint32_t)quarter * 32u) << 16) + (uint32_t)c0, v);
            const int col = n0 + c0;
            const size_t o = (size_t)row * ep.ldc + col;
            if (ep.mode == EPI_F32) {
                if (sectors) {
                    store_row16(ep.out_f32 + zoff + o, v);
                } else {
                    // a caller's C off the 32-byte grid: columns across the lanes, two rows a store
#pragma unroll
                    for (int k = 0; k < W; ++k) scr[lane * (W + 1) + k] = v[k];
                    __syncwarp();
#pragma unroll 8
                    for (int r = (int)lane / W; r < 32; r += 32 / W)
                        ep.out_f32[zoff + (size_t)(m0 + quarter * 32 + r) * ep.ldc + col + lane % W] =
                            scr[r * (W + 1) + lane % W];
                    __syncwarp();
                }
            } else if (ep.mode == EPI_BIAS_GELU) {
#pragma unroll
                for (int k = 0; k < W; ++k) v[k] += z[k];
                if (ep.out_f32) store_row16(ep.out_f32 + o, v);
                uint32_t h[W / 2];
#pragma unroll
                for (int k = 0; k < W / 2; ++k)
                    h[k] = bf16_bits(__float2bfloat16_rn(gelu(v[2 * k])), __float2bfloat16_rn(gelu(v[2 * k + 1])));
                store_row16(ep.out_bf16 + o, h);
            } else {
                uint32_t h[W / 2];
#pragma unroll
                for (int k = 0; k < W / 2; ++k)
                    h[k] = bf16_bits(__float2bfloat16_rn(v[2 * k] * gelu_grad(z[2 * k])),
                                     __float2bfloat16_rn(v[2 * k + 1] * gelu_grad(z[2 * k + 1])));
                store_row16(ep.out_bf16 + o, h);
                // the column sums of the 32 rows, rows in order
                uint32_t *pairs = reinterpret_cast<uint32_t *>(scr);
#pragma unroll
                for (int k = 0; k < W / 2; ++k) pairs[lane * (W / 2 + 1) + k] = h[k];
                __syncwarp();
                float cs = 0.f;
#pragma unroll
                for (int r = 0; r < 32; ++r) {
                    const uint32_t q = pairs[r * (W / 2 + 1) + (lane % W >> 1)];
                    cs += __uint_as_float((lane & 1) ? q & 0xffff0000u : q << 16);
                }
                __syncwarp();
                if (lane < W) ep.colsum[(size_t)((m0 >> 5) + quarter) * ep.ldc + col + lane] = cs;
            }
            if (c0 + W < (group + 1) * (BN_ / 4)) request(col + W);
        }
    }
    titan::ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) titan::ptx::tmem_dealloc(taddr, kTmemCols);
}

// split K (gridDim.z slices): slice z multiplies k-columns [z K, (z + 1) K) of A
// and B and writes its partial product to its own M x ldc block of out_f32.
template <int BN_, bool AMN, bool BMN>
__global__ void __launch_bounds__(kGemmThreads, resident<BN_>())
k_gemm_tn(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b, int K, EpiArgs ep,
          uint32_t spin_limit, int *__restrict__ err) {
    gemm_tile<BN_, AMN, BMN>(&tma_a, &tma_b, (int)blockIdx.y * BM, (int)blockIdx.x * BN_, (int)blockIdx.z * K, K / BK,
                             ep, (size_t)blockIdx.z * gridDim.y * BM * ep.ldc, spin_limit, err);
}

// The three weight gradients of a step in one launch: dW_l^T (hid x in_l) =
// dZ_l^T A_{l-1}, both operands as back-propagation left them, [batch][...], K
// their slow dimension.  Blocks run layer by layer, K slice by K slice, tile by
// tile; a slice's partial product lands in its own block of out[l].
struct WgradArgs {
    CUtensorMap a[3], b[3];
    float *out[3];
    int first[3], tiles[3], tiles_n[3], ld[3], kslice[3];   // first block, tiles a slice, tiles per tile row, in_l
};

__global__ void __launch_bounds__(kGemmThreads, resident<BN>())
k_wgrad(const __grid_constant__ WgradArgs w, int hid, uint32_t spin_limit, int *__restrict__ err) {
    const int t = (int)blockIdx.x;
    const int l = t >= w.first[1] ? (t >= w.first[2] ? 2 : 1) : 0;
    const int z = (t - w.first[l]) / w.tiles[l], in_slice = (t - w.first[l]) % w.tiles[l];
    EpiArgs ep{EPI_F32, w.ld[l], nullptr, w.out[l], nullptr, nullptr};
    gemm_tile<BN, true, true>(&w.a[l], &w.b[l], in_slice / w.tiles_n[l] * BM, in_slice % w.tiles_n[l] * BN,
                               z * w.kslice[l], w.kslice[l] / BK, ep, (size_t)z * hid * w.ld[l], spin_limit, err);
}

// ---- large products: CTA pairs, persistent
//
// C[M, N] = A[M, K] B[N, K]^T in 256 x 256 tiles, one tile at a time per pair of
// CTAs (cta_group::2: each CTA stages its 128 rows of A and 128 of B's 256 rows,
// so a k-block costs 32 KB of shared memory and L2 traffic per CTA where the
// one-CTA 128 x 256 tile costs 48, which bounded that kernel by shared-memory
// bandwidth).  A pair keeps taking tiles; two accumulators of 256 TMEM columns
// let a tile's epilogue run beside the next tile's products.
//   warp 0                 - TMA producer of this CTA's halves (6-stage ring)
//   warp 1, leading CTA    - MMA issuer for the pair
//   warps 4 .. 7           - epilogue: TMEM lanes 32 (w - 4) .. + 31 of this CTA's 128 rows
// Barriers: full[s] lives in the leader (both CTAs' bytes), empty[s] and
// acc_full[b] in each CTA (multicast commits), acc_empty[b] in the leader (one
// arrival per epilogue warp of both CTAs).  Every wait is bounded; after one
// expires a CTA records it and stops.  Then the CTAs tell each other how far they
// came and wait, bounded, for whatever of that is still to land (the commits in both
// CTAs; after a failure also the copies, whose barriers the leader settles).
// 8192^3: 818 us with one-CTA tiles, 704 (1,562 TFLOP/s) with pairs issued by one lane,
// 587 to 605 (1,818 to 1,874) issued from whole warps (see gemm_tile); the same bits.
constexpr int kPairStages = 6, kPairTile = 256, kPairThreads = 256;
constexpr uint32_t kPairHalf = 128 * BK * 2;             // bytes of one CTA's half of A or B per stage
constexpr size_t kPairSmem = (size_t)kPairStages * 2 * kPairHalf + 1024;

__global__ void __launch_bounds__(kPairThreads, 1)
k_gemm_pair(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b, int K, int tiles_m,
            int tiles_n, int ldc, float *__restrict__ C, uint32_t spin_limit, int *__restrict__ err) {
    namespace px = titan::ptx;
    extern __shared__ uint8_t gsm_raw[];
    __shared__ uint64_t full[kPairStages], empty[kPairStages], acc_full[2], acc_empty[2], done;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    // k-blocks whose copies this CTA issued; in the leader, k-blocks and tiles whose products were
    // issued; the same, and `failed`, of the other CTA (written by it at the end)
    __shared__ int n_issued, n_mma, n_acc, peer[4];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // known to be the same in every lane
    const uint32_t rank = px::cluster_ctarank();
    const int pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1), tiles = tiles_m * tiles_n;
    const uint32_t raw = px::smem_u32(gsm_raw);
    uint8_t *gsm = gsm_raw + (((raw + 1023u) & ~1023u) - raw);
    auto tileA = [&](int s) { return gsm + (size_t)s * (2 * kPairHalf); };
    auto tileB = [&](int s) { return gsm + (size_t)s * (2 * kPairHalf) + kPairHalf; };
    const int num_kb = K / BK;
    // tiles in bands of 8 tile rows, column by column within a band: the tiles in
    // flight at one time then read about as many rows of A as of B
    auto tile_at = [&](int t, int &m0, int &n0) {
        const int band = t / (8 * tiles_n), r0 = 8 * band, rows = min(8, tiles_m - r0), in = t - r0 * tiles_n;
        m0 = (r0 + in % rows) * kPairTile;
        n0 = in / rows * kPairTile;
    };

    if (warp == 0) px::tmem_alloc_pair(&tmem_base, 512);
    if (tid == 32) {
        for (int s = 0; s < kPairStages; ++s) {
            px::mbar_init(&full[s], 1);
            px::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            px::mbar_init(&acc_full[b], 1);
            px::mbar_init(&acc_empty[b], 8);
        }
        px::mbar_init(&done, 1);
        px::fence_mbar_init();
        failed = n_issued = n_mma = n_acc = 0;
    }
    px::tc_fence_before();
    __syncthreads();
    px::cluster_sync();                                    // both CTAs' barriers are ready
    px::tc_fence_after();
    const uint32_t taddr = tmem_base;

    if (warp == 0) {                                       // TMA producer (one lane issues, as in gemm_tile)
        const bool leader = px::elect_one();
        const uint32_t bar0 = px::cluster_smem(&full[0], 0);
        int it = 0;
        uint32_t s = 0, parity = 1;
        bool ok = true;
        for (int t = pair; t < tiles && ok; t += pairs) {
            int m0, n0;
            tile_at(t, m0, n0);
            for (int kb = 0; kb < num_kb; ++kb, ++it) {
                if (it >= kPairStages && !px::mbar_wait_warp(&empty[s], parity, spin_limit)) {
                    ok = false;
                    break;
                }
                if (leader) {
                    if (rank == 0) px::mbar_arrive_expect_tx(&full[s], 4 * kPairHalf);
                    const uint32_t bar = bar0 + 8 * s;
                    px::tma_load_2d_pair(tileA(s), &tma_a, kb * BK, m0 + 128 * (int)rank, bar);
                    px::tma_load_2d_pair(tileB(s), &tma_b, kb * BK, n0 + 128 * (int)rank, bar);
                }
                __syncwarp();
                if (++s == kPairStages) {
                    s = 0;
                    parity ^= 1;
                }
            }
        }
        if (!ok && leader) atomicExch(&failed, 1);
        if (leader) n_issued = it;
    } else if (warp == 1 && rank == 0) {                   // MMA issuer
        constexpr uint32_t idesc2 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kPairTile >> 3) << 17) |
                                    ((uint32_t)(kPairTile >> 4) << 24);
        const bool leader = px::elect_one();
        uint64_t da = px::smem_desc_sw128(px::smem_u32(tileA(0))), db = px::smem_desc_sw128(px::smem_u32(tileB(0)));
        constexpr int64_t kStep = 2 * kPairHalf >> 4;
        uint32_t s = 0, parity = 0;
        int i = 0, mma = 0;
        bool ok = true, ready = false;                     // ready: the next k-block was seen to have arrived
        for (int t = pair; t < tiles && ok; t += pairs, ++i) {
            const int b = i & 1;
            if (i >= 2 && !px::mbar_wait_warp(&acc_empty[b], ((i >> 1) & 1) ^ 1, spin_limit)) {
                ok = false;
                break;
            }
            px::tc_fence_after();
            for (int kb = 0; kb < num_kb; ++kb, ++mma) {
                if (!ready && !px::mbar_wait_warp(&full[s], parity, spin_limit)) {
                    ok = false;
                    break;
                }
                px::tc_fence_after();
                const uint32_t s1 = s + 1 == kPairStages ? 0 : s + 1, parity1 = parity ^ (s1 == 0);
                ready = (kb + 1 < num_kb || t + pairs < tiles) && __all_sync(0xffffffffu, px::mbar_test(&full[s1], parity1));
                if (leader) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        px::tc_mma_bf16_pair(taddr + (uint32_t)(b * kPairTile), da + 2 * k, db + 2 * k, idesc2, (kb | k) != 0);
                    px::tc_commit_pair(&empty[s]);
                }
                __syncwarp();
                da += s1 ? kStep : kStep - kPairStages * kStep;
                db += s1 ? kStep : kStep - kPairStages * kStep;
                s = s1;
                parity = parity1;
            }
            if (leader) px::tc_commit_pair(&acc_full[b]);
        }
        if (leader) {
            px::tc_commit_pair(&done);                     // fires when every issued MMA is done
            n_mma = mma;
            n_acc = i;
            if (!ok) atomicExch(&failed, 1);
        }
    } else if (warp >= 4) {                                // epilogue
        const uint32_t q = warp & 3;
        int i = 0;
        for (int t = pair; t < tiles; t += pairs, ++i) {
            const int b = i & 1;
            int m0, n0;
            tile_at(t, m0, n0);
            if (!px::mbar_wait_warp(&acc_full[b], (i >> 1) & 1, spin_limit)) {
                atomicExch(&failed, 1);
                break;
            }
            px::tc_fence_after();
            float *row = C + (size_t)(m0 + 128 * (int)rank + 32 * (int)q + (int)lane) * ldc + n0;
#pragma unroll 1
            for (int c0 = 0; c0 < kPairTile; c0 += 32) {
                float v[32];
                px::tmem_ld32(taddr + ((q * 32u) << 16) + (uint32_t)(b * kPairTile + c0), v);
                // whole 32-byte sectors of this lane's row
#pragma unroll
                for (int x = 0; x < 32; x += 8)
                    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(row + c0 + x),
                                 "f"(v[x]), "f"(v[x + 1]), "f"(v[x + 2]), "f"(v[x + 3]), "f"(v[x + 4]), "f"(v[x + 5]),
                                 "f"(v[x + 6]), "f"(v[x + 7])
                                 : "memory");
            }
            px::tc_fence_before();
            __syncwarp();
            if (lane == 0) px::mbar_arrive_cluster(px::cluster_smem(&acc_empty[b], 0));
        }
    }
    __syncwarp();
    px::tc_fence_before();
    __syncthreads();
    if (tid == 0 && failed) {
        *reinterpret_cast<volatile int *>(err) = 1;        // may live in pinned host memory
        __threadfence_system();
    }
    if (tid < 4)
        px::st_cluster(px::cluster_smem(&peer[tid], rank ^ 1), tid == 0 ? failed : tid == 1 ? n_issued : tid == 2 ? n_mma : n_acc);
    px::cluster_sync();                                    // neither CTA issues anything any more
    const bool bad = failed || peer[0];
    if (warp == 0) {
        const int mma = rank ? peer[2] : n_mma, acc = rank ? peer[3] : n_acc;
        px::mbar_wait_warp(&done, 0, kDrainPolls);
        // the last releases of the ring, which no producer waited for
        for (int j = titan::ring_tail(mma, kPairStages); j < mma; ++j)
            px::mbar_wait_warp(&empty[titan::ring_slot(j, kPairStages)], titan::ring_parity(j, kPairStages), kDrainPolls);
        if (bad) {                                         // and what an epilogue or the issuer did not
            for (int j = titan::ring_tail(acc, 2); j < acc; ++j)
                px::mbar_wait_warp(&acc_full[titan::ring_slot(j, 2)], titan::ring_parity(j, 2), kDrainPolls);
            if (rank == 0)
                for (int j = mma; j < max(n_issued, peer[1]); ++j) {
                    uint64_t *bar = &full[titan::ring_slot(j, kPairStages)];
                    const titan::PairSettle fix = titan::pair_settle(j, n_issued, peer[1], 2 * kPairHalf);
                    if (lane == 0 && fix.expect) px::mbar_arrive_expect_tx(bar, fix.expect);
                    if (lane == 0 && fix.cancel) px::mbar_complete_tx(bar, fix.cancel);
                    __syncwarp();
                    px::mbar_wait_warp(bar, titan::ring_parity(j, kPairStages), kDrainPolls);
                }
        }
    }
    __syncwarp();
    if (bad) px::cluster_sync();                           // the other CTA's copies report to the leader
    px::tc_fence_after();
    if (warp == 0) px::tmem_dealloc_pair(taddr, 512);
}

// ------------------------------------------------------------------ CUDA-core kernels

__global__ void k_f32_to_bf16(const float *__restrict__ in, __nv_bfloat16 *__restrict__ out, size_t n) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = __float2bfloat16_rn(in[i]);
}

// The kernels of a pass are launched as programmatic dependents of one another:
// each starts while the one before it drains, and touches nothing of global
// memory before grid_dep_wait().  What an earlier kernel of the chain wrote is read
// through L2 (an L1 line may be older than the wait).

// A training step's own copy of its batch (the caller's arrays are free again
// once it has run): n16 16-byte pieces of x, B targets.
__global__ void k_take_batch(const uint4 *__restrict__ x, uint4 *__restrict__ gx, size_t n16, const float *__restrict__ t,
                             float *__restrict__ gt, uint32_t B) {
    titan::ptx::grid_dep_launch();
    titan::ptx::grid_dep_wait();
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    for (size_t k = i; k < n16; k += step) gx[k] = __ldcg(x + k);
    for (size_t k = i; k < B; k += step) gt[k] = __ldcg(t + k);
}

// This warp's dot product of a BF16 row of H with w, the same on every lane.
__device__ __forceinline__ float row_dot(const __nv_bfloat16 *H, const float *w, int cols, uint32_t lane) {
    float s = 0.f;
#pragma unroll 8
    for (int c = (int)lane; c < cols; c += 32)
        s += __bfloat162float(__ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short *>(H) + c))) * __ldcg(w + c);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// y[b] = H[b, :] . w + bias (one warp per row).
__global__ void k_out_layer(const __nv_bfloat16 *__restrict__ H, const float *__restrict__ w, const float *__restrict__ b,
                            float *__restrict__ y, int rows, int cols) {
    titan::ptx::grid_dep_launch();
    titan::ptx::grid_dep_wait();
    const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float s = row_dot(H + (size_t)row * cols, w, cols, lane);
    if (lane == 0) y[row] = s + __ldcg(b);
}

// The head of a training pass, a block per kHeadRows rows: the output layer's y,
// diff = y - t, dy = 2 diff / B, and from them per column
//   part[c]   = sum of dy H[., c]          (the block's share of dw4)
//   dZ[b, c]  = dy w4[c] GELU'(Z[b, c])    in BF16
//   part_b[c] = sum of that dZ             (of the last hidden layer's db)
// every sum in row order; the blocks' shares are added where they are used.  It
// replaces four kernels (output layer, loss in one block, backward by columns,
// transpose) that passed y and dy through memory; what bounds it is the GELU
// derivative's arithmetic.
constexpr int kHeadRows = 32, kHeadThreads = 512;

__global__ void __launch_bounds__(kHeadThreads, 2)
k_head(const __nv_bfloat16 *__restrict__ H, const float *__restrict__ Z, const float *__restrict__ t,
       const float *__restrict__ w, const float *__restrict__ b, int B, int cols, __nv_bfloat16 *__restrict__ dZ,
       float *__restrict__ part, float *__restrict__ part_b, float *__restrict__ diff,
       unsigned long long *__restrict__ tick) {
    __shared__ float s_dy[kHeadRows];
    titan::ptx::grid_dep_launch();
    titan::ptx::grid_dep_wait();
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t b0 = (size_t)blockIdx.x * kHeadRows;
#pragma unroll
    for (uint32_t r = warp; r < kHeadRows; r += kHeadThreads / 32) {
        const float s = row_dot(H + (b0 + r) * cols, w, cols, lane);
        if (lane == 0) {
            const float d = s + __ldcg(b) - __ldcg(t + b0 + r);
            s_dy[r] = 2.f * d / (float)B;
            diff[b0 + r] = d;
        }
    }
    __syncthreads();
    if (tick && blockIdx.x == 0 && tid == 0) atomicAdd(tick, 1ull);   // the Adam step counter (in L2), read by later kernels
    for (int c = (int)tid; c < cols; c += kHeadThreads) {
        const float wc = __ldcg(w + c);
        float s = 0.f, sb = 0.f;
#pragma unroll 1
        for (int r0 = 0; r0 < kHeadRows; r0 += 16) {           // 16 rows' loads in flight
            float hv[16], zv[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const size_t o = (b0 + r0 + r) * cols + c;
                hv[r] = __bfloat162float(__ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short *>(H) + o)));
                zv[r] = __ldcg(Z + o);
            }
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const float d = s_dy[r0 + r];
                s += d * hv[r];
                const __nv_bfloat16 g = __float2bfloat16_rn(d * wc * gelu_grad(zv[r]));
                dZ[(b0 + r0 + r) * cols + c] = g;
                sb += __bfloat162float(g);
            }
        }
        part[(size_t)blockIdx.x * cols + c] = s;
        part_b[(size_t)blockIdx.x * cols + c] = sb;
    }
}

// The sum over chunks of part[k][c0 + x] for the 32 columns from c0, in a fixed
// order: for each j < 32 the chunks j, j + 32, ... in turn, then those 32 sums
// pairwise (256 threads, thread 32 q + x taking j = q, q + 8, q + 16, q + 24).
// Returned to threads 0 .. 31.
__device__ __forceinline__ float column_sum(const float *part, int chunks, int cols, int c0, float (*s)[33]) {
    const int x = threadIdx.x & 31, q = threadIdx.x >> 5;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    int k = q;
    for (; k + 120 < chunks; k += 128) {              // 16 loads in flight
        float p[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u] = __ldcg(part + (size_t)(k + 8 * u) * cols + c0 + x);
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u & 3] += p[u];
    }
    for (; k < chunks; k += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k + 8 * u < chunks) v[u] += __ldcg(part + (size_t)(k + 8 * u) * cols + c0 + x);
#pragma unroll
    for (int u = 0; u < 4; ++u) s[q + 8 * u][x] = v[u];
    __syncthreads();
    for (int o = 16; o; o >>= 1) {
        for (int j = q; j < o; j += 8) s[j][x] += s[j + o][x];
        __syncthreads();
    }
    return s[0][x];
}

// The sums of diff^2 (x) and dy = 2 diff / B (y) over the batch in a fixed order: for
// each i < 1,024 the rows i, i + 1,024, ... in turn, then those sums pairwise.
__device__ __forceinline__ float2 loss_sum(const float *diff, uint32_t B, float2 *s) {
    float2 v[4] = {};
    for (uint32_t k0 = threadIdx.x; k0 < B; k0 += 4096) {
        float d[16];                                  // all in flight before the first division
#pragma unroll
        for (int j = 0; j < 16; ++j) d[j] = k0 + 256 * j < B ? __ldcg(diff + k0 + 256 * j) : 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (k0 + 256 * j < B) {
                v[j & 3].x += d[j] * d[j];
                v[j & 3].y += 2.f * d[j] / (float)B;
            }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) s[threadIdx.x + 256 * u] = v[u];
    __syncthreads();
    for (uint32_t o = 512; o; o >>= 1) {
        for (uint32_t i = threadIdx.x; i < o; i += 256) {
            s[i].x += s[i + o].x;
            s[i].y += s[i + o].y;
        }
        __syncthreads();
    }
    return s[0];
}

// What the gradients are formed from, and Adam's state.  Weights: the K slices'
// partial products of each layer; vectors (b1, b2, b3, w4): sums by column of 32 rows
// each; loss and b4: the head's y - t.
struct GradArgs {
    titan::MlpLayout at;
    const float *part[3];                 // [splits][hid][in_l] (one slice: in the gradient array)
    uint32_t splits[3], hid;
    const float *vpart[4];
    const float *diff;
    uint32_t B;
    float *loss;                          // may be null
};
struct AdamArgs {
    float *p, *m, *v;
    __nv_bfloat16 *wt[3];                 // the BF16 copies of the new weights, same layout
    const float *lr;                      // device memory, with the step counter
    const unsigned long long *t;
    float b1, b2, eps;
};

__device__ __forceinline__ float adam_one(const AdamArgs &a, float gi, float &m, float &v, float pi, float c1, float c2,
                                          float lr) {
    const float mi = __fmaf_rn(1.f - a.b1, gi, a.b1 * m);
    const float vi = __fmaf_rn((1.f - a.b2) * gi, gi, a.b2 * v);
    m = mi;
    v = vi;
    return pi - lr * (mi / c1) / (sqrtf(vi / c2) + a.eps);
}

// Forms every gradient and hands it on: first blocks of 32 columns of the four
// vectors and one for the loss and b4 (the longest chains), then blocks of 1,024
// weights layer by layer (four per thread).  state(layer, index) requests what
// weight(layer, index, state, gradient of four) needs besides the gradient, so that
// it arrives together with the slices; scalar(index, gradient) takes the others.
template <class S, class W, class V>
__device__ __forceinline__ void for_gradients(const GradArgs &g, S &&state, W &&weight, V &&scalar) {
    __shared__ union {
        float col[32][33];
        float2 loss[1024];
    } s;
    const uint32_t tid = threadIdx.x, per = g.hid >> 5;
    uint32_t blk = blockIdx.x;
    if (blk > 4 * per) {
        blk -= 4 * per + 1;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const uint32_t blocks = titan::grad_blocks(g.at.n_w[l]);
            if (blk < blocks) {
                const size_t i = titan::grad_index(blk, tid);
                const uint32_t splits = g.splits[l];          // at most 8
                const auto st = state(l, i);
                float4 r[8];
#pragma unroll
                for (uint32_t z = 0; z < 8; ++z)
                    if (z < splits) r[z] = __ldcg(reinterpret_cast<const float4 *>(g.part[l] + z * g.at.n_w[l] + i));
                float4 q = r[0];
#pragma unroll
                for (uint32_t z = 1; z < 8; ++z)              // slices in order
                    if (z < splits) {
                        q.x += r[z].x;
                        q.y += r[z].y;
                        q.z += r[z].z;
                        q.w += r[z].w;
                    }
                weight(l, i, st, q);
                return;
            }
            blk -= blocks;
        }
        return;
    }
    if (blk < 4 * per) {
        const uint32_t k = blk / per, c0 = 32 * (blk - k * per);
        const float *part = k == 0 ? g.vpart[0] : k == 1 ? g.vpart[1] : k == 2 ? g.vpart[2] : g.vpart[3];
        const size_t off = k == 0 ? g.at.b[0] : k == 1 ? g.at.b[1] : k == 2 ? g.at.b[2] : g.at.w4;
        const float v = column_sum(part, (int)(g.B / 32), (int)g.hid, (int)c0, s.col);
        if (tid < 32) scalar(off + c0 + tid, v);
        return;
    }
    const float2 v = loss_sum(g.diff, g.B, s.loss);
    if (tid == 0) {
        if (g.loss) *g.loss = v.x / (float)g.B;
        scalar(g.at.b4, v.y);
    }
}

struct AdamState {
    float4 p, m, v;
};

// One Adam step on every parameter.  The slices and chunk sums are added here, in
// registers, instead of by seven kernels through a gradient array, and four weights
// per thread keep all of a thread's loads in flight together (24 bytes of state a
// weight, 4 a slice, 2 for the copy: bound by L2 and HBM).
__global__ void __launch_bounds__(256) k_adam(GradArgs g, AdamArgs a) {
    titan::ptx::grid_dep_launch();
    titan::ptx::grid_dep_wait();
    const float tf = (float)__ldcg(a.t), lr = __ldcg(a.lr);
    auto corrections = [&](float &c1, float &c2) {      // after the loads are on their way
        c1 = 1.f - powf(a.b1, tf);
        c2 = 1.f - powf(a.b2, tf);
    };
    for_gradients(
        g,
        [&](int l, size_t i) {
            const size_t o = g.at.w[l] + i;
            return AdamState{__ldcg(reinterpret_cast<float4 *>(a.p + o)), __ldcg(reinterpret_cast<float4 *>(a.m + o)),
                             __ldcg(reinterpret_cast<float4 *>(a.v + o))};
        },
        [&](int l, size_t i, const AdamState &st, float4 q) {
            const size_t o = g.at.w[l] + i;
            float4 p = st.p, m = st.m, v = st.v;
            float c1, c2;
            corrections(c1, c2);
            p.x = adam_one(a, q.x, m.x, v.x, p.x, c1, c2, lr);
            p.y = adam_one(a, q.y, m.y, v.y, p.y, c1, c2, lr);
            p.z = adam_one(a, q.z, m.z, v.z, p.z, c1, c2, lr);
            p.w = adam_one(a, q.w, m.w, v.w, p.w, c1, c2, lr);
            *reinterpret_cast<float4 *>(a.m + o) = m;
            *reinterpret_cast<float4 *>(a.v + o) = v;
            *reinterpret_cast<float4 *>(a.p + o) = p;
            *reinterpret_cast<uint2 *>(a.wt[l] + i) =
                make_uint2(bf16_bits(__float2bfloat16_rn(p.x), __float2bfloat16_rn(p.y)),
                           bf16_bits(__float2bfloat16_rn(p.z), __float2bfloat16_rn(p.w)));
        },
        [&](size_t i, float q) {
            float m = __ldcg(a.m + i), v = __ldcg(a.v + i), c1, c2;
            corrections(c1, c2);
            a.p[i] = adam_one(a, q, m, v, __ldcg(a.p + i), c1, c2, lr);
            a.m[i] = m;
            a.v[i] = v;
        });
}

// The same gradients into the flat array out (a layer of one slice is there already).
__global__ void __launch_bounds__(256) k_form_gradient(GradArgs g, float *out) {
    titan::ptx::grid_dep_launch();
    titan::ptx::grid_dep_wait();
    for_gradients(
        g, [](int, size_t) { return 0; },
        [&](int l, size_t i, int, float4 q) { *reinterpret_cast<float4 *>(out + g.at.w[l] + i) = q; },
        [&](size_t i, float q) { out[i] = q; });
}

// ------------------------------------------------------------------ host helpers

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Tensor map of a row-major [rows, cols] BF16 matrix read in boxes of box_rows rows of 64.
bool make_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows = 128) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 2};
    const cuuint32_t box[2] = {BK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Launches kern as a programmatic dependent of the operation before it on st (it
// may start early and waits in grid_dep_wait).
template <typename... Par, typename... Arg>
cudaError_t launch_dependent(void (*kern)(Par...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Arg &&...arg) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Arg>(arg)...);
}

// The dynamic shared memory of a GEMM kernel, allowed once per device.
template <typename Kern>
cudaError_t allow_smem(Kern kern, size_t bytes, std::atomic<uint64_t> &set) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (set.load() & (1ull << (dev & 63))) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) set.fetch_or(1ull << (dev & 63));
    return e;
}

// C[M, N] = A B^T with the given epilogue; A is [M, K], B [N, K] or, with BMN,
// [K, N].  M, N multiples of 128, K a multiple of 64; A, B 16-byte aligned, rows
// contiguous.
template <int BN_, bool BMN>
cudaError_t gemm_tn_launch(const CUtensorMap &ma, const CUtensorMap &mb, int M, int N, int K, const EpiArgs &ep,
                           cudaStream_t st, uint32_t spin_limit, int *err) {
    static std::atomic<uint64_t> set{0};
    const auto kern = k_gemm_tn<BN_, false, BMN>;
    cudaError_t e = allow_smem(kern, gemm_smem<BN_>(), set);
    if (e != cudaSuccess) return e;
    return launch_dependent(kern, dim3(N / BN_, M / BM), kGemmThreads, gemm_smem<BN_>(), st, ma, mb, K, ep, spin_limit, err);
}

cudaError_t gemm_pair_launch(const CUtensorMap &ma, const CUtensorMap &mb, int M, int N, int K, const EpiArgs &ep,
                             cudaStream_t st, uint32_t spin_limit, int *err, int sms) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem);
    if (e != cudaSuccess) return e;
    const int tm = M / kPairTile, tn = N / kPairTile;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)std::min<int64_t>(sms / 2, (int64_t)tm * tn));
    cfg.blockDim = dim3(kPairThreads);
    cfg.dynamicSmemBytes = kPairSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_gemm_pair, ma, mb, K, tm, tn, ep.ldc, ep.out_f32, spin_limit, err);
}

template <bool BMN = false>
cudaError_t gemm_tn(const void *A, const void *B, int M, int N, int K, const EpiArgs &ep, cudaStream_t st,
                    uint32_t spin_limit, int *err) {
    if (M % BM || N % BN || K % BK || M <= 0 || N <= 0 || K <= 0) return cudaErrorInvalidValue;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return cudaErrorInvalidValue;
    const int width = titan::gemm_tile_width(M, N, K, ep.mode != EPI_F32);
    CUtensorMap ma, mb;
    if (!make_map(&ma, A, M, K)) return cudaErrorInvalidValue;
    // the pairs' epilogue writes whole 32-byte sectors
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!BMN && ep.mode == EPI_F32 && titan::gemm_takes_pairs(M, N, K, sms) &&
        !(reinterpret_cast<uintptr_t>(ep.out_f32) & 31)) {
        if (!make_map(&mb, B, N, K)) return cudaErrorInvalidValue;
        return gemm_pair_launch(ma, mb, M, N, K, ep, st, spin_limit, err, sms);
    }
    if (!(BMN ? make_map(&mb, B, K, N, 64) : make_map(&mb, B, N, K, (uint32_t)width)))
        return cudaErrorInvalidValue;
    if (width == 256) return gemm_tn_launch<256, BMN>(ma, mb, M, N, K, ep, st, spin_limit, err);
    if (width == 64) return gemm_tn_launch<64, BMN>(ma, mb, M, N, K, ep, st, spin_limit, err);
    return gemm_tn_launch<128, BMN>(ma, mb, M, N, K, ep, st, spin_limit, err);
}

cudaError_t wgrad_launch(const WgradArgs &w, int blocks, int hid, cudaStream_t st, uint32_t spin_limit, int *err) {
    static std::atomic<uint64_t> set{0};
    cudaError_t e = allow_smem(k_wgrad, gemm_smem<BN>(), set);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_wgrad, dim3(blocks), kGemmThreads, gemm_smem<BN>(), st, w, hid, spin_limit, err);
}

inline unsigned nblk(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ------------------------------------------------------------------ the MLP

struct titan_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    uint32_t in = 0, hid = 0;
    uint32_t spin_limit = 1u << 22;
    titan::MlpLayout at;                                   // of the parameters in p, g, m, v
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    // BF16 W^T [hid][in_l]: B operand of the forward product and, read with hid as
    // its K, of the input gradient
    __nv_bfloat16 *wt[3] = {nullptr, nullptr, nullptr};
    uint32_t cap = 0;                                      // batch capacity of the activations
    float *Z[3] = {nullptr, nullptr, nullptr};
    __nv_bfloat16 *H[3] = {nullptr, nullptr, nullptr};
    __nv_bfloat16 *dZ[3] = {nullptr, nullptr, nullptr};
    float *part = nullptr;                                 // dw4: sums of 32 rows [B / 32][hidden]
    float *partb[3] = {nullptr, nullptr, nullptr};         // the same for db_l
    float *diff = nullptr;                                 // y - t
    float *wsk = nullptr;                                  // K slices of the weight gradients (layers of several)
    size_t wsk_cap = 0;                                    // floats
    volatile int *err_host = nullptr;                      // bounded-wait flag: pinned, mapped
    int *err = nullptr;
    // a training step's own copy of its batch, learning rate and step count
    __nv_bfloat16 *gx = nullptr;
    float *gt = nullptr, *d_lr = nullptr;
    unsigned long long *d_step = nullptr;
    uint32_t g_cap = 0;
    float lr_set = -1.f;
    std::vector<void *> allocs;
    std::string error;
};

namespace {

titan_status mfail(titan_mlp *m, titan_status st, const std::string &msg) {
    if (m) m->error = msg;
    else titan::set_thread_error(msg);
    return st;
}

#define MLP_CK(m, call)                                                                          \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess)                                                                   \
            return mfail((m), e_ == cudaErrorMemoryAllocation ? TITAN_E_OOM : TITAN_E_CUDA,       \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                    \
    } while (0)

template <typename T>
cudaError_t malloc_t(titan_mlp *m, T **p, size_t count) {
    void *raw = nullptr;
    cudaError_t e = cudaMalloc(&raw, std::max<size_t>(count, 1) * sizeof(T));
    if (e == cudaSuccess) {
        m->allocs.push_back(raw);
        *p = static_cast<T *>(raw);
    }
    return e;
}

uint32_t layer_in(const titan_mlp *m, int l) { return l == 0 ? m->in : m->hid; }

// K slices of a weight-gradient product (hid x in, summed over the batch B):
// its hid/128 x in/128 tiles alone fill a small part of the 152 SMs, so the
// batch is cut into up to 8 slices of at least 4 k-blocks while the tiles
// times the slices stay within one wave.
int wgrad_splits(uint32_t hid, uint32_t in, uint32_t B) {
    const uint32_t tiles = (hid / BM) * (in / 128);
    int s = 1;
    while (s < 8 && tiles * (uint32_t)(2 * s) <= 152 && B % (uint32_t)(2 * s * BK) == 0 && B / (2 * s) >= 4 * BK)
        s *= 2;
    return s;
}

// Refreshes the BF16 hidden-layer weights from the FP32 master.
cudaError_t refresh_bf16(titan_mlp *m) {
    for (int l = 0; l < 3; ++l) {
        const size_t n = (size_t)m->hid * layer_in(m, l);
        k_f32_to_bf16<<<nblk(n, 256), 256, 0, m->stream>>>(m->p + m->at.w[l], m->wt[l], n);
    }
    return cudaGetLastError();
}

cudaError_t ensure_batch(titan_mlp *m, uint32_t B) {
    if (B <= m->cap) return cudaSuccess;
    cudaError_t e;
    for (int l = 0; l < 3; ++l) {
        if ((e = malloc_t(m, &m->Z[l], (size_t)B * m->hid)) != cudaSuccess) return e;
        if ((e = malloc_t(m, &m->H[l], (size_t)B * m->hid)) != cudaSuccess) return e;
        if ((e = malloc_t(m, &m->dZ[l], (size_t)B * m->hid)) != cudaSuccess) return e;
        if ((e = malloc_t(m, &m->partb[l], (size_t)(B / 32) * m->hid)) != cudaSuccess) return e;
    }
    if ((e = malloc_t(m, &m->part, (size_t)(B / 32) * m->hid)) != cudaSuccess) return e;
    if ((e = malloc_t(m, &m->diff, B)) != cudaSuccess) return e;
    m->cap = B;
    return cudaSuccess;
}

// The slices of the weight gradients (their number depends on the batch).  A layer of
// one slice needs none: its product goes straight to the gradient array.
cudaError_t ensure_slices(titan_mlp *m, uint32_t B) {
    size_t ws = 0;
    for (int l = 0; l < 3; ++l) {
        const int splits = wgrad_splits(m->hid, layer_in(m, l), B);
        if (splits > 1) ws += splits * m->at.n_w[l];
    }
    if (ws <= m->wsk_cap) return cudaSuccess;
    cudaError_t e = malloc_t(m, &m->wsk, ws);
    if (e == cudaSuccess) m->wsk_cap = ws;
    return e;
}

// keep: the pre-activations are written too (a backward pass follows).
cudaError_t hidden_layers(titan_mlp *m, const __nv_bfloat16 *x, uint32_t B, bool keep) {
    cudaError_t e;
    const __nv_bfloat16 *a = x;
    for (int l = 0; l < 3; ++l) {
        EpiArgs ep{EPI_BIAS_GELU, (int)m->hid, m->p + m->at.b[l], keep ? m->Z[l] : nullptr, m->H[l], nullptr};
        if ((e = gemm_tn(a, m->wt[l], (int)B, (int)m->hid, (int)layer_in(m, l), ep, m->stream, m->spin_limit, m->err)) != cudaSuccess)
            return e;
        a = m->H[l];
    }
    return cudaSuccess;
}

// Forward and backward for a batch in device memory: 7 launches on one stream, each
// a programmatic dependent of the one before.  Leaves what the gradients are formed
// from in *g.  train: the head advances the Adam step counter.
cudaError_t backward_pass(titan_mlp *m, const __nv_bfloat16 *x, const float *t, uint32_t B, float *loss, GradArgs *g,
                          bool train) {
    cudaError_t e;
    const int hid = (int)m->hid;
    if ((e = ensure_slices(m, B)) != cudaSuccess) return e;
    if ((e = hidden_layers(m, x, B, true)) != cudaSuccess) return e;
    if ((e = launch_dependent(k_head, dim3(B / kHeadRows), kHeadThreads, 0, m->stream, m->H[2], m->Z[2], t,
                              m->p + m->at.w4, m->p + m->at.b4, (int)B, hid, m->dZ[2], m->part, m->partb[2], m->diff,
                              train ? m->d_step : nullptr)) != cudaSuccess)
        return e;
    for (int l = 2; l > 0; --l) {
        // dZ_{l-1} = (dZ_l W_l^T) * GELU'(Z_{l-1}):  A = dZ_l, B = W_l^T [hid][in] with hid as K
        EpiArgs ep{EPI_GELU_GRAD, hid, nullptr, nullptr, m->dZ[l - 1], m->Z[l - 1], m->partb[l - 1]};
        if ((e = gemm_tn<true>(m->dZ[l], m->wt[l], (int)B, hid, hid, ep, m->stream, m->spin_limit, m->err)) != cudaSuccess)
            return e;
    }
    WgradArgs w;
    int blocks = 0;
    size_t at = 0;
    for (int l = 0; l < 3; ++l) {
        const uint32_t in = layer_in(m, l);
        const int splits = wgrad_splits(m->hid, in, B);
        if (!make_map(&w.a[l], m->dZ[l], B, m->hid, 64) || !make_map(&w.b[l], l ? m->H[l - 1] : x, B, in, 64))
            return cudaErrorInvalidValue;
        w.out[l] = splits > 1 ? m->wsk + at : m->g + m->at.w[l];
        w.first[l] = blocks;
        w.tiles_n[l] = (int)(in / BN);
        w.tiles[l] = (int)(m->hid / BM) * w.tiles_n[l];
        w.ld[l] = (int)in;
        w.kslice[l] = (int)B / splits;
        blocks += splits * w.tiles[l];
        if (splits > 1) at += splits * m->at.n_w[l];
        g->part[l] = w.out[l];
        g->splits[l] = (uint32_t)splits;
        g->vpart[l] = m->partb[l];
    }
    g->at = m->at;
    g->hid = m->hid;
    g->vpart[3] = m->part;
    g->diff = m->diff;
    g->B = B;
    g->loss = loss;
    return wgrad_launch(w, blocks, hid, m->stream, m->spin_limit, m->err);
}

// The grid of k_adam and k_form_gradient (see for_gradients).
unsigned gradient_blocks(const GradArgs &g) {
    unsigned blocks = 4 * (g.hid >> 5) + 1;
    for (size_t n : g.at.n_w) blocks += titan::grad_blocks(n);
    return blocks;
}

titan_status check_err(titan_mlp *m) {
    MLP_CK(m, cudaStreamSynchronize(m->stream));
    if (*m->err_host) {
        *m->err_host = 0;
        return mfail(m, TITAN_E_TIMEOUT, "a bounded wait in the tensor-core GEMM expired");
    }
    return TITAN_OK;
}

}  // namespace

extern "C" {

// One bounded-wait flag per device ordinal for the standalone GEMM, in
// pinned host memory mapped into the device: a call reads it without
// waiting for its stream.
namespace {
std::mutex g_gemm_mu;
volatile int *g_gemm_flag[64] = {};
int *g_gemm_flag_dev[64] = {};

titan_status gemm_flag(int *dev_out, volatile int **host, int **dev_ptr, const char *who) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return mfail(nullptr, TITAN_E_CUDA, std::string(who) + ": no current device");
    std::lock_guard<std::mutex> lk(g_gemm_mu);
    if (!g_gemm_flag[dev]) {
        void *h = nullptr, *d = nullptr;
        if (cudaHostAlloc(&h, sizeof(int), cudaHostAllocMapped) != cudaSuccess)
            return mfail(nullptr, TITAN_E_OOM, std::string(who) + ": error flag");
        *static_cast<volatile int *>(h) = 0;
        if (cudaHostGetDevicePointer(&d, h, 0) != cudaSuccess) {
            cudaFreeHost(h);
            return mfail(nullptr, TITAN_E_CUDA, std::string(who) + ": error flag");
        }
        g_gemm_flag[dev] = static_cast<volatile int *>(h);
        g_gemm_flag_dev[dev] = static_cast<int *>(d);
    }
    *dev_out = dev;
    *host = g_gemm_flag[dev];
    *dev_ptr = g_gemm_flag_dev[dev];
    return TITAN_OK;
}
}  // namespace

titan_status titan_gemm_bf16_tn(uint32_t M, uint32_t N, uint32_t K, const uint16_t *A_dev, const uint16_t *B_dev,
                                float *C_dev, void *stream) {
    if (!A_dev || !B_dev || !C_dev) return mfail(nullptr, TITAN_E_INVALID, "titan_gemm_bf16_tn: null pointer");
    if (M % BM || N % BN || K % BK || !M || !N || !K)
        return mfail(nullptr, TITAN_E_INVALID, "titan_gemm_bf16_tn: M and N must be multiples of 128, K of 64");
    int dev = 0;
    volatile int *flag = nullptr;
    int *err = nullptr;
    titan_status fs = gemm_flag(&dev, &flag, &err, "titan_gemm_bf16_tn");
    if (fs != TITAN_OK) return fs;
    if (*flag) {                     // an earlier call's kernel gave up on a wait
        *flag = 0;
        return mfail(nullptr, TITAN_E_TIMEOUT, "titan_gemm_bf16_tn: a bounded wait expired in an earlier call");
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    EpiArgs ep{EPI_F32, (int)N, nullptr, C_dev, nullptr, nullptr};
    cudaError_t e = gemm_tn(A_dev, B_dev, (int)M, (int)N, (int)K, ep, st, 1u << 22, err);
    if (e != cudaSuccess) return mfail(nullptr, TITAN_E_CUDA, std::string("titan_gemm_bf16_tn: ") + cudaGetErrorString(e));
    return TITAN_OK;
}

titan_status titan_gemm_check(void) {
    int dev = 0;
    volatile int *flag = nullptr;
    int *err = nullptr;
    titan_status fs = gemm_flag(&dev, &flag, &err, "titan_gemm_check");
    if (fs != TITAN_OK) return fs;
    if (*flag) {
        *flag = 0;
        return mfail(nullptr, TITAN_E_TIMEOUT, "titan_gemm_bf16_tn: a bounded wait expired");
    }
    return TITAN_OK;
}

titan_status titan_mlp_create(uint32_t in, uint32_t hidden, uint64_t seed, int32_t device, void *stream,
                              titan_mlp **out) {
    if (!out || in % 128 || hidden % 128 || !in || !hidden)
        return mfail(nullptr, TITAN_E_INVALID, "titan_mlp_create: in and hidden must be positive multiples of 128");
    titan_mlp *m = new titan_mlp();
    m->device = device;
    m->in = in;
    m->hid = hidden;
    m->at = titan::mlp_layout(in, hidden);
    const size_t o = m->at.total;
    auto bail = [&](titan_status st) {
        titan::set_thread_error(m->error);
        for (void *p : m->allocs) cudaFree(p);
        if (m->err_host) cudaFreeHost(const_cast<int *>(m->err_host));
        if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
        delete m;
        return st;
    };
#define C_CK(call)                                                                               \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess) return bail(mfail(m, TITAN_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_))); \
    } while (0)
    C_CK(cudaSetDevice(device));
    if (!encode_fn()) return bail(mfail(m, TITAN_E_UNSUPPORTED, "cuTensorMapEncodeTiled is not available"));
    if (stream) m->stream = static_cast<cudaStream_t>(stream);
    else { C_CK(cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking)); m->own_stream = true; }
    C_CK(malloc_t(m, &m->p, o));
    C_CK(malloc_t(m, &m->g, o));
    C_CK(malloc_t(m, &m->m, o));
    C_CK(malloc_t(m, &m->v, o));
    {
        void *h = nullptr, *d = nullptr;
        C_CK(cudaHostAlloc(&h, sizeof(int), cudaHostAllocMapped));
        m->err_host = static_cast<volatile int *>(h);
        *m->err_host = 0;
        C_CK(cudaHostGetDevicePointer(&d, h, 0));
        m->err = static_cast<int *>(d);
    }
    C_CK(malloc_t(m, &m->d_lr, 1));
    C_CK(malloc_t(m, &m->d_step, 1));
    C_CK(cudaMemset(m->d_step, 0, sizeof(unsigned long long)));
    for (int l = 0; l < 3; ++l) {
        C_CK(malloc_t(m, &m->wt[l], (size_t)hidden * layer_in(m, l)));
    }
    // He-style initialisation (uniform, variance 2 / fan_in for GELU layers), zero biases
    std::vector<float> h(o, 0.f);
    std::mt19937_64 rng(seed);
    for (int l = 0; l < 3; ++l) {
        const float a = std::sqrt(6.0f / (float)layer_in(m, l));
        std::uniform_real_distribution<float> U(-a, a);
        for (size_t k = 0; k < (size_t)hidden * layer_in(m, l); ++k) h[m->at.w[l] + k] = U(rng);
    }
    {
        const float a = std::sqrt(3.0f / (float)hidden);
        std::uniform_real_distribution<float> U(-a, a);
        for (uint32_t k = 0; k < hidden; ++k) h[m->at.w4 + k] = U(rng);
    }
    C_CK(cudaMemcpy(m->p, h.data(), o * 4, cudaMemcpyHostToDevice));
    C_CK(cudaMemset(m->m, 0, o * 4));
    C_CK(cudaMemset(m->v, 0, o * 4));
    C_CK(cudaMemset(m->g, 0, o * 4));
    C_CK(refresh_bf16(m));
    C_CK(cudaStreamSynchronize(m->stream));
#undef C_CK
    *out = m;
    return TITAN_OK;
}

uint64_t titan_mlp_param_count(const titan_mlp *m) { return m ? m->at.total : 0; }

titan_status titan_mlp_get_params(titan_mlp *m, float *host) {
    if (!m || !host) return TITAN_E_INVALID;
    MLP_CK(m, cudaStreamSynchronize(m->stream));
    MLP_CK(m, cudaMemcpy(host, m->p, m->at.total * 4, cudaMemcpyDeviceToHost));
    return TITAN_OK;
}

titan_status titan_mlp_set_params(titan_mlp *m, const float *host) {
    if (!m || !host) return TITAN_E_INVALID;
    MLP_CK(m, cudaStreamSynchronize(m->stream));
    MLP_CK(m, cudaMemcpy(m->p, host, m->at.total * 4, cudaMemcpyHostToDevice));
    MLP_CK(m, refresh_bf16(m));
    return check_err(m);
}

titan_status titan_mlp_forward(titan_mlp *m, const uint16_t *x_dev, uint32_t batch, float *y_dev) {
    if (!m || !x_dev || !y_dev || batch % 128 || !batch)
        return mfail(m, TITAN_E_INVALID, "titan_mlp_forward: batch must be a positive multiple of 128");
    MLP_CK(m, cudaSetDevice(m->device));
    MLP_CK(m, ensure_batch(m, batch));
    MLP_CK(m, hidden_layers(m, reinterpret_cast<const __nv_bfloat16 *>(x_dev), batch, false));
    MLP_CK(m, launch_dependent(k_out_layer, dim3(nblk(batch, 8)), 256, 0, m->stream, m->H[2], m->p + m->at.w4,
                               m->p + m->at.b4, y_dev, (int)batch, (int)m->hid));
    return check_err(m);
}

titan_status titan_mlp_gradient(titan_mlp *m, const uint16_t *x_dev, const float *t_dev, uint32_t batch,
                                float *loss_dev, float *grad_dev) {
    if (!m || !x_dev || !t_dev || batch % 128 || !batch)
        return mfail(m, TITAN_E_INVALID, "titan_mlp_gradient: batch must be a positive multiple of 128");
    MLP_CK(m, cudaSetDevice(m->device));
    MLP_CK(m, ensure_batch(m, batch));
    GradArgs g;
    MLP_CK(m, backward_pass(m, reinterpret_cast<const __nv_bfloat16 *>(x_dev), t_dev, batch, loss_dev, &g, false));
    MLP_CK(m, launch_dependent(k_form_gradient, dim3(gradient_blocks(g)), 256, 0, m->stream, g, m->g));
    if (grad_dev) MLP_CK(m, cudaMemcpyAsync(grad_dev, m->g, m->at.total * 4, cudaMemcpyDeviceToDevice, m->stream));
    return check_err(m);
}

titan_status titan_mlp_train_step(titan_mlp *m, const uint16_t *x_dev, const float *t_dev, uint32_t batch, float lr,
                                  float *loss_dev) {
    if (!m || !x_dev || !t_dev || batch % 128 || !batch)
        return mfail(m, TITAN_E_INVALID, "titan_mlp_train_step: batch must be a positive multiple of 128");
    MLP_CK(m, cudaSetDevice(m->device));
    MLP_CK(m, ensure_batch(m, batch));
    if (batch > m->g_cap) {
        MLP_CK(m, malloc_t(m, &m->gx, (size_t)batch * m->in));
        MLP_CK(m, malloc_t(m, &m->gt, batch));
        m->g_cap = batch;
    }
    if (lr != m->lr_set) {                              // pageable source: staged before the call returns
        MLP_CK(m, cudaMemcpyAsync(m->d_lr, &lr, sizeof(float), cudaMemcpyHostToDevice, m->stream));
        m->lr_set = lr;
    }
    size_t n16 = (size_t)batch * m->in / 8;
    if (reinterpret_cast<uintptr_t>(x_dev) & 15) {      // a view off the 16-byte grid
        MLP_CK(m, cudaMemcpyAsync(m->gx, x_dev, n16 * 16, cudaMemcpyDeviceToDevice, m->stream));
        n16 = 0;
    }
    MLP_CK(m, launch_dependent(k_take_batch, dim3((unsigned)std::min<size_t>(nblk(std::max<size_t>(n16, batch), 256), 152 * 8)), 256, 0, m->stream,
                               reinterpret_cast<const uint4 *>(x_dev), reinterpret_cast<uint4 *>(m->gx), n16, t_dev, m->gt,
                               batch));
    GradArgs g;
    MLP_CK(m, backward_pass(m, m->gx, m->gt, batch, loss_dev, &g, true));
    AdamArgs a{m->p, m->m, m->v, {m->wt[0], m->wt[1], m->wt[2]}, m->d_lr, m->d_step, 0.9f, 0.999f, 1e-8f};
    MLP_CK(m, launch_dependent(k_adam, dim3(gradient_blocks(g)), 256, 0, m->stream, g, a));
    return TITAN_OK;
}

titan_status titan_mlp_sync(titan_mlp *m) { return m ? check_err(m) : TITAN_E_INVALID; }

const char *titan_mlp_last_error(const titan_mlp *m) { return m ? m->error.c_str() : ""; }

titan_status titan_mlp_destroy(titan_mlp *m) {
    if (!m) return TITAN_OK;
    cudaStreamSynchronize(m->stream);
    if (m->err_host) cudaFreeHost(const_cast<int *>(m->err_host));
    for (void *p : m->allocs) cudaFree(p);
    if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
    delete m;
    return TITAN_OK;
}

}  // extern "C"
