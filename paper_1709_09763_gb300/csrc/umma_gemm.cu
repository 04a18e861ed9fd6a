// Tensor-core GEMM for sm_103a: C[M][N] = A[M][K] . B[N][K]^T, A and B BF16 row-major (K
// contiguous), FP32 accumulation in tensor memory, fused epilogues. Used by the surrogate network
// (forward, backward, weight gradients) and by the KL synthesis.
//
// Per CTA one 128 x BN output tile:
//  * thread 0 (producer) streams 64-wide K chunks of A (128 rows) and B (BN rows) into a ring of
//    STAGES shared-memory slots with TMA (cp.async.bulk.tensor, 128-byte swizzle), signalling a
//    "full" mbarrier per slot with the transaction byte count;
//  * thread 32 (issuer) waits for a full slot, issues four tcgen05.mma.kind::f16 (K = 16 each)
//    accumulating into TMEM, and releases the slot through tcgen05.commit on its "empty" mbarrier;
//  * after the last chunk a commit on the "done" mbarrier hands the accumulator to all four warps,
//    which read their 32 TMEM lanes (= tile rows) with tcgen05.ld and apply the epilogue.
// Every wait is bounded: on time-out the CTA sets *err, stops issuing, and still frees its TMEM.
// Out-of-range rows and K columns are zero-filled by TMA; stores are masked to M x N.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <atomic>
#include <mutex>
#include <unordered_map>

#include "internal.h"
#include "launch.h"
#include "umma_gemm.h"

namespace mls2mc {

namespace {

constexpr uint32_t kSpinLimit = 1u << 22;   // bounded mbarrier waits (seconds at most)
constexpr int BM = 128, BK = 64;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// TMA store of a 32 x 32 FP32 box (128-byte swizzled rows in shared memory) at column x, row y of
// the output; rows and columns beyond the tensor are not written. x is a multiple of 32 (128 bytes).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"((uint64_t)map),
                 "r"(src), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until at most one committed store group still reads shared memory
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void st_shared_v4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// shared-memory matrix descriptor, K-major operand with 128-byte swizzle: 8-row groups of
// 128-byte rows, 1024 bytes apart (stride byte offset); leading offset unused for this layout
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1u << 46;          // descriptor version of the 5th-generation tensor core
    d |= (uint64_t)2u << 61;          // 128-byte swizzle
    return d;
}

// instruction descriptor of kind::f16: BF16 A and B (K-major), FP32 accumulator, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32-byte vector accesses (addresses multiples of 32)
__device__ __forceinline__ void ld_v8(const float* p, float* v) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}
__device__ __forceinline__ void st_v8(void* p, const float* v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.3989422804014327f;
}

// FP32 epilogues of one accumulator value at (row, col), inside M x N
__device__ __forceinline__ void epilogue(const GemmEpi& e, int row, int col, float acc, size_t zoff) {
    e.out_f32[zoff + (size_t)row * e.ld_out + col] = e.kind == kEpiExp ? expf(acc) : acc + (e.bias ? e.bias[col] : 0.0f);
}

template <int BN, int STAGES>
__global__ void __launch_bounds__(128, 3)
umma_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmC, int M, int N, int K, int cps, GemmEpi epi, int* err) {
    constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    // split K (cps > 0): this CTA takes the K chunks [kb, kb + nk) and writes its partial product
    // to slice blockIdx.z of the output (a workspace the caller reduces)
    const int nk_all = (K + BK - 1) / BK;
    const int kb = cps > 0 ? (int)blockIdx.z * cps : 0;
    const int nk = cps > 0 ? min(cps, nk_all - kb) : nk_all;
    const size_t zoff = (size_t)blockIdx.z * (size_t)M * (size_t)epi.ld_out;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&done_bar), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"((uint32_t)BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    grid_wait();   // barriers and tensor memory are set up while the predecessor ends
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    if (threadIdx.x == 0) {
        // producer: TMA loads of chunk k into slot k % STAGES once the MMAs of chunk k - STAGES are done
        for (int k = 0; k < nk; ++k) {
            const int s = k % STAGES;
            if (k >= STAGES && !mbar_wait(smem_u32(&empty_bar[s]), ((k / STAGES) - 1) & 1)) {
                atomicExch(&abort_flag, 1);
                break;
            }
            if (*(volatile int*)&abort_flag) break;
            const uint32_t a_dst = base + s * STAGE_BYTES, b_dst = a_dst + A_BYTES;
            mbar_expect_tx(smem_u32(&full_bar[s]), STAGE_BYTES);
            tma_load_2d(a_dst, &tmA, smem_u32(&full_bar[s]), (kb + k) * BK, m0);
            tma_load_2d(b_dst, &tmB, smem_u32(&full_bar[s]), (kb + k) * BK, n0);
        }
    } else if (threadIdx.x == 32) {
        // issuer: four K = 16 MMAs per chunk; the start address advances 32 bytes per step
        constexpr uint32_t idesc = idesc_bf16(BM, BN);
        bool ok = true;
        for (int k = 0; k < nk; ++k) {
            const int s = k % STAGES;
            if (!mbar_wait(smem_u32(&full_bar[s]), (k / STAGES) & 1)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a_src = base + s * STAGE_BYTES, b_src = a_src + A_BYTES;
#pragma unroll
            for (int j = 0; j < BK / 16; ++j)
                umma_bf16(tmem, sw128_desc(a_src + 32 * j), sw128_desc(b_src + 32 * j), idesc, (k | j) != 0);
            umma_commit(smem_u32(&empty_bar[s]));
        }
        if (ok) umma_commit(smem_u32(&done_bar));
        else atomicExch(&abort_flag, 1);
    }
    __syncwarp();

    // epilogue: warp w owns TMEM lanes (tile rows) 32w .. 32w + 31
    // (the vote brings the lanes together again: tensor memory is read by whole warps, .sync.aligned)
    const bool done = __all_sync(0xffffffffu, mbar_wait(smem_u32(&done_bar), 0));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (done) {
        const uint32_t t_row = tmem + ((uint32_t)(32 * warp) << 16);
        if (epi.tma_out) {
            // FP32 output (exp applied, or stored as is) by TMA: each lane holds one row of a 32 x 32
            // block, writes it as eight 16-byte chunks into a 128-byte swizzled staging row (chunk c
            // of row r at c ^ (r & 7): a warp's chunk stores spread over all banks), and lane 0 stores
            // the block with one bulk copy. Two staging buffers per warp in the free pipeline slots,
            // so a block is written while the previous one is still being read.
            const uint32_t stage0 = base + (uint32_t)warp * 8192u;
            int buf = 0;
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 32, buf ^= 1) {
                float v[32];
                tmem_ld32(t_row + (uint32_t)c0, v);
                if (epi.kind == kEpiExp) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = expf(v[i]);
                }
                const uint32_t sb = stage0 + (uint32_t)buf * 4096u;
                if (lane == 0) bulk_wait_read1();   // the store issued from this buffer two blocks ago
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    st_shared_v4(sb + (uint32_t)lane * 128u + ((uint32_t)(c ^ (lane & 7)) << 4), v[4 * c],
                                 v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                // boxes reaching past the output are clipped by the copy; boxes wholly past it are skipped
                if (lane == 0 && n0 + c0 < N && m0 + 32 * warp < M) {
                    tma_store_2d(&tmC, sb, n0 + c0, m0 + 32 * warp);
                    bulk_commit();
                }
            }
            if (lane == 0) bulk_wait_all();
            __syncwarp();
        } else if (epi.kind == kEpiStoreF32 || epi.kind == kEpiExp) {
            // 32 x 32 blocks staged through shared memory (the pipeline slots are free now): each
            // lane holds one row, then each store instruction writes 32 consecutive columns of one row
            float* stage = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw))) + warp * (32 * 33);
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 32) {
                float v[32];
                tmem_ld32(t_row + (uint32_t)c0, v);
#pragma unroll
                for (int i = 0; i < 32; ++i) stage[lane * 33 + i] = v[i];
                __syncwarp();
                const int col = n0 + c0 + lane;
#pragma unroll 4
                for (int rr = 0; rr < 32; ++rr) {
                    const int row = m0 + 32 * warp + rr;
                    if (row < M && col < N) epilogue(epi, row, col, stage[rr * 33 + lane], zoff);
                }
                __syncwarp();
            }
        } else {
            // bias + GELU (forward) and GELU' (input gradient), N a multiple of 32: a lane holds 32
            // consecutive columns of its row and works on them in registers (32 independent chains). Row-major
            // operands move as 32-byte vectors, whole sectors; the transposed copy is 32 consecutive rows per
            // store instruction as it is. (Staging 32 x 32 blocks through shared memory twice, one column per
            // lane, left a chain of erf per shared-memory read on two warps a scheduler: 19 us forward and 28 us
            // backward per 8192 x 256 x 256 product, now 11 and 12 us.)
            const int row = m0 + 32 * warp + lane;
            const bool in = row < M;
            // rows past the end read the last one: a branch here could leave the warp apart at tmem_ld32
            const float* pre_in =
                epi.kind == kEpiGeluBackward ? epi.pre_in + (size_t)min(row, M - 1) * epi.ld_pre : nullptr;
#pragma unroll 1
            for (int c0 = 0; c0 < BN && n0 + c0 < N; c0 += 32) {
                const int col = n0 + c0;
                float x[32], v[32];
                if (epi.kind == kEpiBiasGelu) {
#pragma unroll
                    for (int i = 0; i < 32; i += 8) ld_v8(epi.bias + col + i, x + i);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; i += 8) ld_v8(pre_in + col + i, x + i);
                }
                tmem_ld32(t_row + (uint32_t)c0, v);
                if (epi.kind == kEpiBiasGelu) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] += x[i];
                    if (epi.pre && in) {
#pragma unroll
                        for (int i = 0; i < 32; i += 8) st_v8(epi.pre + (size_t)row * epi.ld_pre + col + i, v + i);
                    }
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = gelu_f(v[i]);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] *= gelu_grad_f(x[i]);
                }
                __nv_bfloat162 h[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    h[i] = __nv_bfloat162(__float2bfloat16_rn(v[2 * i]), __float2bfloat16_rn(v[2 * i + 1]));
                if (in) {
                    __nv_bfloat16* act = epi.act + (size_t)row * epi.ld_act + col;
                    st_v8(act, reinterpret_cast<const float*>(h));
                    st_v8(act + 16, reinterpret_cast<const float*>(h + 8));
                    if (epi.act_t) {
                        __nv_bfloat16* at = epi.act_t + (size_t)col * epi.ld_act_t + row;
#pragma unroll
                        for (int i = 0; i < 32; ++i) at[(size_t)i * epi.ld_act_t] = i & 1 ? h[i / 2].y : h[i / 2].x;
                    }
                }
                __syncwarp();   // the warp reads tensor memory together
            }
        }
    } else if (lane == 0) {
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
    }
}

// out[r][c] = sum over the splits z = 0 .. splits - 1 (in order) of ws[z][r][c], rows r < M,
// columns c < N, row stride ld in both. Bound by the latency of the loads: 16 are in flight per thread,
// and blocks of at most 128 threads (one row each) reach every SM (256 x 256 outputs of 19 splits:
// 7.4 us in flat blocks of 256 with eight loads in flight, now 6.1 us; 256 x 64 of 64 splits: 13.1,
// now 10.3 us).
constexpr int kReduceThreads = 128;
__global__ void __launch_bounds__(kReduceThreads) splitk_reduce_kernel(const float* ws, int splits, int M, int N, int ld,
                                                                       float* out) {
    grid_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const size_t i = (size_t)blockIdx.y * ld + c, slice = (size_t)M * ld;
    float acc = 0.0f;
#pragma unroll 16
    for (int z = 0; z < splits; ++z) acc += ws[(size_t)z * slice + i];   // in split order
    out[i] = acc;
}

// ---- host side -------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// 2-D BF16 tensor map: rows x cols (cols contiguous, row stride ld elements), box 64 x box_rows
bool make_map(CUtensorMap* map, const void* ptr, int rows, int cols, int ld, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    if (((uintptr_t)ptr & 15u) != 0 || (ld * 2) % 16 != 0) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// 2-D FP32 tensor map of an output: rows x cols (row stride ld elements), box 32 x 32, 128-byte
// swizzle (the epilogue's staging layout)
bool make_out_map(CUtensorMap* map, const void* ptr, int rows, int cols, int ld) {
    auto fn = encode_fn();
    if (!fn) return false;
    if (((uintptr_t)ptr & 15u) != 0 || (ld * 4) % 16 != 0) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
    cuuint32_t box[2] = {32, 32};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// encoded maps of this thread, keyed by everything a map encodes (address, shape, stride, box):
// a key fully determines its map, so entries never go stale
struct MapKey {
    const void* ptr;
    int rows, cols, ld, box_rows;   // box_rows < 0: an FP32 output map (make_out_map)
    bool operator==(const MapKey& o) const {
        return ptr == o.ptr && rows == o.rows && cols == o.cols && ld == o.ld && box_rows == o.box_rows;
    }
};
struct MapKeyHash {
    size_t operator()(const MapKey& k) const {
        size_t h = std::hash<const void*>()(k.ptr);
        for (int v : {k.rows, k.cols, k.ld, k.box_rows}) h = h * 1000003u ^ (size_t)(unsigned)v;
        return h;
    }
};

bool cached_map(CUtensorMap* map, const void* ptr, int rows, int cols, int ld, int box_rows) {
    thread_local std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
    const MapKey key{ptr, rows, cols, ld, box_rows};
    auto it = cache.find(key);
    if (it != cache.end()) {
        *map = it->second;
        return true;
    }
    if (!(box_rows < 0 ? make_out_map(map, ptr, rows, cols, ld) : make_map(map, ptr, rows, cols, ld, box_rows)))
        return false;
    if (cache.size() >= 512) cache.clear();
    cache.emplace(key, *map);
    return true;
}

template <int BN, int STAGES>
cudaError_t launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tc, int M, int N, int K,
                        int splits, int cps, const GemmEpi& epi, int* err, cudaStream_t st) {
    const size_t smem = (size_t)STAGES * (BM * BK * 2 + BN * BK * 2) + 1024;
    auto kern = umma_gemm_kernel<BN, STAGES>;
    static std::atomic<unsigned long long> attr_set{0};   // one bit per device
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(attr_set.load() & bit)) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_set.fetch_or(bit);
    }
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, splits);
    const cudaError_t e = launch_after(kern, grid, dim3(128), smem, st, ta, tb, tc, M, N, K, cps, epi, err);
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t umma_gemm(const void* A, int lda, const void* B, int ldb, int M, int N, int K, const GemmEpi& epi,
                      int* err, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (epi.kind == kEpiBiasGelu || epi.kind == kEpiGeluBackward) {
        // the GELU epilogues' 32-byte vectors (the network's hidden layers: 256 wide, rows of 256)
        const bool fwd = epi.kind == kEpiBiasGelu;
        const void* f32s[2] = {fwd ? (const void*)epi.bias : (const void*)epi.pre_in, fwd ? (const void*)epi.pre : nullptr};
        if (N % 32 != 0 || epi.ld_act % 16 != 0 || epi.ld_pre % 8 != 0 || ((uintptr_t)f32s[0] & 31u) != 0 ||
            ((uintptr_t)f32s[1] & 31u) != 0 || ((uintptr_t)epi.act & 31u) != 0)
            return cudaErrorInvalidValue;
    }
    // 128-wide output tiles, or 64-wide ones where 128-wide tiles would leave SMs without one (the
    // surrogate's 256-wide layers: 128 tiles of 128 x 128 at a minibatch of 8192 against 256 of
    // 128 x 64, whose GELU epilogues then run on twice the warps)
    int bn = N <= 64 ? 64 : 128;
    if (bn == 128 && (long long)((N + 127) / 128) * ((M + BM - 1) / BM) < 152) bn = 64;
    CUtensorMap ta, tb, tc;
    if (!cached_map(&ta, A, M, K, lda, BM) || !cached_map(&tb, B, N, K, ldb, bn)) return cudaErrorInvalidValue;
    GemmEpi e2 = epi;
    e2.tma_out = 0;
    std::memset(&tc, 0, sizeof tc);
    // split K: a plain FP32 product with few output tiles and a long K (the surrogate's weight
    // gradients: 256 x 256 outputs over a minibatch of thousands) runs on about a CTA per SM, each
    // split writing its partial tile to the caller's workspace, then summed in split order
    const int tiles = ((N + bn - 1) / bn) * ((M + BM - 1) / BM), nk = (K + BK - 1) / BK;
    int splits = 1, cps = 0;
    if (epi.kind == kEpiStoreF32 && !epi.bias && epi.ws && tiles < 38 && nk >= 8) {
        const size_t slice = (size_t)M * epi.ld_out;
        const int max_splits = (int)std::min<size_t>(epi.ws_floats / slice, 1024);
        if (max_splits >= 2) {
            cps = std::max(2, (nk * tiles + 151) / 152);
            cps = std::max(cps, (nk + max_splits - 1) / max_splits);
            splits = (nk + cps - 1) / cps;
            if (splits < 2) splits = 1, cps = 0;
        }
    }
    if (splits > 1) {
        e2.out_f32 = epi.ws;
        cudaError_t e = bn == 64 ? launch_gemm<64, 2>(ta, tb, tc, M, N, K, splits, cps, e2, err, st)
                                 : launch_gemm<128, 2>(ta, tb, tc, M, N, K, splits, cps, e2, err, st);
        if (e != cudaSuccess) return e;
        const int threads = std::min(kReduceThreads, (N + 31) / 32 * 32);   // M < 38 tiles of 128 rows
        e = launch_after(splitk_reduce_kernel, dim3((N + threads - 1) / threads, M), dim3(threads), 0, st, epi.ws, splits, M,
                         N, epi.ld_out, epi.out_f32);
        count_launches(1);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    // FP32 outputs without a bias (the KL synthesis) leave by TMA stores when their map encodes
    if ((epi.kind == kEpiExp || (epi.kind == kEpiStoreF32 && !epi.bias)) && cached_map(&tc, epi.out_f32, M, N, epi.ld_out, -1))
        e2.tma_out = 1;
    // two stages (65 KB of shared memory): three CTAs per SM, so that one CTA's epilogue overlaps
    // the loads and MMAs of the others (the contractions here have short K)
    if (bn == 64) return launch_gemm<64, 2>(ta, tb, tc, M, N, K, 1, 0, e2, err, st);
    return launch_gemm<128, 2>(ta, tb, tc, M, N, K, 1, 0, e2, err, st);
}

}  // namespace mls2mc

extern "C" int smc_gemm_bf16(int M, int N, int K, const uint16_t* A, const uint16_t* B, float* C) {
    using namespace mls2mc;
    if (M <= 0 || N <= 0 || K <= 0 || K % 8 != 0 || !A || !B || !C) return SMC_EINVAL;
    void *dA = nullptr, *dB = nullptr;
    float* dC = nullptr;
    int* dErr = nullptr;
    cudaError_t e = cudaMalloc(&dA, (size_t)M * K * 2);
    if (e == cudaSuccess) e = cudaMalloc(&dB, (size_t)N * K * 2);
    if (e == cudaSuccess) e = cudaMalloc((void**)&dC, (size_t)M * N * 4);
    if (e == cudaSuccess) e = cudaMalloc((void**)&dErr, 4);
    if (e == cudaSuccess) e = cudaMemcpy(dA, A, (size_t)M * K * 2, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dB, B, (size_t)N * K * 2, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(dErr, 0, 4);
    GemmEpi epi;
    epi.kind = kEpiStoreF32;
    epi.out_f32 = dC;
    epi.ld_out = N;
    if (e == cudaSuccess) e = umma_gemm(dA, K, dB, K, M, N, K, epi, dErr, nullptr);
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpy(C, dC, (size_t)M * N * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&herr, dErr, 4, cudaMemcpyDeviceToHost);
    cudaFree(dA);
    cudaFree(dB);
    cudaFree(dC);
    cudaFree(dErr);
    if (e != cudaSuccess) return SMC_ECUDA;
    return herr ? SMC_ETIMEOUT : SMC_OK;
}
