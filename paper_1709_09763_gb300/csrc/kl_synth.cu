// KL synthesis on the tensor cores (mixed path): kappa[j][e] = exp(sum_k theta_jk Psi_ke)
// (Sec. 5, Eq. truncKL, kappa = exp(u)).
//
// The contraction particles x K by K x triangles runs as one BF16 GEMM with FP32 accumulation.
// To keep u at FP32 accuracy, theta and Psi are each split into three BF16 pieces
// (x = x1 + x2 + x3, each piece the BF16 rounding of what the previous ones left), and the six
// cross products whose size is above 2^-24 relative are concatenated along K, smallest first:
// (2,2), (1,3), (3,1), (1,2), (2,1), (1,1), i.e. A' = [t2 t1 t3 t1 t2 t1], B' = [P2 P3 P1 P2 P1 P1],
// K' = 6K (padded to a multiple of 8 with zeros). The accumulator then stays small while the small
// products enter and the truncation of its last steps acts at the size of u only: measured on the
// GB300, G within 5.3e-8 of the FP64 oracle for 32 terms (1/16 .. 1/64) and 2.9e-8 for the 320-term
// flow cell (1/16, 1/32), against 2.6e-7 and 1.8e-7 with the largest products first. The epilogue
// applies exp and writes kappa as FP32 [n][E], which the solve kernel reads instead of forming u
// itself.
//
// Expansions beyond 256 terms are synthesised in groups of 64. The error of u from the tensor cores'
// FP32 accumulation follows a round-toward-zero model of the accumulator, one rounding per K = 16
// step (measured: at K = 320 the G errors of a single 1920-wide contraction correlate 1.00 with
// that model and reach 1.6e-6), which shrinks |u| systematically. One contraction stays within
// 1e-6 up to K = 256 (measured at 256 and 128 terms); beyond, each group of 64 terms is its own
// GEMM (the layout above, per group) into an FP32 partial, and the partials are summed in FP64
// before exp (measured at K = 320 on 1/16: G within 3.0e-7; the model gave 2.7e-7).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <cstdint>
#include <vector>

#include "handle.h"
#include "launch.h"
#include "smc_device.h"
#include "umma_gemm.h"

namespace mls2mc {

namespace {

// theta split of the Kg terms starting at k0 (the whole expansion, or one group of it): out [n][Kp].
// A thread takes V = 2 neighbouring terms of a particle (1 where Kg is odd, for the alignment of the
// 4-byte stores): theta is read and converted once (a conversion from FP64 is an FP64 instruction, at
// 64 cycles a warp) instead of once for each of the six blocks, and the block is kx x ry threads over
// terms and particles, so no index is divided. Bound by launch and memory latency: 5.9 us at
// 4000 x 32 with a thread per output and its 64-bit division, now 3.5 us.
constexpr int kSplitThreads = 128;

// the split of one particle's terms th into its row, by threads x = 0 .. kx - 1
template <int V>
__device__ __forceinline__ void split_row(const double* th, int Kg, int Kp, int x0, int kx, __nv_bfloat16* row) {
    for (int k = x0 * V; k < Kg; k += kx * V) {
        __nv_bfloat16 p1[V], p2[V], p3[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            // theta rounded to FP32 (24 bits, all that three BF16 pieces carry); each remainder is
            // exact in FP32, so no FP64 arithmetic is needed
            const float x = (float)th[k + i];
            p1[i] = __float2bfloat16_rn(x);
            const float r1 = x - __bfloat162float(p1[i]);
            p2[i] = __float2bfloat16_rn(r1);
            const float r2 = r1 - __bfloat162float(p2[i]);
            p3[i] = __float2bfloat16_rn(r2);
        }
        // A' blocks: t2 t1 t3 t1 t2 t1
        const __nv_bfloat16* const sel[6] = {p2, p1, p3, p1, p2, p1};
#pragma unroll
        for (int b = 0; b < 6; ++b) {
            __nv_bfloat16* o = row + b * Kg + k;
            if constexpr (V == 2)
                *reinterpret_cast<__nv_bfloat162*>(o) = __nv_bfloat162(sel[b][0], sel[b][1]);
            else
                *o = sel[b][0];
        }
    }
    for (int c = 6 * Kg + x0; c < Kp; c += kx) row[c] = __float2bfloat16_rn(0.0f);
}

template <int V>
__global__ void __launch_bounds__(kSplitThreads)
    theta_split_kernel(const double* theta, int n, int K, int k0, int Kg, int Kp, __nv_bfloat16* out, int* ticket) {
    grid_wait();
    if (ticket && blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) *ticket = 0;
    const long long j = (long long)blockIdx.x * blockDim.y + threadIdx.y;
    if (j < n)
        split_row<V>(theta + (size_t)j * K + k0, Kg, Kp, (int)threadIdx.x, (int)blockDim.x, out + (size_t)j * Kp);
}

// many problems' splits: blockIdx.y is the problem, the blocks in x stride over its particles
__global__ void __launch_bounds__(kSplitThreads) theta_split_multi_kernel(const __grid_constant__ SplitTasks L) {
    const SplitTask& t = L.t[blockIdx.y];
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(t.out);
    const bool pair = t.K % 2 == 0;
    const int kx = min(pair ? t.K / 2 : t.K, kSplitThreads), ry = kSplitThreads / kx;
    const int x = (int)threadIdx.x % kx, y = (int)threadIdx.x / kx;
    if (y >= ry) return;
    for (long long j = (long long)blockIdx.x * ry + y; j < t.n; j += (long long)gridDim.x * ry) {
        if (pair) split_row<2>(t.theta + (size_t)j * t.K, t.K, t.Kp, x, kx, out + (size_t)j * t.Kp);
        else split_row<1>(t.theta + (size_t)j * t.K, t.K, t.Kp, x, kx, out + (size_t)j * t.Kp);
    }
}

void theta_split_launch(const double* theta, int n, int K, int k0, int Kg, int Kp, __nv_bfloat16* out, int* ticket,
                        cudaStream_t st) {
    const int terms = Kg % 2 == 0 ? Kg / 2 : Kg;
    const int kx = std::min(terms, kSplitThreads), ry = kSplitThreads / kx;
    const dim3 block(kx, ry);
    const unsigned grid = (unsigned)(((long long)n + ry - 1) / ry);
    launch_after(Kg % 2 == 0 ? theta_split_kernel<2> : theta_split_kernel<1>, grid, block, 0, st, theta, n, K, k0, Kg, Kp,
                 out, ticket);
    count_launches(1);
}

// kappa[t] = exp(sum over groups of part[g][t]), the sum and exp in FP64
__global__ void sum_exp_kernel(const float* part, int groups, long long nE, float* kappa) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nE; t += stride) {
        double u = 0.0;
        for (int g = 0; g < groups; ++g) u += (double)part[(size_t)g * nE + t];
        kappa[t] = (float)exp(u);
    }
}

constexpr int kSynthGroup = 64;     // terms per accumulation of a grouped synthesis
constexpr int kSingleMax = 256;     // up to this many terms: one contraction (measured within 1e-6)

// terms of group g (the whole expansion when it is synthesised in one contraction)
int group_terms(int K, int g) {
    if (K <= kSingleMax) return K;
    return K - g * kSynthGroup < kSynthGroup ? K - g * kSynthGroup : kSynthGroup;
}

uint16_t bf16_bits_host(double x) {
    const __nv_bfloat16 b = __float2bfloat16_rn((float)x);
    uint16_t u;
    std::memcpy(&u, &b, 2);
    return u;
}

double bf16_value_host(uint16_t u) {
    uint32_t w = (uint32_t)u << 16;
    float f;
    std::memcpy(&f, &w, 4);
    return (double)f;
}

}  // namespace

int kl_split_width(int K) { return (6 * K + 7) / 8 * 8; }

int kl_groups(int K) { return K <= kSingleMax ? 1 : (K + kSynthGroup - 1) / kSynthGroup; }

int kl_split_total(int K) {
    int s = 0;
    for (int g = 0; g < kl_groups(K); ++g) s += kl_split_width(group_terms(K, g));
    return s;
}

// B' = [P2 P3 P1 P2 P1 P1] as BF16 bits, per group of terms an [E][Kp] block (K-major rows, one
// per triangle), the groups one after the other (one group, the whole table, for K <= 256)
std::vector<uint16_t> kl_split_table(const std::vector<double>& psi, int K, int E) {
    std::vector<uint16_t> out((size_t)E * kl_split_total(K), 0);
    size_t base = 0;
    for (int g = 0; g < kl_groups(K); ++g) {
        const int k0 = g * kSynthGroup, Kg = group_terms(K, g), Kp = kl_split_width(Kg);
        for (int e = 0; e < E; ++e)
            for (int k = 0; k < Kg; ++k) {
                const double x = psi[(size_t)(k0 + k) * E + e];
                const uint16_t p1 = bf16_bits_host(x);
                const double r1 = x - bf16_value_host(p1);
                const uint16_t p2 = bf16_bits_host(r1);
                const double r2 = r1 - bf16_value_host(p2);
                const uint16_t p3 = bf16_bits_host(r2);
                const uint16_t sel[6] = {p2, p3, p1, p2, p1, p1};
                for (int b = 0; b < 6; ++b) out[base + (size_t)e * Kp + b * Kg + k] = sel[b];
            }
        base += (size_t)E * Kp;
    }
    return out;
}

// grow the synthesis buffers to hold n particles on `level` (no launch); a no-op when they do
int Handle::synth_reserve(int level, int n) {
    const Level& L = levels[level];
    const int E = 2 * L.N * L.N, Kt = kl_split_total(K), G = kl_groups(K);
    const size_t need_k = (size_t)n * E, need_t = (size_t)n * Kt;
    if (need_k > synth_kappa_cap || need_t > synth_theta_cap) {
        // both buffers grow to at least their previous size: alternating shapes never shrink them
        const size_t cap_k = std::max(need_k, synth_kappa_cap), cap_t = std::max(need_t, synth_theta_cap);
        cudaFree(synth_kappa_buf);
        cudaFree(synth_theta_buf);
        synth_kappa_buf = nullptr;
        synth_theta_buf = nullptr;
        synth_kappa_cap = synth_theta_cap = 0;
        cudaError_t e = cudaMalloc((void**)&synth_kappa_buf, cap_k * 4);
        if (e == cudaSuccess) e = cudaMalloc((void**)&synth_theta_buf, cap_t * 2);
        if (e != cudaSuccess) return fail(SMC_ENOMEM, "synthesis buffers for %d particles: %s", n, cudaGetErrorString(e));
        synth_kappa_cap = cap_k;
        synth_theta_cap = cap_t;
    }
    const size_t need_p = G > 1 ? (size_t)G * n * E : 0;   // FP32 partials of the term groups
    if (need_p > synth_part_cap) {
        cudaFree(synth_part_buf);
        synth_part_buf = nullptr;
        synth_part_cap = 0;
        cudaError_t e = cudaMalloc((void**)&synth_part_buf, need_p * 4);
        if (e != cudaSuccess) return fail(SMC_ENOMEM, "synthesis partials for %d particles: %s", n, cudaGetErrorString(e));
        synth_part_cap = need_p;
    }
    if (!synth_err) {
        cudaError_t e = cudaMalloc((void**)&synth_err, 4);
        if (e == cudaSuccess) e = cudaMemset(synth_err, 0, 4);
        if (e != cudaSuccess) return fail(SMC_ENOMEM, "synthesis flag");
    }
    return SMC_OK;
}

cudaError_t theta_split_multi_launch(const std::vector<SplitTask>& tasks, cudaStream_t st) {
    SplitTasks L;
    for (size_t i0 = 0; i0 < tasks.size(); i0 += kMaxTasks) {
        L.count = (int)std::min<size_t>(kMaxTasks, tasks.size() - i0);
        int blocks = 1;
        for (int i = 0; i < L.count; ++i) {
            L.t[i] = tasks[i0 + i];
            const int terms = L.t[i].K % 2 == 0 ? L.t[i].K / 2 : L.t[i].K, ry = kSplitThreads / std::min(terms, kSplitThreads);
            blocks = std::max(blocks, std::min(64, (int)(((long long)L.t[i].n + ry - 1) / ry)));
        }
        theta_split_multi_kernel<<<dim3(blocks, L.count), kSplitThreads, 0, st>>>(L);
        count_launches(1);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int Handle::synth_kappa(int level, int n, const double* theta, cudaStream_t st, bool split, int* ticket) {
    const Level& L = levels[level];
    const int E = 2 * L.N * L.N, Kt = kl_split_total(K), G = kl_groups(K);
    RC_CHECK(synth_reserve(level, n));
    if (G == 1) {
        if (split)
            theta_split_launch(theta, n, K, 0, K, Kt, reinterpret_cast<__nv_bfloat16*>(synth_theta_buf), ticket, st);
        GemmEpi epi;
        epi.kind = kEpiExp;
        epi.out_f32 = synth_kappa_buf;
        epi.ld_out = E;
        cudaError_t e = umma_gemm(synth_theta_buf, Kt, L.psi_split, Kt, n, E, Kt, epi, synth_err, st);
        if (e != cudaSuccess) return cuda_fail(e, "KL synthesis GEMM");
        return SMC_OK;
    }
    size_t off_t = 0, off_b = 0;   // group offsets in the theta split and in the table (elements)
    for (int g = 0; g < G; ++g) {
        const int Kg = group_terms(K, g), Kp = kl_split_width(Kg);
        theta_split_launch(theta, n, K, g * kSynthGroup, Kg, Kp, reinterpret_cast<__nv_bfloat16*>(synth_theta_buf + off_t),
                           ticket, st);
        GemmEpi epi;
        epi.kind = kEpiStoreF32;
        epi.out_f32 = synth_part_buf + (size_t)g * n * E;
        epi.ld_out = E;
        cudaError_t e = umma_gemm(synth_theta_buf + off_t, Kp, L.psi_split + off_b, Kp, n, E, Kp, epi, synth_err, st);
        if (e != cudaSuccess) return cuda_fail(e, "KL synthesis GEMM of a term group");
        off_t += (size_t)n * Kp;
        off_b += (size_t)E * Kp;
    }
    const long long nE = (long long)n * E;
    const int blocks = (int)std::min<long long>((nE + 255) / 256, 152LL * 8);
    sum_exp_kernel<<<blocks, 256, 0, st>>>(synth_part_buf, G, nE, synth_kappa_buf);
    count_launches(1);
    return SMC_OK;
}

}  // namespace mls2mc
