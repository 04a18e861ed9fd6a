// Register-tiled form of the mixed-precision forward solve on 1/32 .. 1/256 (Dirichlet problem).
//
// The algorithm is the one of fem_solve.cu (KL field -> kappa -> 5-point stencil -> CG with a
// V(1,1) red-black multigrid preconditioner, double-float refinement, observations, misfit); what
// differs is who owns what. A thread owns a 4 x 4 patch of fine nodes and keeps the patch's CG
// residual r, sweep values e and all 40 edge weights in registers; only the patch's rim goes through
// shared memory. The 2 x 2 nodes of the next level that lie under the patch belong to the same thread, so
// restriction and prolongation mostly stay in registers as well. The levels below (1/8 of a 1/32 mesh, 1/16 of
// a 1/64 mesh, 1/32 of the larger ones) are solved as whole grids, two nodes per thread, 1/8 and 1/4 in warp 0.
//
// Shared-memory layout: one array per position of the patch, indexed by thread ("position-major"),
// X[(4 b + a) S + q] for node (4 tx + a, 4 ty + b) of patch q. A read of one's own or a neighbouring patch's
// position is 32 consecutive words for a warp: no bank conflicts. The arrays have one more row of patches
// below and above, so a neighbour is an immediate offset. Node column 0 and row 0 are Dirichlet nodes whose
// stored values are always 0 (their inverse diagonal is 0), so the node to the right of column N - 1 may be read
// as the next row's column 0; what is read to the left of column 0 is only ever used by Dirichlet nodes, whose
// results are masked.
//
// 1/128 and 1/256 spread one particle over a cluster of two or eight CTAs of 512 threads, one CTA an SM, each
// with a band of patch rows. The extra rows of the exchange arrays are then the neighbour CTAs' border
// rows, written by them through distributed shared memory; every phase that others read ends at a
// cluster barrier (660 cycles; stores that complete on the receiver's mbarrier instead came to 540, so the
// barriers stay). The two finest levels (three on 1/256) are distributed, 1/32 and below are solved by every
// CTA from a right-hand side that each CTA writes into all of them.
//
// Why this split: with one node per register slot and everything else in shared memory (the form of
// fem_solve.cu) a node update reads nine words from shared memory, 21 block barriers an iteration; that
// form (two 512-thread blocks an SM on 1/64) took 1.99 ms for 4000 particles on 1/64 and 0.42 ms on
// 1/32. Here a patch of 16 nodes reads 8 rim words per half sweep, 18 barriers an iteration (1/32: 13), 256
// threads of 128 registers, two blocks an SM (1/64) or 64 threads, eight blocks (1/32): 0.78 ms and 0.18 ms. On
// 1/128 (8000 particles) one node per slot on two CTAs of 1024 threads took 31.5 ms, this form 13.1 ms; on
// 1/256 (1001 particles) the fine levels in device memory took 34.2 ms, this form 13.2 ms.
// What bounds it is latency: one 1/64 particle alone on an SM takes 0.87 of the time that two take
// together. A spill is what hurts most: the direction p lives in shared memory and addresses are formed
// where they are used, so that (but for a dozen words around the whole levels in the cluster forms) no register is
// spilled in the iteration (1/64: 0.86 ms with a 20-word spill).
// The flow cell's solve is not in this form, to keep its bits: its observations move by 7e-9 with the order of the
// dot products (a solve in a thousand then stops one iteration earlier or later, a large step there).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "fem_device.h"
#include "internal.h"
#include "launch.h"

namespace mls2mc {

namespace {

// geometry of one form: 1/N on a cluster of C CTAs, each owning R rows of patches
template <int N_, int C_>
struct Geo {
    static constexpr int N = N_, C = C_, TX = N / 4;
    static constexpr bool H = C > 1;
    static constexpr int R = N / 4 / C;
    static constexpr int T = TX * R, NW = T / 32;
    static constexpr bool L2 = N == 256;         // a distributed one-node-per-thread level (1/64)
    // the fine inverse diagonals are correctly rounded and in shared memory; on 1/128 there is no room for them and the
    // sweeps form approximate ones, as that level always has. On 1/256 they take the place of the CG correction d,
    // which is in device memory there (read and written once an iteration). 1001 particles: 13.53 ms; 12.99 with
    // approximate ones, 13.98 with them and not d in device memory, 14.97 with a rounded reciprocal in the sweeps
    static constexpr bool STORED = N != 128, DG = N == 256;
    static constexpr int TOP = L2 ? N / 8 : N / 4;   // finest level that every CTA solves as a whole
    // blocks per SM: registers for 128 a thread
    static constexpr int MINB = 65536 / (128 * T);
    // exchange arrays have a row of patches below and one above the CTA's own: the neighbour CTAs', or 0;
    // and, as the node above right of the last patch, a 0 (padded to 16 bytes)
    static constexpr int S = T + 2 * TX + 4;
    // ---- shared memory, in floats ----
    static constexpr int E = 0;              // sweep values, later p or d: rim positions [16][S]; the
                                             // inner positions' slots carry red residuals
    static constexpr int D = E + 16 * S;     // CG correction d, float4 [4][T] (unless DG)
    static constexpr int PV = D + 16 * T;    // CG direction p, float4 [4][T] (not in registers during the V-cycle)
    static constexpr int ID = DG ? D : PV + 16 * T;   // fine inverse diagonals, float4 [red 2, black 2][T]
    // next level: weights (E, W, N, S) of (0,0) (1,1) (1,0) (0,1)
    static constexpr int W1 = PV + 16 * T + (STORED && !DG ? 16 * T : 0);
    static constexpr int WH = W1 + 16 * T;   // those of (1,1) in the row of patches below this CTA, float4 [TX]
    static constexpr int E1 = WH + 4 * TX;   // its values [4][S], positions A + 2 B
    // its right-hand side, float4 [T], out of registers while the levels below run on a cluster's CTAs
    static constexpr bool VS = H;
    static constexpr int V1 = E1 + 4 * S;
    // distributed 1/64 (on 1/256): weights, inverse diagonal, values
    static constexpr int W2 = V1 + (VS ? 4 * T : 0);
    static constexpr int ID2 = W2 + (L2 ? 4 * T : 0);
    static constexpr int E2 = ID2 + (L2 ? T : 0);
    static constexpr int RR = E2 + (L2 ? S : 0);   // red residuals of the whole level [2 TOP][2 TOP]
    __host__ __device__ static constexpr int nodes(int M) { return M * M; }
    // whole levels M = TOP .. 8: weights float4, inverse diagonal, values, right-hand side or residual
    static constexpr int LV = RR + (L2 ? nodes(2 * TOP) : 0);
    __host__ __device__ static constexpr int lv(int M) { return M == TOP ? LV : lv(2 * M) + 7 * nodes(2 * M); }
    __host__ __device__ static constexpr int lw(int M) { return lv(M); }
    __host__ __device__ static constexpr int lid(int M) { return lv(M) + 4 * nodes(M); }
    __host__ __device__ static constexpr int le(int M) { return lv(M) + 5 * nodes(M); }
    __host__ __device__ static constexpr int lr(int M) { return lv(M) + 6 * nodes(M); }
    static constexpr int ND = 9;             // unknowns of 1/4: values [4][4], rhs, dense inverse
    static constexpr int E4 = lv(8) + 7 * nodes(8);
    static constexpr int R4 = E4 + 16, DINV = R4 + 16;
    static constexpr int RED = DINV + (ND * ND + 3) / 4 * 4;   // reduction buffers [2][C NW]
    static constexpr int SC = RED + 2 * ((C * NW + 3) / 4 * 4);   // stopping thresholds
    static constexpr int FLOATS = SC + 4;
    // set-up staging of kappa (cells of one level, lower then upper halves): the next level in E [8][S]; the
    // level below it, whole, in PV; lower ones in D
    static constexpr int KG = PV;
    __host__ __device__ static constexpr int kst(int M) {
        return M == TOP ? (L2 ? D : PV) : M == 16 ? D + (L2 ? 2 * TOP * TOP : 0) : kst(16) + (M == 8 ? 512 : 640);
    }
    // float4s of refinement state of one CTA (device memory): r hi, r lo, x hi, x lo and, with DG, d
    static constexpr int REF4 = (DG ? 20 : 16) * T;
    static_assert(FLOATS * 4 <= 226 * 1024, "shared memory of one block");
    static_assert(N != 64 || FLOATS * 4 <= 113 * 1024, "two blocks of 1/64 on an SM");
};

// ---- thread-block clusters: distributed shared memory --------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
// the address of the same location in CTA `rank` of the cluster (volatile: formed where it is used)
__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_peer(float* p, int rank, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_addr(p, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void st_peer(int* p, int rank, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(peer_addr(p, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_peer(float4* p, int rank, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(peer_addr(p, rank)), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ float2 ld_peer2(const float2* p, int rank) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
                 : "=f"(v.x), "=f"(v.y)
                 : "r"(peer_addr(p, rank))
                 : "memory");
    return v;
}
// barrier of everything that solves one particle: the block, or the cluster (release / acquire, which also
// orders distributed shared memory). All CTAs of a cluster hold bit-identical scalars, so they take the
// same branches and the same number of barriers.
template <int C>
__device__ __forceinline__ void sync_all() {
    if constexpr (C == 1) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// sum over all threads that solve the particle (the same value in every one): warp sums, then, in one CTA,
// in warp order; over a cluster every warp sums all the partials with the same butterfly
template <class G>
__device__ __forceinline__ float total(float v, float* sm, int parity, int rank) {
    constexpr int NP = (G::C * G::NW + 3) / 4 * 4;
    float* buf = sm + G::RED + parity * NP;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if constexpr (G::C == 1) {
        if (lane == 0) buf[threadIdx.x >> 5] = v;
        __syncthreads();
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < G::NW; ++i) s += buf[i];
        return s;
    } else {
        if (lane < G::C) st_peer(buf + rank * G::NW + (threadIdx.x >> 5), lane, v);
        sync_all<G::C>();
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < G::C * G::NW; i += 32)
            if (i + lane < G::C * G::NW) s += buf[i + lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        return s;
    }
}

__device__ __forceinline__ float off4(const float4 w, float e, float wv, float n, float s) {
    return w.x * e + w.y * wv + w.z * n + w.w * s;
}

// inverse (row-major, symmetric) of the operator of level 1/4 (9 unknowns) by
// Gauss-Jordan elimination without pivoting (A is positive definite), by one warp: lane u < ND keeps row u
// in registers, the pivot row comes by shuffles. It is a serial chain that the block waits for: one
// matrix entry per lane in shared memory with a branch per case took 12 K cycles, 9 % of a 1/64 solve.
template <class G>
__device__ __forceinline__ void invert4(const float* k4, float* dinv) {
    constexpr int ND = G::ND;
    const int lane = threadIdx.x & 31, u = lane < ND ? lane : ND - 1;
    // kappa of the 4 x 4 cells, lower halves then upper ones
    auto cell = [&](int t, int I, int J) { return k4[16 * t + J * 4 + I]; };
    auto aE = [&](int I, int J) { return 0.5f * (cell(0, I, J) + cell(1, I, J - 1)); };
    auto aN = [&](int I, int J) { return 0.5f * (cell(0, I - 1, J) + cell(1, I, J)); };
    const int I = u % 3 + 1, J = u / 3 + 1;
    const float wE = aE(I, J), wW = aE(I - 1, J), wN = aN(I, J), wS = aN(I, J - 1);
    float a[ND];
#pragma unroll
    for (int v = 0; v < ND; ++v)
        a[v] = v == u ? wE + wW + wN + wS
                      : v == u + 1 && I < 3 ? -wE : v == u - 1 && I > 1 ? -wW : v == u + 3 ? -wN : v == u - 3 ? -wS : 0.f;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        float row[ND];
#pragma unroll
        for (int v = 0; v < ND; ++v) row[v] = __shfl_sync(0xffffffffu, a[v], k);
        const float ip = recip(row[k]);
        const float f = u == k ? -ip : a[k] * ip;   // row k itself becomes row k / pivot
#pragma unroll
        for (int v = 0; v < ND; ++v) a[v] = v == k ? -f : fmaf(-f, row[v], u == k ? 0.f : a[v]);
    }
    if (lane < ND)
#pragma unroll
        for (int v = 0; v < ND; ++v) dinv[ND * u + v] = a[v];
}

// ---- levels that a CTA solves as a whole ---------------------------------------------------------
// Level M as a grid of M columns and M rows (column 0 and row 0: Dirichlet, always 0), node f = M J + I. A thread takes
// a red and a black node side by side, so that every lane has work in both colours. Neighbours wrap as above.
template <int M>
__device__ __forceinline__ int wrap(int f) {
    return f & (M * M - 1);
}
template <class G, int M>
__device__ __forceinline__ float level_off(const float* sm, int f) {
    const float* e = sm + G::le(M);
    return off4(reinterpret_cast<const float4*>(sm + G::lw(M))[f], e[wrap<M>(f + 1)], e[wrap<M>(f - 1)],
                e[wrap<M>(f + M)], e[wrap<M>(f - M)]);
}
// right-hand side of node (I, J) of level M from the red residuals r of level 2 M: P^T has weight 1 at the
// coincident node and 1/2 at the two red diagonal neighbours (the others are black: zero residual)
template <int M>
__device__ __forceinline__ float level_rhs(const float* r, int I, int J) {
    const int f = 2 * J * 2 * M + 2 * I;
    return r[f] + 0.5f * (r[f + 2 * M + 1] + r[wrap<2 * M>(f - 2 * M - 1)]);
}

// barrier of a level: it runs on the whole block, or (1/8) inside warp 0
template <bool WARP>
__device__ __forceinline__ void sync_level() {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
}

// V(1,1) cycle on level M from the right-hand side in lr(M) (M = TOP of a level that is not distributed
// below it) or the residuals of the level above; the values in le(M) still need a barrier
template <class G, int M>
__device__ __forceinline__ void level_cycle(float* sm) {
    constexpr bool WARP = M == 8;
    float *e = sm + G::le(M), *r = sm + G::lr(M);
    const float* id = sm + G::lid(M);
    float vr = 0.f, vb = 0.f;
    int J, cr, cb;   // row, red and black node of this thread
    bool on;
    // formed again after the levels below, from an opaque thread index: hoisted out of the iteration or kept
    // through it they would cost registers that do not exist (spills)
    auto nodes_of_thread = [&] {
        int t = threadIdx.x;
        asm volatile("" : "+r"(t));
        J = t / (M / 2);
        cr = M * J + 2 * (t % (M / 2)) + (J & 1);
        cb = cr ^ 1;
        on = WARP ? true : t < G::nodes(M) / 2;
    };
    nodes_of_thread();
    if (on) {
        if constexpr (M == G::TOP && !G::L2) {
            vr = r[cr];
            vb = r[cb];
        } else {
            const float* above = sm + (M == G::TOP ? G::RR : G::lr(2 * M));
            vr = level_rhs<M>(above, cr % M, J);
            vb = level_rhs<M>(above, cb % M, J);
        }
        e[cr] = vr * id[cr];   // red pre-sweep from zero
    }
    sync_level<WARP>();
    if (on) e[cb] = (vb + level_off<G, M>(sm, cb)) * id[cb];
    sync_level<WARP>();
    if (on) r[cr] = level_off<G, M>(sm, cr);   // red residuals
    sync_level<WARP>();
    const float* ec = sm + (M == 8 ? G::E4 : G::le(M / 2));
    if constexpr (M == 8) {   // 1/4 solved exactly, in warp 0 (the inverse is symmetric: column reads)
        float *r4 = sm + G::R4, *e4 = sm + G::E4;
        const float* di = sm + G::DINV;
        constexpr int ND = G::ND;
        const int t = threadIdx.x;
        if (t < ND) r4[t] = level_rhs<4>(r, t % 3 + 1, t / 3 + 1);
        __syncwarp();
        if (t < ND) {
            float acc = 0.f;
#pragma unroll
            for (int v = 0; v < ND; ++v) acc = fmaf(di[ND * v + t], r4[v], acc);
            e4[(t / 3 + 1) * 4 + t % 3 + 1] = acc;
        }
        sync_level<WARP>();
    } else {
        if constexpr (M / 2 == 8) {
            if (threadIdx.x < 32) level_cycle<G, M / 2>(sm);
        } else {
            level_cycle<G, M / 2>(sm);
        }
        __syncthreads();
    }
    nodes_of_thread();
    if (on) {   // black post-sweep with the prolongation of the correction ec
        constexpr int MC = M / 2;
        const int c0 = (J >> 1) * MC + ((cb % M) >> 1);
        const bool jeven = (J & 1) == 0;
        const float x0 = ec[c0], x1 = ec[wrap<MC>(c0 + MC + 1)];
        const float xu = ec[wrap<MC>(jeven ? c0 + 1 : c0 + MC)], xv = ec[wrap<MC>(jeven ? c0 - MC : c0 - 1)];
        const float dg = 0.5f * (x0 + x1), hf = 0.5f * (xv + xu);
        const float4 w = reinterpret_cast<const float4*>(sm + G::lw(M))[cb];
        const float s = w.x * (e[wrap<M>(cb + 1)] + (jeven ? xu : dg)) + w.y * (e[wrap<M>(cb - 1)] + (jeven ? x0 : hf)) +
                        w.z * (e[wrap<M>(cb + M)] + (jeven ? dg : xu)) + w.w * (e[wrap<M>(cb - M)] + (jeven ? hf : x0));
        e[cb] = (vb + s) * id[cb];
    }
    sync_level<WARP>();
    if (on) e[cr] = (vr + level_off<G, M>(sm, cr)) * id[cr];
}

// weights and inverse diagonals of level M from its cells' kappa (k: lower halves [M][M], then upper ones),
// kappa of the level below; threads tid, tid + nt, ..
template <class G, int M>
__device__ __forceinline__ void level_setup(float* sm, const float* k, float* kc, int tid, int nt) {
    float4* w = reinterpret_cast<float4*>(sm + G::lw(M));
    const float *lo = k, *up = k + M * M;
    for (int f = tid; f < G::nodes(M); f += nt) {
        // wrapped cells left of column 0 and below row 0 belong to Dirichlet nodes only
        const int l = wrap<M>(f - 1), b = wrap<M>(f - M), d = wrap<M>(f - M - 1);
        const float4 v = make_float4(0.5f * (lo[f] + up[b]), 0.5f * (lo[l] + up[d]), 0.5f * (lo[l] + up[f]),
                                     0.5f * (lo[d] + up[b]));
        w[f] = v;
        sm[G::lid(M) + f] = (f % M == 0 || f < M) ? 0.f : recip_coarse(v.x + v.y + v.z + v.w);
        // the wrapped neighbour of the last column is a Dirichlet node of the reader's own colour, read
        // before its first (zero) value is stored
        sm[G::le(M) + f] = 0.f;
        sm[G::lr(M) + f] = 0.f;   // black entries are read by Dirichlet nodes
    }
    constexpr int MC = M / 2;
    for (int c = tid; c < MC * MC; c += nt) {
        const int f = (c / MC) * 2 * M + (c % MC) * 2;
        kc[c] = 0.25f * (lo[f] + lo[f + 1] + up[f + 1] + lo[f + M + 1]);
        kc[MC * MC + c] = 0.25f * (up[f] + up[f + M] + lo[f + M] + up[f + M + 1]);
    }
}
template <class G, int M>
__device__ __forceinline__ void levels_setup(float* sm) {
    if constexpr (M > 8) {
        level_setup<G, M>(sm, sm + G::kst(M), sm + G::kst(M / 2), threadIdx.x, G::T);
        __syncthreads();
        levels_setup<G, M / 2>(sm);
    } else if (threadIdx.x < 32) {   // warp 0 (the others reach the first reduction)
        level_setup<G, 8>(sm, sm + G::kst(8), sm + G::kst(4), threadIdx.x, 32);
        if (threadIdx.x < 16) sm[G::E4 + threadIdx.x] = 0.f;
        __syncwarp();
        invert4<G>(sm + G::kst(4), sm + G::DINV);
    }
}

// the solve of particle `item` of a.n by the calling block or cluster (every thread calls it). sm: this
// CTA's Geo::FLOATS floats, part: [32] doubles, ref: Geo::REF4 float4 of device memory (this CTA's
// refinement state). RHS: the load vector may come from a table (a.rhs). take(): called by one thread of
// rank 0 while the observations are formed (the next ticket).
template <class G, bool RHS, typename Take>
__device__ __forceinline__ void solve_tile(const FemArgs& a, const int item, float* sm, double* part, float4* ref,
                                           const int rank, Take&& take) {
    constexpr int N = G::N, T = G::T, S = G::S, TX = G::TX, C = G::C;
    constexpr bool H = G::H;
    const int tid = threadIdx.x, lane = tid & 31;
    const int tx = tid % TX, ty = rank * G::R + tid / TX;   // patch of the whole mesh
    // exchange-array index of this patch; its neighbours are at q - 1, q + 1, q - TX, q + TX
    const int q = tid + TX, pL = q - 1, pR = q + 1, pB = q - TX, pA = q + TX, pD = pB - 1, pU = pA + 1;
    float* E = sm + G::E;
    float4* D4 = G::DG ? ref + 16 * T : reinterpret_cast<float4*>(sm + G::D);
    float4* PV4 = reinterpret_cast<float4*>(sm + G::PV);
    float4* ID4 = reinterpret_cast<float4*>(sm + G::ID);
    float4* W1 = reinterpret_cast<float4*>(sm + G::W1);
    float* E1 = sm + G::E1;
    float4* W2 = reinterpret_cast<float4*>(sm + G::W2);
    float *ID2 = sm + G::ID2, *E2 = sm + G::E2;
    // a value of this patch into exchange array x; rows of patches at the CTA's border also go to the
    // neighbour CTA (up: its lower halo row, down: its upper one)
    const bool top = H && tid >= T - TX && rank < C - 1, bottom = H && tid < TX && rank > 0;
    auto put = [&](float* x, float v, bool up, bool down) {
        x[q] = v;
        if constexpr (H) {
            if (up && top) st_peer(x + tx, rank + 1, v);
            if (down && bottom) st_peer(x + T + TX + tx, rank - 1, v);
        }
    };
    // a node of the patch on the Dirichlet column or row
    auto fixed = [&](int i, int b) { return (i == 0 && tx == 0) || (b == 0 && ty == 0); };

    // inverse diagonal of a node of the next level (or the one below it) from its weights
    auto inv1 = [&](const float4& x, int A, int B) {
        return fixed(A, B) ? 0.f : recip_coarse(x.x + x.y + x.z + x.w);
    };

    // ---- edge weights: wE[b][k] joins nodes (k - 1, b) and (k, b) of the patch, wN[k][a] (a, k - 1) and (a, k)
    float wE[4][5], wN[5][4];
    {
        const float* kp = a.kappa + (size_t)item * (2 * N * N) + 2 * (4 * ty * N + 4 * tx);
        float lo[5][5], up[5][5];   // kappa of cells (-1 .. 3)^2, index [row + 1][column + 1]
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const bool row = b > 0 || ty > 0;
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
            float2 l = make_float2(0.f, 0.f);
            if (row) {
                u = *reinterpret_cast<const float4*>(kp + 2 * (b - 1) * N);
                v = *reinterpret_cast<const float4*>(kp + 2 * (b - 1) * N + 4);
                if (tx > 0) l = *reinterpret_cast<const float2*>(kp + 2 * (b - 1) * N - 2);
            }
            lo[b][0] = l.x; up[b][0] = l.y;
            lo[b][1] = u.x; up[b][1] = u.y;
            lo[b][2] = u.z; up[b][2] = u.w;
            lo[b][3] = v.x; up[b][3] = v.y;
            lo[b][4] = v.z; up[b][4] = v.w;
        }
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int k = 0; k < 5; ++k) wE[b][k] = 0.5f * (lo[b + 1][k] + up[b][k]);
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) wN[k][i] = 0.5f * (lo[k][i] + up[k][i + 1]);
        // kappa of the next level under the patch (mean of the four triangles inside each coarse one)
        float cl[2][2], cu[2][2];   // [B][A]
#pragma unroll
        for (int B = 0; B < 2; ++B)
#pragma unroll
            for (int A = 0; A < 2; ++A) {
                const int i = 2 * A + 1, j = 2 * B + 1;
                cl[B][A] = 0.25f * (lo[j][i] + lo[j][i + 1] + up[j][i + 1] + lo[j + 1][i + 1]);
                cu[B][A] = 0.25f * (up[j][i] + up[j + 1][i] + lo[j + 1][i] + up[j + 1][i + 1]);
                put(E + (2 * (A + 2 * B)) * S, cl[B][A], B == 1, false);
                put(E + (2 * (A + 2 * B) + 1) * S, cu[B][A], B == 1, false);
            }
        // and of the level below that, whole in every CTA
        constexpr int M = N / 4;
        float* k = sm + G::KG + ty * M + tx;
        const float l2 = 0.25f * (cl[0][0] + cl[0][1] + cu[0][1] + cl[1][1]);
        const float u2 = 0.25f * (cu[0][0] + cu[1][0] + cl[1][0] + cu[1][1]);
        if constexpr (!H) {
            k[0] = l2;
            k[M * M] = u2;
        } else {
#pragma unroll 1
            for (int c = 0; c < C; ++c) {
                st_peer(k, c, l2);
                st_peer(k + M * M, c, u2);
            }
        }
    }
    // fine inverse diagonals: 1 / the sum of the edge weights, 0 on Dirichlet nodes
    auto diag = [&](int i, int b) { return wE[b][i + 1] + wE[b][i] + wN[b + 1][i] + wN[b][i]; };
    auto store_diag = [&] {
#pragma unroll
        for (int c = 0; c < 2; ++c)   // colour c, rows 0 1 and rows 2 3
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int b = 2 * h + k / 2, i = 2 * (k % 2) + ((b & 1) ^ c);
                    const float d = diag(i, b);
                    v[k] = fixed(i, b) ? 0.f : d == 0.f ? 1.f : recip(d);
                }
                ID4[(2 * c + h) * T + tid] = make_float4(v[0], v[1], v[2], v[3]);
            }
    };
    if constexpr (G::STORED && !G::DG) store_diag();
    sync_all<C>();
    {   // next level: the weights of the 2 x 2 nodes
        float lo[3][3], up[3][3];   // cells (-1 .. 1)^2, index [row + 1][column + 1]
        auto K = [&](int pos, int t, int p) { return E[(2 * pos + t) * S + p]; };
        lo[1][0] = K(1, 0, pL); up[1][0] = K(1, 1, pL); lo[2][0] = K(3, 0, pL);
        lo[0][0] = K(3, 0, pD); up[0][0] = K(3, 1, pD);
        lo[0][1] = K(2, 0, pB); up[0][1] = K(2, 1, pB); up[0][2] = K(3, 1, pB);
#pragma unroll
        for (int pos = 0; pos < 4; ++pos) {
            lo[1 + pos / 2][1 + pos % 2] = K(pos, 0, q);
            up[1 + pos / 2][1 + pos % 2] = K(pos, 1, q);
        }
        // nobody's halo: only Dirichlet nodes read it
        if (ty == 0) lo[0][0] = up[0][0] = lo[0][1] = up[0][1] = up[0][2] = 0.f;
        if (tx == 0) lo[0][0] = up[0][0] = lo[1][0] = up[1][0] = lo[2][0] = 0.f;
        auto w = [&](int A, int B) {
            return make_float4(0.5f * (lo[B + 1][A + 1] + up[B][A + 1]), 0.5f * (lo[B + 1][A] + up[B][A]),
                               0.5f * (lo[B + 1][A] + up[B + 1][A + 1]), 0.5f * (lo[B][A] + up[B][A + 1]));
        };
        const float4 w00 = w(0, 0), w11 = w(1, 1), w10 = w(1, 0), w01 = w(0, 1);
        W1[tid] = w00;
        W1[T + tid] = w11;
        W1[2 * T + tid] = w10;
        W1[3 * T + tid] = w01;
        if (top) st_peer(reinterpret_cast<float4*>(sm + G::WH) + tx, rank + 1, w11);
        if constexpr (G::L2) {   // 1/64: the weights of node (tx, ty) from the whole level's cells
            constexpr int M = N / 4;
            const float *lo2 = sm + G::KG, *up2 = lo2 + M * M;
            const int f = ty * M + tx, l = wrap<M>(f - 1), b = wrap<M>(f - M), d = wrap<M>(f - M - 1);
            const float4 v = make_float4(0.5f * (lo2[f] + up2[b]), 0.5f * (lo2[l] + up2[d]), 0.5f * (lo2[l] + up2[f]),
                                         0.5f * (lo2[d] + up2[b]));
            W2[tid] = v;
            ID2[tid] = inv1(v, 0, 0);
            constexpr int MC = M / 2;
            for (int c = tid; c < MC * MC; c += T) {
                const int g = (c / MC) * 2 * M + (c % MC) * 2;
                sm[G::kst(MC) + c] = 0.25f * (lo2[g] + lo2[g + 1] + up2[g + 1] + lo2[g + M + 1]);
                sm[G::kst(MC) + MC * MC + c] = 0.25f * (up2[g] + up2[g + M] + lo2[g + M] + up2[g + M + 1]);
            }
        }
    }
    __syncthreads();   // the staging in E is read
    // halo rows: zero where no neighbour writes them (beyond the mesh, the positions that are not sent,
    // the wrapped column's Dirichlet nodes)
    for (int x = tid; x < 2 * TX + 4; x += T) {
        const int p = x < TX ? x : T + x;
#pragma unroll 1
        for (int pos = 0; pos < 16; ++pos) E[pos * S + p] = 0.f;
#pragma unroll 1
        for (int pos = 0; pos < 4; ++pos) E1[pos * S + p] = 0.f;
        if (rank == 0 && x < TX) reinterpret_cast<float4*>(sm + G::WH)[x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if constexpr (G::L2) {
        for (int x = tid; x < S; x += T) E2[x] = 0.f;
        for (int x = tid; x < G::nodes(2 * G::TOP); x += T) sm[G::RR + x] = 0.f;
    }
    if constexpr (H) sync_all<C>();   // the neighbours write into this CTA's arrays only from here on
    levels_setup<G, G::TOP>(sm);
    if constexpr (G::DG) {   // over the staging that the levels were set up from
        __syncthreads();
        store_diag();
    }

    // ---- rim exchange: colour c's values of the neighbouring patches next to the patch's other colour
    float hL[4], hR[4], hB[4], hA[4];
    auto load_halo = [&](int c) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (((3 + k) & 1) == c) {
                hL[k] = E[(4 * k + 3) * S + pL];
                hB[k] = E[(12 + k) * S + pB];
            } else {
                hR[k] = E[(4 * k) * S + pR];
                hA[k] = E[k * S + pA];
            }
        }
    };
    float r[4][4], e[4][4];
    auto store_rim = [&](int c, const float (&v)[4][4]) {   // c = 2: both colours
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if ((c == 2 || ((i + b) & 1) == c) && (i == 0 || i == 3 || b == 0 || b == 3))
                    put(E + (4 * b + i) * S, v[b][i], b == 3, b == 0);
    };
    // off-diagonal sum at patch node (i, b) of v, rim neighbours from the halo
    auto off = [&](const float (&v)[4][4], int i, int b) {
        return wE[b][i + 1] * (i < 3 ? v[b][i < 3 ? i + 1 : 3] : hR[b]) + wE[b][i] * (i > 0 ? v[b][i > 0 ? i - 1 : 0] : hL[b]) +
               wN[b + 1][i] * (b < 3 ? v[b < 3 ? b + 1 : 3][i] : hA[i]) + wN[b][i] * (b > 0 ? v[b > 0 ? b - 1 : 0][i] : hB[i]);
    };
    auto inv_diag = [&](int c, float (&v)[8]) {   // this thread's inverse diagonals of colour c, in node order
        if constexpr (G::STORED) {
            const float4 x = ID4[2 * c * T + tid], y = ID4[(2 * c + 1) * T + tid];
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int b = k / 2, i = 2 * (k % 2) + ((b & 1) ^ c);
                float w = wE[b][i];
                asm volatile("" : "+f"(w));   // the sum is formed here, not kept in a register through the iteration
                v[k] = fixed(i, b) ? 0.f : recip_coarse(wE[b][i + 1] + w + wN[b + 1][i] + wN[b][i]);
            }
        }
    };

    const float h2 = 1.f / (float(N) * float(N));   // f = 1: exact in FP32
    auto load_b = [&](int i, int b, float& hi, float& lo) {   // the load vector at a node of the patch
        lo = 0.f;
        hi = h2;
        if (RHS && a.rhs) {
            const float2 v = static_cast<const float2*>(a.rhs)[(4 * ty + b) * fem_row_stride(N) + 4 * tx + i];
            hi = v.x;
            lo = v.y;
        }
        if (fixed(i, b)) hi = lo = 0.f;
    };
    int parity = 0, total_it = 0;
    const float bnorm2 = (RHS && a.rhs) ? float(a.bnorm2) : float((N - 1) * (N - 1)) * h2 * h2;
    // thresholds of the outer residual, of the last inner pass and of an inner pass's relative reduction
    // (read after the first barrier below; in shared memory so that they hold no registers meanwhile)
    volatile float* stop = sm + G::SC;
    if (tid == 0) {
        stop[0] = float(a.rtol * a.rtol) * bnorm2;
        stop[1] = float(0.25 * a.rtol * a.rtol) * bnorm2;
        stop[2] = float(a.rtol_in * a.rtol_in);
    }
    bool converged = false;

#pragma unroll 1
    for (int pass = 0; pass < a.max_outer && !converged; ++pass) {
        float rr = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (pass == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float lo;
                    load_b(i, b, r[b][i], lo);
                }
            } else {
                const float4 v = ref[b * T + tid];
                r[b][0] = v.x; r[b][1] = v.y; r[b][2] = v.z; r[b][3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) rr += r[b][i] * r[b][i];
        }
        {   // red pre-sweep of the first cycle
            float id[8];
            inv_diag(0, id);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int b = q / 2, i = 2 * (q % 2) + (b & 1);
                e[b][i] = r[b][i] * id[q];
            }
            store_rim(0, e);
        }
        const float rr0 = total<G>(rr, sm, parity, rank);
        parity ^= 1;
        if (!(rr0 > 0.f)) break;
        const float stop2 = fmaxf(stop[2] * rr0, stop[1]);
        float rz = 0.f;
#pragma unroll 1
        for (int it = 0; it < a.max_inner; ++it) {
            // black pre-sweep
            load_halo(0);
            {
                float id[8];
                inv_diag(1, id);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int b = q / 2, i = 2 * (q % 2) + ((b & 1) ^ 1);
                    e[b][i] = (r[b][i] + off(e, i, b)) * id[q];
                }
            }
            store_rim(1, e);
            sync_all<C>();
            // red residuals (off-diagonal sums of the black values); the three that the neighbours'
            // coarse nodes read go into the slots of inner positions
            float v00, v10, v01, v11;   // coarse right-hand side under the patch
            {
                load_halo(1);
                const float s00 = off(e, 0, 0), s20 = off(e, 2, 0), s02 = off(e, 0, 2), s22 = off(e, 2, 2);
                const float s11 = off(e, 1, 1), s31 = off(e, 3, 1), s13 = off(e, 1, 3), s33 = off(e, 3, 3);
                put(E + 5 * S, s33, true, false);
                put(E + 6 * S, s13, true, false);
                E[9 * S + q] = s31;
                sync_all<C>();
                v00 = s00 + 0.5f * (s11 + E[5 * S + pD]);
                v10 = s20 + 0.5f * (s31 + E[6 * S + pB]);
                v01 = s02 + 0.5f * (s13 + E[9 * S + pL]);
                v11 = s22 + 0.5f * (s33 + s11);
            }
            float e00, e10, e01, e11;   // the coarse nodes of the patch
            {
                e00 = v00 * inv1(W1[tid], 0, 0);
                e11 = v11 * inv1(W1[T + tid], 1, 1);
                put(E1, e00, false, true);
                put(E1 + 3 * S, e11, true, false);
            }
            sync_all<C>();
            {   // coarse black pre-sweep
                const float4 w10 = W1[2 * T + tid], w01 = W1[3 * T + tid];
                e10 = (v10 + off4(w10, E1[pR], e00, e11, E1[3 * S + pB])) * inv1(w10, 1, 0);
                e01 = (v01 + off4(w01, e11, E1[3 * S + pL], E1[pA], e00)) * inv1(w01, 0, 1);
                put(E1 + S, e10, true, true);
                put(E1 + 2 * S, e01, true, false);
            }
            sync_all<C>();
            if constexpr (G::VS) reinterpret_cast<float4*>(sm + G::V1)[tid] = make_float4(v00, v10, v01, v11);
            // right-hand side of the node (tx, ty) two levels down
            {
                const float l10 = E1[S + pL], b01 = E1[2 * S + pB];
                // the weights of the patch below left (tx = 0: any, the node is a Dirichlet node)
                const float4 wD = tid < TX ? reinterpret_cast<const float4*>(sm + G::WH)[tx > 0 ? tx - 1 : 0]
                                           : W1[T + tid - TX - (tx > 0 ? 1 : 0)];
                const float s00 = off4(W1[tid], e10, l10, e01, b01);
                const float s11 = off4(W1[T + tid], E1[2 * S + pR], e01, E1[S + pA], e10);
                const float sdd = off4(wD, b01, E1[2 * S + pD], l10, E1[S + pD]);
                const float v2 = s00 + 0.5f * (s11 + sdd);
                if constexpr (G::L2) {   // distributed level of one node per thread
                    const bool red2 = ((tx + ty) & 1) == 0;
                    if (red2) put(E2, v2 * ID2[tid], true, true);
                    sync_all<C>();
                    if (!red2) put(E2, (v2 + off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB])) * ID2[tid], true, true);
                    sync_all<C>();
                    // red residuals into every CTA's copy of the whole level
                    if (red2) {
                        const float s2 = off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB]);
#pragma unroll 1
                        for (int c = 0; c < C; ++c) st_peer(sm + G::RR + ty * (N / 4) + tx, c, s2);
                    }
                    sync_all<C>();
                    level_cycle<G, G::TOP>(sm);
                    __syncthreads();
                    if (!red2) {   // black post-sweep with the correction of the level below
                        constexpr int MC = G::TOP;
                        const float* ec = sm + G::le(MC);
                        const int c0 = (ty >> 1) * MC + (tx >> 1);
                        const bool jeven = (ty & 1) == 0;
                        const float x0 = ec[wrap<MC>(c0)], x1 = ec[wrap<MC>(c0 + MC + 1)];
                        const float xu = ec[wrap<MC>(jeven ? c0 + 1 : c0 + MC)];
                        const float xv = ec[wrap<MC>(jeven ? c0 - MC : c0 - 1)];
                        const float dg = 0.5f * (x0 + x1), hf = 0.5f * (xv + xu);
                        const float4 w = W2[tid];
                        const float s = w.x * (E2[pR] + (jeven ? xu : dg)) + w.y * (E2[pL] + (jeven ? x0 : hf)) +
                                        w.z * (E2[pA] + (jeven ? dg : xu)) + w.w * (E2[pB] + (jeven ? hf : x0));
                        put(E2, (v2 + s) * ID2[tid], true, true);
                    }
                    sync_all<C>();
                    if (red2) put(E2, (v2 + off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB])) * ID2[tid], true, true);
                    sync_all<C>();
                } else {   // the next level down is whole in every CTA
                    float* x = sm + G::lr(G::TOP) + ty * G::TOP + tx;
                    if constexpr (!H) {
                        *x = v2;
                    } else {
#pragma unroll
                        for (int c = 0; c < C; ++c) st_peer(x, c, v2);
                    }
                    sync_all<C>();
                    if constexpr (G::TOP == 8) {
                        if (tid < 32) level_cycle<G, G::TOP>(sm);
                    } else {
                        level_cycle<G, G::TOP>(sm);
                    }
                    __syncthreads();
                }
            }
            // values of the level of one node per patch: this patch's and the neighbours'
            auto c2 = [&](int p, int dx, int dy) {
                if constexpr (G::L2) return E2[p];
                else return (sm + G::le(G::TOP))[wrap<G::TOP>((ty + dy) * G::TOP + tx + dx)];
            };
            if constexpr (G::VS) {
                const float4 v = reinterpret_cast<const float4*>(sm + G::V1)[tid];
                v00 = v.x; v10 = v.y; v01 = v.z; v11 = v.w;
                e00 = E1[q];
                e11 = E1[3 * S + q];
            }
            {   // 2 x 2 level, black post-sweep: red neighbours with the correction of the level below
                const float c0 = c2(q, 0, 0), cR = c2(pR, 1, 0), cA = c2(pA, 0, 1), cU = c2(pU, 1, 1),
                            cL = c2(pL, -1, 0), cB = c2(pB, 0, -1);
                const float4 w10 = W1[2 * T + tid], w01 = W1[3 * T + tid];
                const float f00 = e00 + c0, f11 = e11 + 0.5f * (c0 + cU);
                const float fR = E1[pR] + cR, fA = E1[pA] + cA;
                const float fB = E1[3 * S + pB] + 0.5f * (cB + cR), fL = E1[3 * S + pL] + 0.5f * (cL + cA);
                e10 = (v10 + off4(w10, fR, f00, f11, fB)) * inv1(w10, 1, 0);
                e01 = (v01 + off4(w01, f11, fL, fA, f00)) * inv1(w01, 0, 1);
                put(E1 + S, e10, true, true);
                put(E1 + 2 * S, e01, true, false);
            }
            sync_all<C>();
            {   // red post-sweep
                const float4 w00 = W1[tid], w11 = W1[T + tid];
                e00 = (v00 + off4(w00, e10, E1[S + pL], e01, E1[2 * S + pB])) * inv1(w00, 0, 0);
                e11 = (v11 + off4(w11, E1[2 * S + pR], e01, E1[S + pA], e10)) * inv1(w11, 1, 1);
                // the fine black sweep reads all four positions of the patches around
                put(E1, e00, true, true);
                put(E1 + 3 * S, e11, true, true);
            }
            sync_all<C>();
            {   // fine black post-sweep: red values plus the prolonged correction
                load_halo(0);
                const float c20 = E1[pR], c21 = E1[2 * S + pR], c02 = E1[pA], c12 = E1[S + pA], c22 = E1[pU];
                const float cm0 = E1[S + pL], cm1 = E1[3 * S + pL], c0m = E1[2 * S + pB], c1m = E1[3 * S + pB];
                e[0][0] += e00;
                e[0][2] += e10;
                e[2][0] += e01;
                e[2][2] += e11;
                e[1][1] += 0.5f * (e00 + e11);
                e[1][3] += 0.5f * (e10 + c21);
                e[3][1] += 0.5f * (e01 + c12);
                e[3][3] += 0.5f * (e11 + c22);
                hL[1] += 0.5f * (cm0 + e01);
                hL[3] += 0.5f * (cm1 + c02);
                hR[0] += c20;
                hR[2] += c21;
                hB[1] += 0.5f * (c0m + e10);
                hB[3] += 0.5f * (c1m + c20);
                hA[0] += c02;
                hA[2] += c12;
                float id[8];
                inv_diag(1, id);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int b = q / 2, i = 2 * (q % 2) + ((b & 1) ^ 1);
                    e[b][i] = (r[b][i] + off(e, i, b)) * id[q];
                }
            }
            store_rim(1, e);
            sync_all<C>();
            float rz_new = 0.f;
            {   // fine red post-sweep: z = e
                load_halo(1);
                float id[8];
                inv_diag(0, id);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int b = q / 2, i = 2 * (q % 2) + (b & 1);
                    e[b][i] = (r[b][i] + off(e, i, b)) * id[q];
                }
            }
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int i = 0; i < 4; ++i) rz_new += r[b][i] * e[b][i];
            rz_new = total<G>(rz_new, sm, parity, rank);
            parity ^= 1;
            const float beta = it == 0 ? 0.f : rz_new / rz;
            rz = rz_new;
            float p[4][4];   // p = z + beta p
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                float4 v = make_float4(e[b][0], e[b][1], e[b][2], e[b][3]);
                if (it > 0) {
                    const float4 o = PV4[b * T + tid];
                    v.x += beta * o.x;
                    v.y += beta * o.y;
                    v.z += beta * o.z;
                    v.w += beta * o.w;
                }
                PV4[b * T + tid] = v;
                p[b][0] = v.x; p[b][1] = v.y; p[b][2] = v.z; p[b][3] = v.w;
            }
            store_rim(2, p);
            sync_all<C>();
            // q = A p in edge form (into e), alpha = rz / p.q
            load_halo(0);
            load_halo(1);
            float pq = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float c = p[b][i];
                    const float vE = i < 3 ? p[b][i < 3 ? i + 1 : 3] : hR[b], vW = i > 0 ? p[b][i > 0 ? i - 1 : 0] : hL[b];
                    const float vN = b < 3 ? p[b < 3 ? b + 1 : 3][i] : hA[i], vS = b > 0 ? p[b > 0 ? b - 1 : 0][i] : hB[i];
                    float q = wE[b][i + 1] * (c - vE) + wE[b][i] * (c - vW) + wN[b + 1][i] * (c - vN) + wN[b][i] * (c - vS);
                    if (fixed(i, b)) q = 0.f;
                    e[b][i] = q;
                    pq += c * q;
                }
            pq = total<G>(pq, sm, parity, rank);
            parity ^= 1;
            const float alpha = rz / pq;
            rr = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                float4 d = it == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : D4[b * T + tid];
                d.x = fmaf(alpha, p[b][0], d.x);
                d.y = fmaf(alpha, p[b][1], d.y);
                d.z = fmaf(alpha, p[b][2], d.z);
                d.w = fmaf(alpha, p[b][3], d.w);
                D4[b * T + tid] = d;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    r[b][i] = fmaf(-alpha, e[b][i], r[b][i]);
                    rr += r[b][i] * r[b][i];
                }
            }
            {   // red pre-sweep of the next cycle
                float id[8];
                inv_diag(0, id);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int b = q / 2, i = 2 * (q % 2) + (b & 1);
                    e[b][i] = r[b][i] * id[q];
                }
                store_rim(0, e);
            }
            rr = total<G>(rr, sm, parity, rank);
            parity ^= 1;
            ++total_it;
            if (!(rr > stop2)) break;   // also leaves on NaN
        }
        // ---- refinement: x += d, r -= A d in double-float arithmetic (edge form) ----
        float p[4][4];   // d
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float4 d = D4[b * T + tid];
            p[b][0] = d.x; p[b][1] = d.y; p[b][2] = d.z; p[b][3] = d.w;
        }
        store_rim(2, p);
        sync_all<C>();
        load_halo(0);
        load_halo(1);
        float rr_out = 0.f;
        // flux w (d_i - d_j) of an edge as an exact-difference, exact-product pair; an edge inside the patch
        // is computed once and enters its two nodes with opposite signs (negation is exact)
        auto flux = [](float w, float di, float dj, float& ph, float& pl) {
            float sh, sl;
            two_sum(di, -dj, sh, sl);    // d_i - d_j exactly
            ph = __fmul_rn(w, sh);       // kept out of FMA contraction
            pl = fmaf(w, sh, -ph);       // exact product error
            pl = fmaf(w, sl, pl);
        };
        float sth[4], stl[4];   // fluxes through the patch rows' lower edges (node below -> node)
#pragma unroll
        for (int i = 0; i < 4; ++i) flux(wN[0][i], hB[i], p[0][i], sth[i], stl[i]);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            float rh[4], rl[4], xh[4], xl[4];
            if (pass == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    load_b(i, b, rh[i], rl[i]);
                    xh[i] = p[b][i];
                    xl[i] = 0.f;
                }
            } else {
                const float4 v0 = ref[b * T + tid], v1 = ref[(4 + b) * T + tid], v2 = ref[(8 + b) * T + tid],
                             v3 = ref[(12 + b) * T + tid];
                rh[0] = v0.x; rh[1] = v0.y; rh[2] = v0.z; rh[3] = v0.w;
                rl[0] = v1.x; rl[1] = v1.y; rl[2] = v1.z; rl[3] = v1.w;
                xh[0] = v2.x; xh[1] = v2.y; xh[2] = v2.z; xh[3] = v2.w;
                xl[0] = v3.x; xl[1] = v3.y; xl[2] = v3.z; xl[3] = v3.w;
#pragma unroll
                for (int i = 0; i < 4; ++i) df_add(xh[i], xl[i], p[b][i], 0.f);
            }
            float wsh, wsl;   // flux through the left edge of the node (left node -> node)
            flux(wE[b][0], hL[b], p[b][0], wsh, wsl);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float eh, el, nh, nl;
                flux(wE[b][i + 1], p[b][i], i < 3 ? p[b][i < 3 ? i + 1 : 3] : hR[b], eh, el);
                flux(wN[b + 1][i], p[b][i], b < 3 ? p[b < 3 ? b + 1 : 3][i] : hA[i], nh, nl);
                df_residual(rh[i], rl[i], eh, el, -wsh, -wsl, nh, nl, -sth[i], -stl[i]);
                if (fixed(i, b)) rh[i] = rl[i] = 0.f;
                rr_out += rh[i] * rh[i];
                wsh = eh;
                wsl = el;
                sth[i] = nh;
                stl[i] = nl;
            }
            ref[b * T + tid] = make_float4(rh[0], rh[1], rh[2], rh[3]);
            ref[(4 + b) * T + tid] = make_float4(rl[0], rl[1], rl[2], rl[3]);
            ref[(8 + b) * T + tid] = make_float4(xh[0], xh[1], xh[2], xh[3]);
            ref[(12 + b) * T + tid] = make_float4(xl[0], xl[1], xl[2], xl[3]);
        }
        rr_out = total<G>(rr_out, sm, parity, rank);
        parity ^= 1;
        converged = rr_out <= stop[0];
    }


    // ---- observations and misfit (FP64): the solution's double-float pairs go to shared memory
    // (over E and the arrays after it); the block (rank 0 of a cluster, reading the others' shared memory) gathers ----
    float2* xs = reinterpret_cast<float2*>(sm + G::E);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        float4 xh = make_float4(0.f, 0.f, 0.f, 0.f), xl = xh;
        if (total_it > 0) {
            xh = ref[(8 + b) * T + tid];
            xl = ref[(12 + b) * T + tid];
        }
        xs[(4 * b) * T + tid] = make_float2(xh.x, xl.x);
        xs[(4 * b + 1) * T + tid] = make_float2(xh.y, xl.y);
        xs[(4 * b + 2) * T + tid] = make_float2(xh.z, xl.z);
        xs[(4 * b + 3) * T + tid] = make_float2(xh.w, xl.w);
    }
    sync_all<C>();
    if (rank != 0) return;
    auto val = [&](int n) -> double {   // n = j (N + 2) + i
        const int j = n / fem_row_stride(N), i = n - j * fem_row_stride(N);
        if (i < 1 || i >= N || j < 1 || j >= N) return 0.0;
        const int row = j >> 2, c = row / G::R;
        const float2* x = xs + (4 * (j & 3) + (i & 3)) * T + (row - c * G::R) * TX + (i >> 2);
        const float2 v = H ? ld_peer2(x, c) : *x;
        return (double)v.x + (double)v.y;
    };
    if (tid == T - 1) take();   // the ticket's latency overlaps the observations
    double misfit = 0.0;
    for (int o = tid; o < a.n_obs; o += T) {
        const double g = a.obs_w[3 * o] * val(a.obs_idx[3 * o]) + a.obs_w[3 * o + 1] * val(a.obs_idx[3 * o + 1]) +
                         a.obs_w[3 * o + 2] * val(a.obs_idx[3 * o + 2]);
        if (a.G) a.G[(size_t)item * a.n_obs + o] = g;
        const double rdf = a.y[o] - g;
        misfit += rdf * rdf;
    }
    const int nw = min(G::NW, (a.n_obs + 31) / 32);   // warps that hold observations
    if (tid < 32 * nw) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) misfit += __shfl_xor_sync(0xffffffffu, misfit, o);
        if (lane == 0) part[tid >> 5] = misfit;
    }
    __syncthreads();
    if (tid == 0) {
        for (int k = 1; k < nw; ++k) misfit += part[k];
        a.Phi[item] = 0.5 * misfit * a.inv_sigma2;
        if (a.iters) a.iters[item] = converged ? total_it : -(total_it + 1);
        if (a.bad && !converged) atomicAdd(a.bad, 1u);
    }
}

// persistent blocks (clusters: rank 0 hands the ticket to the others) take particles from a ticket
// counter; the barrier at the end of a solve keeps every CTA from overwriting memory another still reads,
// and one at the start of a cluster's CTAs (660 cycles a launch) lets rank 0 hand out the first ticket: a
// CTA's shared memory may be written by others only once it has started, which co-scheduling does not give.
// Every block (cluster) draws tickets until one lies past the particles. The counter is 0 before each launch:
// the split of theta that starts the evaluation zeroes it (a memset of its own would be one more launch).
template <class G, bool RHS>
__global__ void __launch_bounds__(G::T, G::MINB) fem_tile_kernel(FemArgs a, float4* ref_scratch, int* counter) {
    extern __shared__ __align__(16) float sm[];
    __shared__ double part[32];
    __shared__ int item_s[2];
    const int rank = G::H ? cluster_rank() : 0;
    float4* ref = ref_scratch + (size_t)blockIdx.x * G::REF4;
    if constexpr (G::H) sync_all<G::C>();   // every CTA runs before the first store into another's memory
    grid_wait();
    auto take = [&](int k) {
        const int item = atomicAdd(counter, 1);
        item_s[k] = item;
        if constexpr (G::H)
            for (int c = 1; c < G::C; ++c) st_peer(&item_s[k], c, item);
    };
    if (rank == 0 && threadIdx.x == 0) take(0);
    sync_all<G::C>();
    for (int k = 0;; k ^= 1) {
        const int item = item_s[k];
        if (item >= a.n) break;   // the same item in every CTA
        solve_tile<G, RHS>(a, item, sm, part, ref, rank, [&] { take(k ^ 1); });
        sync_all<G::C>();
    }
}

// many problems: the same loop over (problem, particle) items; every CTA copies the item's launch
// arguments to shared memory
template <class G>
__global__ void __launch_bounds__(G::T, G::MINB)
    fem_tile_multi(const FemArgs* groups, const int* offsets, const int* item_group, int total_items, float4* ref_scratch,
                   int* counter) {
    extern __shared__ __align__(16) float sm[];
    __shared__ double part[32];
    __shared__ int item_s[2], p_s;
    __shared__ FemArgs args_s;
    const int rank = G::H ? cluster_rank() : 0;
    float4* ref = ref_scratch + (size_t)blockIdx.x * G::REF4;
    if constexpr (G::H) sync_all<G::C>();   // as above
    auto take = [&](int k) {
        const int item = atomicAdd(counter, 1);
        item_s[k] = item;
        if constexpr (G::H)
            for (int c = 1; c < G::C; ++c) st_peer(&item_s[k], c, item);
    };
    if (rank == 0 && threadIdx.x == 0) take(0);
    sync_all<G::C>();
    for (int k = 0; item_s[k] < total_items; k ^= 1) {
        if (threadIdx.x == 0) {
            const int item = item_s[k], g = item_group[item];
            args_s = groups[g];
            p_s = item - offsets[g];
        }
        __syncthreads();
        solve_tile<G, true>(args_s, p_s, sm, part, ref, rank, [&] { take(k ^ 1); });
        sync_all<G::C>();
    }
}

template <class G>
constexpr size_t tile_smem() {
    return sizeof(float) * (size_t)G::FLOATS;
}

template <class G, typename K>
cudaError_t set_smem(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem<G>());
}

template <class G>
void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int grid, cudaStream_t st) {
    cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(G::T, 1, 1);
    cfg.dynamicSmemBytes = tile_smem<G>();
    cfg.stream = st;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = G::C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = G::H ? 1 : 0;
}

// CTAs of kernel `kern` that are resident at once
template <class G, typename K>
int resident(K kern) {
    int dev = 0, sms = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (set_smem<G>(kern) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if constexpr (!G::H) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, G::T, tile_smem<G>()) != cudaSuccess) n = 0;
        n *= sms;
    } else {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        config<G>(cfg, attr, G::C, nullptr);
        if (cudaOccupancyMaxActiveClusters(&n, (const void*)kern, &cfg) != cudaSuccess) n = 0;
        n *= G::C;
    }
    cudaGetLastError();
    return n;
}

template <class G, bool RHS>
cudaError_t launch_one(const FemArgs& a, float* ref_scratch, int grid, int* counter, cudaStream_t st) {
    cudaError_t e = set_smem<G>(fem_tile_kernel<G, RHS>);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    config<G>(cfg, attr[0], grid, st);
    if (may_overlap(st)) overlap_attr(attr[cfg.numAttrs++]);   // launch.h
    e = cudaLaunchKernelEx(&cfg, fem_tile_kernel<G, RHS>, a, reinterpret_cast<float4*>(ref_scratch), counter);
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <class G>
cudaError_t launch_multi(const FemArgs* groups, const int* offsets, const int* item_group, int total, float* ref_scratch,
                         int grid, int* counter, cudaStream_t st) {
    cudaError_t e = set_smem<G>(fem_tile_multi<G>);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    config<G>(cfg, attr, grid, st);
    e = cudaLaunchKernelEx(&cfg, fem_tile_multi<G>, groups, offsets, item_group, total,
                           reinterpret_cast<float4*>(ref_scratch), counter);
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// the compiled forms: f(Geo) for level N
template <typename F>
auto with_form(int N, F&& f) {
    switch (N) {
        case 32: return f(Geo<32, 1>());
        case 128: return f(Geo<128, 2>());
        case 256: return f(Geo<256, 8>());
        default: return f(Geo<64, 1>());
    }
}

// resident CTAs of level N's form (0: it does not fit), queried once per device
int tile_ctas(int N) {
    static std::atomic<int> cached[64][4];
    int dev = 0;
    cudaGetDevice(&dev);
    const int c = N == 32 ? 0 : N == 64 ? 1 : N == 128 ? 2 : 3;
    const bool slot = dev >= 0 && dev < 64;
    if (slot) {
        const int v = cached[dev][c].load(std::memory_order_relaxed);
        if (v > 0) return v;
    }
    const int n = with_form(N, [](auto g) {
        using G = decltype(g);
        return std::min(std::min(resident<G>(fem_tile_kernel<G, false>), resident<G>(fem_tile_kernel<G, true>)),
                        resident<G>(fem_tile_multi<G>));
    });
    if (slot && n > 0) cached[dev][c].store(n, std::memory_order_relaxed);
    return n;
}

// CTAs of a launch over n particles
int tile_grid(int N, int n) {
    const int C = with_form(N, [](auto g) { return decltype(g)::C; });
    return (int)std::min<long long>((long long)C * n, tile_ctas(N) / C * C);
}

}  // namespace

bool fem_tile_form(int N, int precision, bool flow_cell) {
    return N >= 32 && N <= 256 && precision == SMC_MIXED && !flow_cell && tile_ctas(N) > 0;
}

size_t fem_tile_scratch(int N) {
    return with_form(N, [](auto g) { return (size_t)decltype(g)::REF4; }) * 4 * (size_t)tile_ctas(N);
}

cudaError_t fem_tile_launch(const FemArgs& a, float* ref_scratch, int* counter, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    if (!fem_tile_form(a.N, a.precision, a.flow_cell != 0) || !a.kappa) return cudaErrorInvalidValue;
    const int grid = tile_grid(a.N, a.n);
    return with_form(a.N, [&](auto g) {
        using G = decltype(g);
        return a.rhs ? launch_one<G, true>(a, ref_scratch, grid, counter, st)
                     : launch_one<G, false>(a, ref_scratch, grid, counter, st);
    });
}

cudaError_t fem_tile_multi_launch(int N, const FemArgs* groups, const int* offsets, const int* item_group, int total,
                                  float* ref_scratch, int* counter, cudaStream_t st) {
    if (total <= 0) return cudaSuccess;
    if (!fem_tile_form(N, SMC_MIXED, false)) return cudaErrorInvalidValue;
    const int grid = tile_grid(N, total);
    return with_form(N, [&](auto g) {
        return launch_multi<decltype(g)>(groups, offsets, item_group, total, ref_scratch, grid, counter, st);
    });
}

}  // namespace mls2mc
