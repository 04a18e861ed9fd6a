// Register-tiled form of the mixed-precision forward solve on 1/64 and 1/32 (Dirichlet problem).
//
// The algorithm is the one of fem_solve.cu (KL field -> kappa -> 5-point stencil -> CG with a
// V(1,1) red-black multigrid preconditioner, double-float refinement, observations, misfit); what
// differs is who owns what. A thread owns a 4 x 4 patch of fine nodes and keeps the patch's CG
// residual r, direction p, sweep values e and all 40 edge weights in registers; only the patch's rim
// goes through shared memory. The 2 x 2 nodes of the next level that lie under the patch belong to
// the same thread, and on 1/64 the one node of 1/16 too, so restriction and prolongation mostly stay
// in registers as well. The levels 1/8 and 1/4 run in warp 0.
//
// Shared-memory layout: one array per position of the patch, indexed by thread ("position-major"),
// X[(4 b + a) P + thread] for node (4 tx + a, 4 ty + b). A read of one's own or a neighbouring patch's
// position is 32 consecutive words for a warp: no bank conflicts and one register per neighbour.
// Node columns and rows 0 are Dirichlet nodes whose stored values are always 0 (their inverse
// diagonal is 0), so the neighbour index may wrap around: the node to the right of column N - 1 is the
// next row's column 0, the node above row N - 1 is row 0, both 0 as they should be. What wraps on the
// left and below is only ever used by Dirichlet nodes, whose results are masked.
//
// Why this split: with one node per register slot and everything else in shared memory (the form of
// fem_solve.cu) a node update reads nine words from shared memory, 21 block barriers an iteration; that
// form (two 512-thread blocks an SM on 1/64) took 1.99 ms for 4000 particles on 1/64 and 0.42 ms on
// 1/32. Here a patch of 16 nodes reads 8 rim words per half sweep, 16 barriers an iteration, 256 threads
// of 128 registers, two blocks an SM (1/64) or 64 threads, eight blocks (1/32): 0.76 ms and 0.16 ms.
// What bounds it is latency: one 1/64 particle alone on an SM takes 0.87 of the time that two take
// together. A spill is what hurts most: the direction p lives in shared memory and addresses are formed
// where they are used, so that no register is spilled in the iteration (0.86 ms with a 20-word spill).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fem_device.h"
#include "internal.h"

namespace mls2mc {

namespace {

template <int N_>
struct Geo {
    static constexpr int N = N_, TX = N / 4, P = TX * TX, T = P, NW = T / 32;
    static constexpr bool L2 = N == 64;   // a one-node-per-thread level (1/16) between 2 x 2 and warp 0
    // blocks per SM the registers are sized for (128 a thread)
    static constexpr int MINB = 65536 / (128 * T);
    // shared memory, in floats
    static constexpr int E = 0;              // sweep values, later p or d: rim positions [16][P]; the
                                             // inner positions' slots carry red residuals
    static constexpr int D = E + 16 * P;     // CG correction d, float4 [4][P] (set-up: coarse kappa)
    static constexpr int PV = D + 16 * P;    // CG direction p, float4 [4][P] (not in registers during the V-cycle)
    static constexpr int ID = PV + 16 * P;   // inverse diagonals, float4 [red 2, black 2][P]
    static constexpr int W1 = ID + 16 * P;   // next level: weights (E, W, N, S) of (0,0) (1,1) (1,0) (0,1)
    static constexpr int ID1 = W1 + 16 * P;  // its inverse diagonals, float2 [red, black][P]
    static constexpr int E1 = ID1 + 4 * P;   // its values, positions A + 2 B
    static constexpr int W2 = E1 + 4 * P;    // 1/16 (on 1/64): weights, inverse diagonal, values
    static constexpr int ID2 = W2 + (L2 ? 4 * P : 0);
    static constexpr int E2 = ID2 + (L2 ? P : 0);
    static constexpr int R2 = E2 + (L2 ? P : 0);   // (1/16: red residuals)
    static constexpr int W8 = R2 + (L2 ? P : 0);   // 1/8: weights float4 [64], inverse diagonal, values, rhs
    static constexpr int ID8 = W8 + 256, E8 = ID8 + 64, R8 = E8 + 64;
    static constexpr int E4 = R8 + 64;       // 1/4: values [4][4], rhs [9], dense inverse [9][9]
    static constexpr int R4 = E4 + 16, DINV = R4 + 16;
    static constexpr int FLOATS = DINV + 84;
    // set-up staging inside D: kappa of the next level [8][P], of the one below it [2][P], of 1/8
    // [2][64] (1/32: the previous one), of 1/4 [2][16]
    static constexpr int K1 = D, K2 = D + 8 * P, K8 = L2 ? D + 10 * P : K2, K4 = D + 10 * P + 128;
    static constexpr int REF4 = 16 * P;      // float4s of refinement state of one block (device memory)
};

// sum over the block (the same value in every thread): warp sums in lane order, then in warp order
template <int NW>
__device__ __forceinline__ float block_total(float v, float* buf) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.f;
    if constexpr (NW % 4 == 0) {
#pragma unroll
        for (int i = 0; i < NW / 4; ++i) {
            const float4 q = reinterpret_cast<const float4*>(buf)[i];
            s += q.x;
            s += q.y;
            s += q.z;
            s += q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NW; ++i) s += buf[i];
    }
    return s;
}

__device__ __forceinline__ float off4(const float4 w, float e, float wv, float n, float s) {
    return w.x * e + w.y * wv + w.z * n + w.w * s;
}

// inverse (row-major, symmetric) of the 9 x 9 operator of level 1/4 by Gauss-Jordan elimination
// without pivoting (A is positive definite), by one warp: lane u < 9 keeps row u in registers, the pivot
// row comes by shuffles. It is a serial chain that the block waits for: one matrix entry per lane in
// shared memory with a branch per case took 12 K cycles, 9 % of the 1/64 solve.
__device__ __forceinline__ void invert9(const float* k4, float* dinv) {
    const int lane = threadIdx.x & 31, u = lane < 9 ? lane : 8;
    // kappa of the 4 x 4 cells: k4[2 c + t], c = J 4 + I, t = 0 lower, 1 upper half
    auto aE = [&](int I, int J) { return 0.5f * (k4[2 * (J * 4 + I)] + k4[2 * ((J - 1) * 4 + I) + 1]); };
    auto aN = [&](int I, int J) { return 0.5f * (k4[2 * (J * 4 + I - 1)] + k4[2 * (J * 4 + I) + 1]); };
    const int I = u % 3 + 1, J = u / 3 + 1;
    const float wE = aE(I, J), wW = aE(I - 1, J), wN = aN(I, J), wS = aN(I, J - 1);
    float a[9];
#pragma unroll
    for (int v = 0; v < 9; ++v)
        a[v] = v == u ? wE + wW + wN + wS
                      : v == u + 1 && I < 3 ? -wE : v == u - 1 && I > 1 ? -wW : v == u + 3 ? -wN : v == u - 3 ? -wS : 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        float row[9];
#pragma unroll
        for (int v = 0; v < 9; ++v) row[v] = __shfl_sync(0xffffffffu, a[v], k);
        const float ip = recip(row[k]);
        const float f = u == k ? -ip : a[k] * ip;   // row k itself becomes row k / pivot
#pragma unroll
        for (int v = 0; v < 9; ++v) a[v] = v == k ? -f : fmaf(-f, row[v], u == k ? 0.f : a[v]);
    }
    if (lane < 9)
#pragma unroll
        for (int v = 0; v < 9; ++v) dinv[9 * u + v] = a[v];
}

// the solve of particle `item` of a.n by the calling block (every thread of the block calls it).
// sm: Geo<N>::FLOATS floats, red: [2][8] reduction buffers, part: [8], ref: Geo<N>::REF4 float4 of device memory
// (this block's refinement state). RHS: the load vector may come from a table (a.rhs).
// take(): called by the block's last thread while the observations are formed (the next ticket).
template <int N, bool RHS, typename Take>
__device__ __forceinline__ void solve_tile(const FemArgs& a, const int item, float* sm, float (*red)[8], double* part,
                                           float4* ref, Take&& take) {
    using G = Geo<N>;
    constexpr int P = G::P, TX = G::TX, NW = G::NW;
    const int tid = threadIdx.x, lane = tid & 31;
    const int tx = tid % TX, ty = tid / TX;
    // neighbouring patches (wrapped; see above)
    const int pL = (tid - 1) & (P - 1), pR = (tid + 1) & (P - 1), pB = (tid - TX) & (P - 1), pA = (tid + TX) & (P - 1);
    // the diagonal ones, formed where they are used (opaque to the compiler, which would otherwise keep
    // them and the addresses derived from them in registers through the iteration and spill)
    auto diagonal = [&](int off) {
        int t = tid;
        asm volatile("" : "+r"(t));
        return (t + off) & (P - 1);
    };
    float* E = sm + G::E;
    float4* D4 = reinterpret_cast<float4*>(sm + G::D);
    float4* PV4 = reinterpret_cast<float4*>(sm + G::PV);
    float4* ID4 = reinterpret_cast<float4*>(sm + G::ID);
    float4* W1 = reinterpret_cast<float4*>(sm + G::W1);
    float2* ID1 = reinterpret_cast<float2*>(sm + G::ID1);
    float* E1 = sm + G::E1;
    float4* W2 = reinterpret_cast<float4*>(sm + G::W2);
    float* ID2 = sm + G::ID2;
    float* E2 = sm + G::E2;
    float4* W8 = reinterpret_cast<float4*>(sm + G::W8);
    float *ID8 = sm + G::ID8, *E8 = sm + G::E8, *R8 = sm + G::R8, *E4 = sm + G::E4, *R4 = sm + G::R4, *DI = sm + G::DINV;
    // a node of the patch on the Dirichlet column or row
    auto dirichlet = [&](int i, int j) { return (i == 0 && tx == 0) || (j == 0 && ty == 0); };

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
                sm[G::K1 + (2 * (A + 2 * B)) * P + tid] = cl[B][A];
                sm[G::K1 + (2 * (A + 2 * B) + 1) * P + tid] = cu[B][A];
            }
        sm[G::K2 + tid] = 0.25f * (cl[0][0] + cl[0][1] + cu[0][1] + cl[1][1]);
        sm[G::K2 + P + tid] = 0.25f * (cu[0][0] + cu[1][0] + cl[1][0] + cu[1][1]);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)   // inverse diagonals: colour c, rows 0 1 and rows 2 3
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int b = 2 * h + q / 2, i = 2 * (q % 2) + ((b & 1) ^ c);
                const float d = wE[b][i + 1] + wE[b][i] + wN[b + 1][i] + wN[b][i];
                v[q] = dirichlet(i, b) ? 0.f : d == 0.f ? 1.f : recip(d);
            }
            ID4[(2 * c + h) * P + tid] = make_float4(v[0], v[1], v[2], v[3]);
        }
    __syncthreads();
    {   // next level: the weights of the 2 x 2 nodes
        float lo[3][3], up[3][3];   // cells (-1 .. 1)^2, index [row + 1][column + 1]
        const int pD = diagonal(-TX - 1);
        auto K = [&](int pos, int t, int p) { return sm[G::K1 + (2 * pos + t) * P + p]; };
        lo[1][0] = K(1, 0, pL); up[1][0] = K(1, 1, pL); lo[2][0] = K(3, 0, pL);
        lo[0][0] = K(3, 0, pD); up[0][0] = K(3, 1, pD);
        lo[0][1] = K(2, 0, pB); up[0][1] = K(2, 1, pB); up[0][2] = K(3, 1, pB);
#pragma unroll
        for (int pos = 0; pos < 4; ++pos) {
            lo[1 + pos / 2][1 + pos % 2] = K(pos, 0, tid);
            up[1 + pos / 2][1 + pos % 2] = K(pos, 1, tid);
        }
        auto w = [&](int A, int B) {
            return make_float4(0.5f * (lo[B + 1][A + 1] + up[B][A + 1]), 0.5f * (lo[B + 1][A] + up[B][A]),
                               0.5f * (lo[B + 1][A] + up[B + 1][A + 1]), 0.5f * (lo[B][A] + up[B][A + 1]));
        };
        auto inv = [&](const float4& x, int A, int B) {
            return dirichlet(A, B) ? 0.f : recip_coarse(x.x + x.y + x.z + x.w);
        };
        const float4 w00 = w(0, 0), w11 = w(1, 1), w10 = w(1, 0), w01 = w(0, 1);
        W1[tid] = w00;
        W1[P + tid] = w11;
        W1[2 * P + tid] = w10;
        W1[3 * P + tid] = w01;
        ID1[tid] = make_float2(inv(w00, 0, 0), inv(w11, 1, 1));
        ID1[P + tid] = make_float2(inv(w10, 1, 0), inv(w01, 0, 1));
        if constexpr (G::L2) {
            const float *lo2 = sm + G::K2, *up2 = sm + G::K2 + P;
            const float4 v = make_float4(0.5f * (lo2[tid] + up2[pB]), 0.5f * (lo2[pL] + up2[pD]),
                                         0.5f * (lo2[pL] + up2[tid]), 0.5f * (lo2[pD] + up2[pB]));
            W2[tid] = v;
            ID2[tid] = inv(v, 0, 0);
            E2[tid] = 0.f;   // see E8 below
        }
    }
    if (tid < 32) {   // levels 1/8 and 1/4: warp 0 alone (nothing else touches D or the small arrays yet)
        float *k8l = sm + G::K8, *k8u = k8l + 64;
        if constexpr (G::L2) {
            const float *lo2 = sm + G::K2, *up2 = sm + G::K2 + P;
#pragma unroll
            for (int c = lane; c < 64; c += 32) {
                const int f = (c >> 3) * 2 * TX + (c & 7) * 2;   // fine cell (2 I, 2 J) of 16 x 16
                k8l[c] = 0.25f * (lo2[f] + lo2[f + 1] + up2[f + 1] + lo2[f + TX + 1]);
                k8u[c] = 0.25f * (up2[f] + up2[f + TX] + lo2[f + TX] + up2[f + TX + 1]);
            }
            __syncwarp();
        }
#pragma unroll
        for (int c = lane; c < 64; c += 32) {
            const int l = (c - 1) & 63, b = (c - 8) & 63, d = (c - 9) & 63;
            const float4 v = make_float4(0.5f * (k8l[c] + k8u[b]), 0.5f * (k8l[l] + k8u[d]), 0.5f * (k8l[l] + k8u[c]),
                                         0.5f * (k8l[d] + k8u[b]));
            W8[c] = v;
            ID8[c] = ((c & 7) == 0 || c < 8) ? 0.f : recip_coarse(v.x + v.y + v.z + v.w);
            // one node per lane: the wrapped neighbour of the last column is a Dirichlet node of the
            // reader's own colour, read before its first (zero) value is stored
            E8[c] = 0.f;
        }
        float* k4 = sm + G::K4;
        if (lane < 16) {
            const int f = (lane >> 2) * 16 + (lane & 3) * 2;
            k4[2 * lane] = 0.25f * (k8l[f] + k8l[f + 1] + k8u[f + 1] + k8l[f + 9]);
            k4[2 * lane + 1] = 0.25f * (k8u[f] + k8u[f + 8] + k8l[f + 8] + k8u[f + 9]);
            E4[lane] = 0.f;
        }
        __syncwarp();
        invert9(k4, DI);
    }

    // ---- rim exchange: colour c's values of the neighbouring patches next to the patch's other colour
    float hL[4], hR[4], hB[4], hA[4];
    auto load_halo = [&](int c) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (((3 + k) & 1) == c) {
                hL[k] = E[(4 * k + 3) * P + pL];
                hB[k] = E[(12 + k) * P + pB];
            } else {
                hR[k] = E[(4 * k) * P + pR];
                hA[k] = E[k * P + pA];
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
                    E[(4 * b + i) * P + tid] = v[b][i];
    };
    // off-diagonal sum at patch node (i, b) of v, rim neighbours from the halo
    auto off = [&](const float (&v)[4][4], int i, int b) {
        return wE[b][i + 1] * (i < 3 ? v[b][i < 3 ? i + 1 : 3] : hR[b]) + wE[b][i] * (i > 0 ? v[b][i > 0 ? i - 1 : 0] : hL[b]) +
               wN[b + 1][i] * (b < 3 ? v[b < 3 ? b + 1 : 3][i] : hA[i]) + wN[b][i] * (b > 0 ? v[b > 0 ? b - 1 : 0][i] : hB[i]);
    };
    auto inv_diag = [&](int c, float (&v)[8]) {   // this thread's inverse diagonals of colour c, in node order
        const float4 x = ID4[2 * c * P + tid], y = ID4[(2 * c + 1) * P + tid];
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    };

    const float h2 = 1.f / (float(N) * float(N));   // f = 1: exact in FP32
    auto load_b = [&](int i, int b, float& hi, float& lo) {   // the load vector at a node of the patch
        hi = h2;
        lo = 0.f;
        if (RHS && a.rhs) {
            const float2 v = static_cast<const float2*>(a.rhs)[(4 * ty + b) * fem_row_stride(N) + 4 * tx + i];
            hi = v.x;
            lo = v.y;
        }
        if (dirichlet(i, b)) hi = lo = 0.f;
    };
    const float bnorm2 = (RHS && a.rhs) ? float(a.bnorm2) : float((N - 1) * (N - 1)) * h2 * h2;
    const float stop_outer = float(a.rtol * a.rtol) * bnorm2;
    const float stop_last = float(0.25 * a.rtol * a.rtol) * bnorm2;
    const float rtol_in2 = float(a.rtol_in * a.rtol_in);
    int parity = 0, total_it = 0;
    bool converged = false, have_x = false;

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
                const float4 v = ref[b * P + tid];
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
        const float rr0 = block_total<NW>(rr, red[parity]);
        parity ^= 1;
        if (!(rr0 > 0.f)) break;
        const float stop2 = fmaxf(rtol_in2 * rr0, stop_last);
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
            __syncthreads();
            // red residuals (off-diagonal sums of the black values); the three that the neighbours'
            // coarse nodes read go into the slots of inner positions
            float v00, v10, v01, v11;   // coarse right-hand side under the patch
            {
                load_halo(1);
                const float s00 = off(e, 0, 0), s20 = off(e, 2, 0), s02 = off(e, 0, 2), s22 = off(e, 2, 2);
                const float s11 = off(e, 1, 1), s31 = off(e, 3, 1), s13 = off(e, 1, 3), s33 = off(e, 3, 3);
                E[5 * P + tid] = s33;
                E[6 * P + tid] = s13;
                E[9 * P + tid] = s31;
                __syncthreads();
                v00 = s00 + 0.5f * (s11 + E[5 * P + diagonal(-TX - 1)]);
                v10 = s20 + 0.5f * (s31 + E[6 * P + pB]);
                v01 = s02 + 0.5f * (s13 + E[9 * P + pL]);
                v11 = s22 + 0.5f * (s33 + s11);
            }
            float e00, e10, e01, e11;   // the coarse nodes of the patch
            {
                const float2 idr = ID1[tid];
                e00 = v00 * idr.x;
                e11 = v11 * idr.y;
                E1[tid] = e00;
                E1[3 * P + tid] = e11;
            }
            __syncthreads();
            {   // coarse black pre-sweep
                const float2 idb = ID1[P + tid];
                e10 = (v10 + off4(W1[2 * P + tid], E1[pR], e00, e11, E1[3 * P + pB])) * idb.x;
                e01 = (v01 + off4(W1[3 * P + tid], e11, E1[3 * P + pL], E1[pA], e00)) * idb.y;
                E1[P + tid] = e10;
                E1[2 * P + tid] = e01;
            }
            __syncthreads();
            float v2;   // right-hand side of the node (tx, ty) two levels down
            {
                const int pD = diagonal(-TX - 1);
                const float l10 = E1[P + pL], b01 = E1[2 * P + pB];
                const float s00 = off4(W1[tid], e10, l10, e01, b01);
                const float s11 = off4(W1[P + tid], E1[2 * P + pR], e01, E1[P + pA], e10);
                const float sdd = off4(W1[P + pD], b01, E1[2 * P + pD], l10, E1[P + pD]);
                v2 = s00 + 0.5f * (s11 + sdd);
            }
            const bool red2 = ((tx + ty) & 1) == 0;
            float e2 = 0.f;
            if constexpr (G::L2) {
                if (red2) {
                    e2 = v2 * ID2[tid];
                    E2[tid] = e2;
                }
                __syncthreads();
                if (!red2) {
                    e2 = (v2 + off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB])) * ID2[tid];
                    E2[tid] = e2;
                }
                __syncthreads();
                // every node's residual once (red: the off-diagonal sum; a black node's is not used), so
                // that warp 0 only adds up three values per node of 1/8
                sm[G::R2 + tid] = off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB]);
                __syncthreads();
            } else {
                R8[tid] = v2;
                if (red2) E8[tid] = v2 * ID8[tid];
                __syncthreads();
            }
            if (tid < 32) {   // levels 1/8 and 1/4 in warp 0; node c = 8 J + I
                // the lane made opaque: the addresses below are computed here instead of being hoisted
                // out of the iteration into registers that do not exist (spills)
                int ln = lane;
                asm volatile("" : "+r"(ln));
                const int J = ln >> 2;
                const int cr = 8 * J + 2 * (ln & 3) + (J & 1), cb = cr ^ 1;   // this ln's red and black node
                float rr8, rb8;
                if constexpr (G::L2) {
                    const float* R2 = sm + G::R2;
                    const int fr = 2 * J * TX + 2 * (cr & 7), fb = 2 * J * TX + 2 * (cb & 7);
                    rr8 = R2[fr] + 0.5f * (R2[fr + TX + 1] + R2[(fr - TX - 1) & (P - 1)]);
                    rb8 = R2[fb] + 0.5f * (R2[fb + TX + 1] + R2[(fb - TX - 1) & (P - 1)]);
                    E8[cr] = rr8 * ID8[cr];
                    __syncwarp();
                } else {
                    rr8 = R8[cr];
                    rb8 = R8[cb];
                }
                auto s8 = [&](int f) {
                    return off4(W8[f], E8[(f + 1) & 63], E8[(f - 1) & 63], E8[(f + 8) & 63], E8[(f - 8) & 63]);
                };
                E8[cb] = (rb8 + s8(cb)) * ID8[cb];
                __syncwarp();
                R8[cr] = s8(cr);   // red residuals
                __syncwarp();
                if (ln < 9) {
                    const int f = (ln / 3 + 1) * 16 + (ln % 3 + 1) * 2;
                    R4[ln] = R8[f] + 0.5f * (R8[f + 9] + R8[f - 9]);
                }
                __syncwarp();
                if (ln < 9) {   // 1/4 solved exactly (the inverse is symmetric: column reads)
                    float acc = 0.f;
#pragma unroll
                    for (int v = 0; v < 9; ++v) acc = fmaf(DI[9 * v + ln], R4[v], acc);
                    E4[(ln / 3 + 1) * 4 + ln % 3 + 1] = acc;
                }
                __syncwarp();
                {   // black post-sweep with the prolongation
                    const int c0 = (J >> 1) * 4 + ((cb & 7) >> 1);
                    const bool jeven = (J & 1) == 0;
                    const float x0 = E4[c0], x1 = E4[(c0 + 5) & 15];
                    const float xu = E4[(jeven ? c0 + 1 : c0 + 4) & 15], xv = E4[(jeven ? c0 - 4 : c0 - 1) & 15];
                    const float dg = 0.5f * (x0 + x1), hf = 0.5f * (xv + xu);
                    const float4 w = W8[cb];
                    const float s = w.x * (E8[(cb + 1) & 63] + (jeven ? xu : dg)) + w.y * (E8[(cb - 1) & 63] + (jeven ? x0 : hf)) +
                                    w.z * (E8[(cb + 8) & 63] + (jeven ? dg : xu)) + w.w * (E8[(cb - 8) & 63] + (jeven ? hf : x0));
                    E8[cb] = (rb8 + s) * ID8[cb];
                }
                __syncwarp();
                E8[cr] = (rr8 + s8(cr)) * ID8[cr];
            }
            __syncthreads();
            const float* e2s = E2;   // values of the level of one node per thread
            if constexpr (G::L2) {
                if (!red2) {   // black post-sweep with the correction of 1/8
                    const int c0 = (ty >> 1) * 8 + (tx >> 1);
                    const bool jeven = (ty & 1) == 0;
                    const float x0 = E8[c0], x1 = E8[(c0 + 9) & 63];
                    const float xu = E8[(jeven ? c0 + 1 : c0 + 8) & 63], xv = E8[(jeven ? c0 - 8 : c0 - 1) & 63];
                    const float dg = 0.5f * (x0 + x1), hf = 0.5f * (xv + xu);
                    const float4 w = W2[tid];
                    const float s = w.x * (E2[pR] + (jeven ? xu : dg)) + w.y * (E2[pL] + (jeven ? x0 : hf)) +
                                    w.z * (E2[pA] + (jeven ? dg : xu)) + w.w * (E2[pB] + (jeven ? hf : x0));
                    E2[tid] = (v2 + s) * ID2[tid];
                }
                __syncthreads();
                if (red2) E2[tid] = (v2 + off4(W2[tid], E2[pR], E2[pL], E2[pA], E2[pB])) * ID2[tid];
                __syncthreads();
            } else {
                e2s = E8;
            }
            {   // 2 x 2 level, black post-sweep: red neighbours with the correction of the level below
                const float c0 = e2s[tid], cR = e2s[pR], cA = e2s[pA], cU = e2s[diagonal(TX + 1)], cL = e2s[pL], cB = e2s[pB];
                const float2 idb = ID1[P + tid];
                const float f00 = e00 + c0, f11 = e11 + 0.5f * (c0 + cU);
                const float fR = E1[pR] + cR, fA = E1[pA] + cA;
                const float fB = E1[3 * P + pB] + 0.5f * (cB + cR), fL = E1[3 * P + pL] + 0.5f * (cL + cA);
                e10 = (v10 + off4(W1[2 * P + tid], fR, f00, f11, fB)) * idb.x;
                e01 = (v01 + off4(W1[3 * P + tid], f11, fL, fA, f00)) * idb.y;
                E1[P + tid] = e10;
                E1[2 * P + tid] = e01;
            }
            __syncthreads();
            {   // red post-sweep
                const float2 idr = ID1[tid];
                e00 = (v00 + off4(W1[tid], e10, E1[P + pL], e01, E1[2 * P + pB])) * idr.x;
                e11 = (v11 + off4(W1[P + tid], E1[2 * P + pR], e01, E1[P + pA], e10)) * idr.y;
                E1[tid] = e00;
                E1[3 * P + tid] = e11;
            }
            __syncthreads();
            {   // fine black post-sweep: red values plus the prolonged correction
                load_halo(0);
                const float c20 = E1[pR], c21 = E1[2 * P + pR], c02 = E1[pA], c12 = E1[P + pA], c22 = E1[diagonal(TX + 1)];
                const float cm0 = E1[P + pL], cm1 = E1[3 * P + pL], c0m = E1[2 * P + pB], c1m = E1[3 * P + pB];
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
            __syncthreads();
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
            rz_new = block_total<NW>(rz_new, red[parity]);
            parity ^= 1;
            const float beta = it == 0 ? 0.f : rz_new / rz;
            rz = rz_new;
            float p[4][4];   // p = z + beta p
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                float4 v = make_float4(e[b][0], e[b][1], e[b][2], e[b][3]);
                if (it > 0) {
                    const float4 o = PV4[b * P + tid];
                    v.x += beta * o.x;
                    v.y += beta * o.y;
                    v.z += beta * o.z;
                    v.w += beta * o.w;
                }
                PV4[b * P + tid] = v;
                p[b][0] = v.x; p[b][1] = v.y; p[b][2] = v.z; p[b][3] = v.w;
            }
            store_rim(2, p);
            __syncthreads();
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
                    if (dirichlet(i, b)) q = 0.f;
                    e[b][i] = q;
                    pq += c * q;
                }
            pq = block_total<NW>(pq, red[parity]);
            parity ^= 1;
            const float alpha = rz / pq;
            rr = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                float4 d = it == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : D4[b * P + tid];
                d.x = fmaf(alpha, p[b][0], d.x);
                d.y = fmaf(alpha, p[b][1], d.y);
                d.z = fmaf(alpha, p[b][2], d.z);
                d.w = fmaf(alpha, p[b][3], d.w);
                D4[b * P + tid] = d;
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
            rr = block_total<NW>(rr, red[parity]);
            parity ^= 1;
            ++total_it;
            if (!(rr > stop2)) break;   // also leaves on NaN
        }
        // ---- refinement: x += d, r -= A d in double-float arithmetic (edge form) ----
        float p[4][4];   // d
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float4 d = D4[b * P + tid];
            p[b][0] = d.x; p[b][1] = d.y; p[b][2] = d.z; p[b][3] = d.w;
        }
        store_rim(2, p);
        __syncthreads();
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
                const float4 v0 = ref[b * P + tid], v1 = ref[(4 + b) * P + tid], v2 = ref[(8 + b) * P + tid],
                             v3 = ref[(12 + b) * P + tid];
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
                // r -= (east + north) - (west + south): high parts by TwoSum, the rest in one low part
                float h = rh[i], l = rl[i], t;
                two_sum(h, -eh, h, t);
                l += t - el;
                two_sum(h, wsh, h, t);
                l += t + wsl;
                two_sum(h, -nh, h, t);
                l += t - nl;
                two_sum(h, sth[i], h, t);
                l += t + stl[i];
                rh[i] = h + l;
                rl[i] = l - (rh[i] - h);
                if (dirichlet(i, b)) rh[i] = rl[i] = 0.f;
                rr_out += rh[i] * rh[i];
                wsh = eh;
                wsl = el;
                sth[i] = nh;
                stl[i] = nl;
            }
            ref[b * P + tid] = make_float4(rh[0], rh[1], rh[2], rh[3]);
            ref[(4 + b) * P + tid] = make_float4(rl[0], rl[1], rl[2], rl[3]);
            ref[(8 + b) * P + tid] = make_float4(xh[0], xh[1], xh[2], xh[3]);
            ref[(12 + b) * P + tid] = make_float4(xl[0], xl[1], xl[2], xl[3]);
        }
        have_x = true;
        rr_out = block_total<NW>(rr_out, red[parity]);
        parity ^= 1;
        converged = rr_out <= stop_outer;
    }

    // ---- observations and misfit (FP64): the solution's double-float pairs go to shared memory
    // (over E and D), one warp gathers ----
    float2* xs = reinterpret_cast<float2*>(sm + G::E);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        float4 xh = make_float4(0.f, 0.f, 0.f, 0.f), xl = xh;
        if (have_x) {
            xh = ref[(8 + b) * P + tid];
            xl = ref[(12 + b) * P + tid];
        }
        xs[(4 * b) * P + tid] = make_float2(xh.x, xl.x);
        xs[(4 * b + 1) * P + tid] = make_float2(xh.y, xl.y);
        xs[(4 * b + 2) * P + tid] = make_float2(xh.z, xl.z);
        xs[(4 * b + 3) * P + tid] = make_float2(xh.w, xl.w);
    }
    __syncthreads();
    auto val = [&](int n) -> double {   // n = j (N + 2) + i
        const int j = n / fem_row_stride(N), i = n - j * fem_row_stride(N);
        if (i < 1 || i >= N || j < 1 || j >= N) return 0.0;
        const float2 v = xs[(4 * (j & 3) + (i & 3)) * P + (j >> 2) * TX + (i >> 2)];
        return (double)v.x + (double)v.y;
    };
    if (tid == G::T - 1) take();   // the ticket's latency overlaps the observations
    double misfit = 0.0;
    for (int o = tid; o < a.n_obs; o += G::T) {
        const double g = a.obs_w[3 * o] * val(a.obs_idx[3 * o]) + a.obs_w[3 * o + 1] * val(a.obs_idx[3 * o + 1]) +
                         a.obs_w[3 * o + 2] * val(a.obs_idx[3 * o + 2]);
        if (a.G) a.G[(size_t)item * a.n_obs + o] = g;
        const double rdf = a.y[o] - g;
        misfit += rdf * rdf;
    }
    const int nw = min(NW, (a.n_obs + 31) / 32);   // warps that hold observations
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
    }
}

// persistent blocks take particles from a ticket counter
template <int N, bool RHS>
__global__ void __launch_bounds__(Geo<N>::T, Geo<N>::MINB) fem_tile_kernel(FemArgs a, float4* ref_scratch, int* counter) {
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(16) float red[2][8];
    __shared__ double part[8];
    __shared__ int item_s;
    float4* ref = ref_scratch + (size_t)blockIdx.x * Geo<N>::REF4;
    if (threadIdx.x == 32) item_s = atomicAdd(counter, 1);
    __syncthreads();
    for (;;) {
        const int item = item_s;
        if (item >= a.n) break;
        solve_tile<N, RHS>(a, item, sm, red, part, ref, [&] { item_s = atomicAdd(counter, 1); });
        __syncthreads();
    }
}

// many problems: the same loop over (problem, particle) items; the item's launch arguments are copied
// to shared memory (two copies: the next item's arrive while the current one's are in use)
template <int N>
__global__ void __launch_bounds__(Geo<N>::T, Geo<N>::MINB)
    fem_tile_multi(const FemArgs* groups, const int* offsets, const int* item_group, int total, float4* ref_scratch,
                   int* counter) {
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(16) float red[2][8];
    __shared__ double part[8];
    __shared__ int item_s[2], p_s[2];
    __shared__ FemArgs args_s[2];
    float4* ref = ref_scratch + (size_t)blockIdx.x * Geo<N>::REF4;
    auto take = [&](int k) {
        const int item = atomicAdd(counter, 1);
        item_s[k] = item;
        if (item < total) {
            const int g = item_group[item];
            args_s[k] = groups[g];
            p_s[k] = item - offsets[g];
        }
    };
    if (threadIdx.x == 32) take(0);
    __syncthreads();
    for (int k = 0; item_s[k] < total; k ^= 1) {
        solve_tile<N, true>(args_s[k], p_s[k], sm, red, part, ref, [&] { take(k ^ 1); });
        __syncthreads();
    }
}

template <int N>
constexpr size_t tile_smem() {
    return sizeof(float) * (size_t)Geo<N>::FLOATS;
}

template <int N>
cudaError_t set_smem() {
    cudaError_t e = cudaFuncSetAttribute(fem_tile_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tile_smem<N>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fem_tile_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)tile_smem<N>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fem_tile_multi<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem<N>());
    return e;
}

template <int N>
int resident_blocks() {
    int dev = 0, sms = 0, per_sm = 0, multi = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (set_smem<N>() != cudaSuccess) return 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fem_tile_kernel<N, false>, Geo<N>::T, tile_smem<N>());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&multi, fem_tile_multi<N>, Geo<N>::T, tile_smem<N>());
    return sms * std::max(1, std::max(per_sm, multi));
}

template <int N>
cudaError_t launch(const FemArgs& a, float* ref_scratch, int grid, int* counter, cudaStream_t st) {
    cudaError_t e = set_smem<N>();
    if (e != cudaSuccess) return e;
    float4* ref = reinterpret_cast<float4*>(ref_scratch);
    if (a.rhs) fem_tile_kernel<N, true><<<grid, Geo<N>::T, tile_smem<N>(), st>>>(a, ref, counter);
    else fem_tile_kernel<N, false><<<grid, Geo<N>::T, tile_smem<N>(), st>>>(a, ref, counter);
    count_launches(1);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_multi(const FemArgs* groups, const int* offsets, const int* item_group, int total, float* ref_scratch,
                         int grid, int* counter, cudaStream_t st) {
    cudaError_t e = set_smem<N>();
    if (e != cudaSuccess) return e;
    fem_tile_multi<N><<<grid, Geo<N>::T, tile_smem<N>(), st>>>(groups, offsets, item_group, total,
                                                               reinterpret_cast<float4*>(ref_scratch), counter);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

bool fem_tile_form(int N, int precision, bool flow_cell) {
    return (N == 64 || N == 32) && precision == SMC_MIXED && !flow_cell;
}

int fem_tile_blocks(int N) {
    static int cached[64][2] = {};   // resident blocks, queried once per device and level
    int dev = 0;
    cudaGetDevice(&dev);
    const int c = N == 64 ? 0 : 1;
    if (dev >= 0 && dev < 64 && cached[dev][c] > 0) return cached[dev][c];
    const int blocks = N == 64 ? resident_blocks<64>() : N == 32 ? resident_blocks<32>() : 0;
    if (dev >= 0 && dev < 64 && blocks > 0) cached[dev][c] = blocks;
    return blocks;
}

size_t fem_tile_scratch(int N) {
    const size_t f4 = N == 64 ? Geo<64>::REF4 : Geo<32>::REF4;
    return (size_t)fem_tile_blocks(N) * f4 * 4;
}

cudaError_t fem_tile_launch(const FemArgs& a, float* ref_scratch, int* counter, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    if (!fem_tile_form(a.N, a.precision, a.flow_cell != 0) || !a.kappa) return cudaErrorInvalidValue;
    const int grid = std::min(a.n, fem_tile_blocks(a.N));
    if (grid < 1) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    return a.N == 64 ? launch<64>(a, ref_scratch, grid, counter, st) : launch<32>(a, ref_scratch, grid, counter, st);
}

cudaError_t fem_tile_multi_launch(int N, const FemArgs* groups, const int* offsets, const int* item_group, int total,
                                  float* ref_scratch, int* counter, cudaStream_t st) {
    if (total <= 0) return cudaSuccess;
    const int grid = std::min(total, fem_tile_blocks(N));
    if (grid < 1) return cudaErrorInvalidConfiguration;
    if (N == 64) return launch_multi<64>(groups, offsets, item_group, total, ref_scratch, grid, counter, st);
    if (N == 32) return launch_multi<32>(groups, offsets, item_group, total, ref_scratch, grid, counter, st);
    return cudaErrorInvalidValue;
}

}  // namespace mls2mc
