// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/mls2mc.h"

namespace mls2mc {

// ---- host set-up (kl_host.cpp) ---------------------------------------------------------
void kl_eig_1d(double corr_len, int n_modes, std::vector<double>& lam, std::vector<double>& omega);
void kl_table(int N, double corr_len, double variance, int K, std::vector<double>& psi,
              std::vector<double>& lambda);
// eigen-decomposition of a symmetric n x n matrix a (row-major, destroyed) (sym_eigen.cpp):
// eigenvalues to w (unordered), eigenvector i to row i of vt; false if the QR iteration stalls
bool symmetric_eigen(int n, std::vector<double>& a, std::vector<double>& w, std::vector<double>& vt);
// Matern (smoothness 3/2) KL table by the Nystrom method (matern_host.cpp); K <= matern_max_terms()
// (false if the eigen-solve failed)
int matern_max_terms();
bool matern_kl_table(int N, double corr_len, double variance, int K, std::vector<double>& psi,
                     std::vector<double>& lambda);
// load vector of the nine-source term of Example 5.1 at the nodes of level N (padded row layout
// below, zero at Dirichlet nodes and padding); bnorm2 = sum of squares over the interior nodes
void nine_source_load(int N, std::vector<double>& b, double& bnorm2);
// Nodes of a level with NL cells per side are stored row by row with row stride NL + 2 (one
// padding word per row, never read): with an even stride, nodes of one red-black colour in two
// adjacent rows fall on shared-memory banks of opposite parity.
__host__ __device__ constexpr int fem_row_stride(int NL) { return NL + 2; }
// node indices j * fem_row_stride(N) + i of the three P1 vertices of each observation
void obs_table(int N, int n_obs, const double* xy, std::vector<int>& idx, std::vector<double>& wts);

// ---- kernel launch counter (api.cpp): every kernel the library launches is counted ------
void count_launches(long long n);
long long launch_count();

// ---- forward solve (fem_solve.cu) -------------------------------------------------------
struct FemArgs {
    int N;                  // cells per side of this level (power of two, 4..256)
    int precision;          // SMC_FP64 or SMC_MIXED
    int n;                  // particles
    int K;                  // KL terms
    const double* theta;    // [n][K] device
    const void* psi;        // [K][2N^2] device, double (FP64) or float (MIXED)
    const float* kappa;     // [n][2N^2] kappa = exp(u) per triangle (MIXED: from the tensor-core synthesis), or null
    const int* obs_idx;     // [n_obs][3] node indices j * fem_row_stride(N) + i
    const double* obs_w;    // [n_obs][3] P1 weights
    int n_obs;
    const double* y;        // [n_obs]
    double inv_sigma2;      // 1 / sigma^2
    double* G;              // [n][n_obs] or null
    double* Phi;            // [n]
    int* iters;             // [n] or null
    double rtol;            // FP64 relative residual target
    double rtol_in;         // relative reduction of each inner CG pass
    int max_outer;          // refinement passes
    int max_inner;          // inner CG iterations per pass
    const void* rhs;        // load vector at the nodes (padded row layout): double (FP64) or float2
                            // (MIXED: hi, lo with hi + lo = the FP64 value); null: f = 1 (b = h^2)
    double bnorm2;          // sum of squares of the load vector over the interior nodes (with rhs)
    int flow_cell;          // 1: the flow cell of Example 5.3 (p = 0 / 1 on x = 0 / 1, no flow on
                            // y = 0, 1, f = 0; levels 1/8 .. 1/256, FP64 to 1/32; no batched form)
    unsigned* bad;          // += solves that did not reach rtol, or null (fem_tile_launch only)
};
// Returns cudaSuccess or the launch error.
// T = the block size (one of fem_block_sizes; <= 0: the first)
cudaError_t fem_eval_launch(const FemArgs& a, cudaStream_t stream, int T = 0);
std::vector<int> fem_block_sizes(int N, int precision);
// those of them that are different kernels, the default first: what the autotuner times
std::vector<int> fem_block_forms(int N, int precision);
// the size used when none is set
int fem_default_block(int N, int precision);
// large levels (1/h = 128, 256; mixed precision, kappa from the synthesis): hierarchy in global
// scratch, blocks x fem_global_slice(N) floats; *counter (device) is reset by the launch
size_t fem_global_slice(int N, bool FC = false);   // FC: the flow cell's layout
int fem_global_blocks(int N);
cudaError_t fem_eval_global_launch(const FemArgs& a, float* scratch, int blocks, int* counter, cudaStream_t st);
// large levels of many problems (groups, offsets, item_group as for fem_eval_persistent_launch;
// *counter zero before the launch), blocks x fem_global_slice(N) floats of scratch
cudaError_t fem_eval_global_multi_launch(int N, const FemArgs* groups, const int* offsets, const int* item_group,
                                         int total, float* scratch, int blocks, int* counter, cudaStream_t st);
// persistent multi-problem launch: groups[g] (device array) are the launch arguments of one
// problem at level size N; offsets[g] (device) the first work item of group g; item_group[i]
// (device) the group of item i; *counter (device, zero before the launch) hands out the total
// items to the blocks
cudaError_t fem_eval_persistent_launch(int N, int precision, int T, const FemArgs* groups, const int* offsets,
                                       const int* item_group, int total, int* counter, cudaStream_t st);
// register-tiled form of the mixed solve (fem_tile.cu): 1/32 and 1/64 on one CTA (every block size of those
// levels), 1/128 on a cluster of two CTAs (block size -1024), 1/256 of eight; not the flow cell. Where a
// cluster does not fit, 1/128 and 1/256 run in the device-memory form above. fem_tile_scratch floats of device
// scratch hold the refinement state. *counter (device) is 0 before a launch (fem_tile_launch: zeroed by the
// evaluation's Handle::synth_kappa); fem_tile_multi_launch: arguments as fem_eval_persistent_launch
bool fem_tile_form(int N, int precision, bool flow_cell);
size_t fem_tile_scratch(int N);
cudaError_t fem_tile_launch(const FemArgs& a, float* scratch, int* counter, cudaStream_t st);
cudaError_t fem_tile_multi_launch(int N, const FemArgs* groups, const int* offsets, const int* item_group, int total,
                                  float* scratch, int* counter, cudaStream_t st);
// device scratch (floats) of a many-problem launch on level N: the large levels', the tile form's, else 0
size_t fem_multi_scratch(int N, int precision);
bool fem_level_supported(int N, int precision);

}  // namespace mls2mc
