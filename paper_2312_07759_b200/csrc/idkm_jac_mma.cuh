// Explicit Jacobian J_C = dF/dC on the tensor cores (tcgen05), for codebooks of more than 8 centroids in d = 2 or 4.
//
//   J[(j,a),(l,b)] = sum_i P_ija (delta_jl - A_il) n_ilb = Dg - X^T Y,   P_ija = A_ij (w_ia - F_ja) / (S_j tau),
//   X_i[(j,a)] = P_ija,   Y_i[(l,b)] = A_il n_ilb,   Dg[(j,a),(j,b)] = sum_i P_ija n_ijb       (Section 4.2)
//
// X^T Y is a contraction over the m weights with k d rows and columns: a matrix product of m (k d)^2 multiply-adds that
// replaces adj_max_iter passes over the weights.
#pragma once
#include "idkm_kernels.cuh"

namespace idkm {

constexpr int JM_THREADS = 512;        // 8 accumulating warps (the first also issues the products), 8 producing warps
constexpr int JM_ROWS = 64;            // weights per stage
constexpr int JM_M = 128;              // rows (j, a) of a tile
constexpr int JM_FOLD = 256;           // stages after which the fp32 sums move into the fp64 partial
constexpr int JM_UNITS = 148;          // blocks the splits of one call are dealt to
constexpr int JM_SYNC_WORDS = 32;
constexpr size_t JM_PART_MAX = 96u << 20;   // workspace for partial tiles

struct JacMmaParams {
  const float* W;
  const float *C, *S, *F, *gvec;
  float* u;
  const float2* rowstat;
  LayerState* st;
  float* hist_adj;
  double* part;            // one partial tile per slot (idkm_jac_mma.cu)
  unsigned int* gtickets;  // arrivals of the groups of blocks that add up their partials; zero at rest
  double* ub;              // [2][L][kdp] the adjoint, by permuted coordinate, alternating by step
  double* pn;              // [2][L][blocks per layer][2] squares of the step and of the adjoint
  unsigned int* sync;      // [L][JM_SYNC_WORDS] barrier words of the solve
  float scale;             // log2(e) / tau
  double inv_tau_d;
  float tol, alpha;
  int max_iter, k, n_layers;
  int tiles_m, tiles_n;
  int solve_blocks;        // blocks per layer of the solve kernel; 0: the last unit of a layer solves
  int missing_arrivals;    // host-side fault injection, 0 in production: of the solve's barrier, for k d <= 64 of a full stage's
  long long spin_limit;    // SM clock ticks of every wait
  long long row_off[MAX_LAYERS + 1];
  int unit_first[MAX_LAYERS + 1];
  int group_first[MAX_LAYERS];
};

struct JacMmaPlan {
  int nt;                  // columns of a tile: 128 or 256
  int tiles_m, tiles_n, kdp;
};
// false: this codebook has no such pass
bool jac_mma_plan(int d, int k, JacMmaPlan* out);
int jac_mma_units_max(const JacMmaPlan& pl, int n_layers);
int jac_mma_groups_max(int n_layers);
size_t jac_mma_part_bytes(const JacMmaPlan& pl, int d, int k, int n_layers);
int jac_mma_split(const JacMmaPlan& pl, int d, JacMmaParams* p);   // fills the unit table, returns the number of units
cudaError_t launch_jac_mma(int d, const JacMmaPlan& pl, const JacMmaParams& p, int units, cudaStream_t stream);
cudaError_t launch_jac_solve(int d, const JacMmaPlan& pl, const JacMmaParams& p, cudaStream_t stream);

}  // namespace idkm
