// Algorithm 1's whole loop over one layer in one cooperative launch for pairs and quadruples of weights and codebooks of more than 16
// centroids (more than 8 at d = 4), in fp32.  The column sums S_j = sum_i A_ij, N_j = sum_i A_ij w_i are taken by warp matrix
// instructions at d = 4 and more than 32 centroids, on the CUDA cores otherwise.  Further description in idkm_mma_loop_impl.cuh.
#pragma once
#include "idkm_kernels.cuh"

namespace idkm {

struct MmaLoopParams {
  SmallLoopParams s;   // partials: [2][grid][PLEN] (one_stage) or [grid][PLEN]
  double* totals;      // [PLEN]
  int one_stage;       // 1: every block adds all partials (one barrier an iteration)
};
typedef cudaError_t (*MmaLoopLaunchFn)(const MmaLoopParams& p, int grid, cudaStream_t stream);
struct MmaLoopEntry {
  MmaLoopLaunchFn launch;
  int kp, plen;
};
constexpr int N_MMA_LOOP = 5;
// [codebook size: 16 (d = 4 only), 32, 64, 128, 256]; _sq: squared distance
extern const MmaLoopEntry k_mma_loop_d2[N_MMA_LOOP], k_mma_loop_d4[N_MMA_LOOP], k_mma_loop_d2_sq[N_MMA_LOOP], k_mma_loop_d4_sq[N_MMA_LOOP];

}  // namespace idkm
