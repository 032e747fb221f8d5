// Scalar weights (d = 1), Euclidean distance: the path that does not visit (weight, centroid) pairs.
//
// With the centroids sorted, v_0 <= ... <= v_{k-1}, a weight w with v_{s-1} < w <= v_s ("interval s", s = 0 .. k, the
// outer two open) has the attention row
//   exp(-(w - v_j)/tau) = exp(-(w - v_{s-1})/tau) exp(-(v_{s-1} - v_j)/tau)   for j <  s,
//   exp(-(v_j - w)/tau) = exp(-(v_s - w)/tau)     exp(-(v_j - v_s)/tau)       for j >= s,
// so A_j(w) = lambda(w) p_j for j < s and mu(w) q_j for j >= s, lambda + mu = 1, with
//   P_i = sum_{j<=i} exp(-(v_i - v_j)/tau),  p_j = exp(-(v_{s-1} - v_j)/tau) / P_{s-1},
//   Q_i = sum_{j>=i} exp(-(v_j - v_i)/tau),  q_j = exp(-(v_j - v_s)/tau) / Q_s,
//   mu / lambda = exp(2 (w - e_s) / tau),    e_s = (v_{s-1} + v_s) / 2 - (tau / 2) ln(Q_s / P_{s-1})
// (Algorithm 1, steps 3-4, exactly).  Everything the method sums over weights is a handful of sums per interval, and what
// a centroid receives from all intervals are first-order linear recurrences over the sorted centroids with the
// coefficients a_j = exp(-(v_{j+1} - v_j)/tau) (Algorithm 1, step 5; Sections 4.1-4.3).
#pragma once
#include "idkm_kernels.cuh"
#include "idkm_scalar_bins.h"

namespace idkm {

constexpr int SC_T = 512;              // threads of a block of the loop kernel (128 registers each)
constexpr int SC_WARPS = SC_T / 32;
constexpr int SC_REC_SMEM = 3584;      // coarse bins whose records fit in shared memory (36 bytes each)
constexpr int SC_REC_BYTES = 36;
constexpr int SC_SYNC_WORDS = 32;      // barrier words of one layer (one 128-byte line)
constexpr int SD_TWO_ROWS_K = 32;      // loop without bins: up to this many centroids two rows of sums for every block
__host__ __device__ constexpr int SD_SUMS(int k) { return 6 * (k + 1); }
constexpr int SC_PSCALE = 65534;       // a weight's place in its fine bin is kept in 1 / 65534 of the bin's width

// Per-layer tables the loop leaves for the passes that follow: doubles, [SC_NTAB][k + 1], sorted order.  V: relative to
// v_0, which entry V[k] holds; A: a_j; RP, RQ: 1 / P_j, 1 / Q_j; L: sums of lambda over interval j + 1, M: of mu over
// interval j, X: of lambda mu over interval j + 1 (0: plain, 1: times w - v_0); S, F: column sum (0 if dead), F - v_0.
enum ScTable { TB_V = 0, TB_A, TB_RP, TB_RQ, TB_L0, TB_L1, TB_M0, TB_M1, TB_X0, TB_X1, TB_S, TB_F, SC_NTAB };
// Per-interval tables of the streaming passes: floats, [SC_NFTAB][k + 1].  V: the sorted centroids; E, O: e_s rounded to
// fp32 and what its rounding adds to the exponent; R, D: average of the centroids to the right, left minus right
// average; U0, U1, U2, U3, U4: coefficients of dL/dW.
enum ScFTable { FT_V = 0, FT_E, FT_O, FT_R, FT_D, FT_U0, FT_U1, FT_U2, FT_U3, FT_U4, SC_NFTAB };

struct ScalarPtrs {            // per-call pointers into the workspace (and the call's tensors)
  const float* W;
  const float* G;
  const float* C0;
  void* Wq;
  float* dW;
  float* dC;                   // [L][k] or null: copy of the adjoint
  float* C;                    // [L][k] working / returned centroids
  float *S, *F, *gvec, *u;     // [L][k]
  LayerState* st;
  float *hist_fwd, *hist_adj;  // [L][HIST_CAP]
  unsigned int* sync;          // [L][SC_SYNC_WORDS]
  unsigned short* grouped;     // [m] places of the weights inside their fine bins, grouped by fine bin (scratch)
  unsigned int* gcount;        // [fine bins]
  unsigned int* fstart;        // [fine bins + L] first element of every fine bin
  long long* frec;             // [fine bins][4] moments
  unsigned char* crec;         // [fine bins + L][SC_REC_BYTES] coarse records of layers with many coarse bins
  float4* bstat;               // [blocks] minimum, maximum, non-finite flag, number of zeros (bits)
  double* tab;                 // [L][SC_NTAB][k + 1]
  int* perm;                   // [L][k] sorted position -> centroid index
  float* ftab;                 // [L][SC_NFTAB][k + 1]
  double* gpart;               // partial sums of the codebook gradient, [blocks + groups][3 (k + 1)], and of the loop without
                               // bins, rows of SD_SUMS(k), [blocks] twice (k <= SD_TWO_ROWS_K) or [blocks + L]
  unsigned int* gtick;         // [groups] arrival counters, zero at rest
  unsigned int* pair_ticks[2]; // arrival counters of the pairwise passes, which may follow: zeroed with the rest
  int n_pair_ticks[2];
};

struct ScalarParams {
  ScalarPtrs p;
  int n_layers, k;
  double inv_tau_d;
  float tol, alpha;
  int max_iter, wq_dtype;
  int n_group_rows;            // rows of gpart after the blocks' own (one per group)
  int missing_arrivals;        // host-side fault injection for the timeout path, 0 in production
  long long spin_limit;
  long long row_off[MAX_LAYERS + 1];
  int blk_first[MAX_LAYERS + 1];   // blocks of each layer
  int fine_off[MAX_LAYERS + 1];    // first fine bin of each layer; capacity = difference
};

// ---- linear recurrences over the sorted centroids --------------------------------------------------------------
// One centroid per thread, the first kw = (k + 31) / 32 warps (all of which must call).  FWD: X_j = x_j + c_j X_{j-1},
// otherwise X_j = x_j + c_j X_{j+1}; threads without a centroid pass c = 0, x = 0.
__device__ __forceinline__ void sc_bar(int warps) { asm volatile("bar.sync 1, %0;" ::"r"(warps * 32) : "memory"); }
__device__ __forceinline__ void sc_sync(int kw) {
  if (kw == 1) __syncwarp();
  else sc_bar(kw);
}
template <int NX, bool FWD>
__device__ __forceinline__ void lin_scan(double c, double (&x)[NX], int k, double* tmp /* [8][4] */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = k < 32 ? k : 32;
  for (int o = 1; o < n; o <<= 1) {
    const bool has = FWD ? (lane >= o) : (lane + o < 32);
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const double y = FWD ? __shfl_up_sync(0xffffffffu, x[i], o) : __shfl_down_sync(0xffffffffu, x[i], o);
      if (has) x[i] = fma(c, y, x[i]);
    }
    const double cc = FWD ? __shfl_up_sync(0xffffffffu, c, o) : __shfl_down_sync(0xffffffffu, c, o);
    if (has) c *= cc;
  }
  const int kw = (k + 31) >> 5;
  if (kw == 1) return;
  sc_bar(kw);   // the previous scan's totals have been read
  if (lane == (FWD ? 31 : 0)) {
    tmp[warp * 4] = c;
#pragma unroll
    for (int i = 0; i < NX; ++i) tmp[warp * 4 + 1 + i] = x[i];
  }
  sc_bar(kw);
#pragma unroll
  for (int i = 0; i < NX; ++i) {
    double carry = 0.0;
    if (FWD) {
      for (int w = 0; w < warp; ++w) carry = fma(tmp[w * 4], carry, tmp[w * 4 + 1 + i]);
    } else {
      for (int w = kw - 1; w > warp; --w) carry = fma(tmp[w * 4], carry, tmp[w * 4 + 1 + i]);
    }
    x[i] = fma(c, carry, x[i]);
  }
}

// Sums over the k threads; result in all threads of the first kw warps.
template <int NX>
__device__ __forceinline__ void sc_reduce(double (&x)[NX], int k, double* tmp /* [8][4], NX <= 4 */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if (o < k || k > 16)   // (lanes from k on hold zeros; every lane gets the sum)
#pragma unroll
      for (int i = 0; i < NX; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], o);
  if (k <= 16) {
    // sums live in groups of the next power of two of k: the first group's value is everybody's
#pragma unroll
    for (int i = 0; i < NX; ++i) x[i] = __shfl_sync(0xffffffffu, x[i], 0);
  }
  const int kw = (k + 31) >> 5;
  if (kw == 1) return;
  sc_bar(kw);
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < NX; ++i) tmp[warp * 4 + i] = x[i];
  sc_bar(kw);
#pragma unroll
  for (int i = 0; i < NX; ++i) {
    double s = 0.0;
    for (int w = 0; w < kw; ++w) s += tmp[w * 4 + i];
    x[i] = s;
  }
}

// lambda and mu from the exponent z = log2(mu / lambda)
__device__ __forceinline__ void sc_lambda(float z, float& lam, float& mu) {
  const float rho = ex2_approx(fminf(fmaxf(z, -126.f), 126.f));
  lam = rcp_approx(1.f + rho);
  mu = rho * lam;
}

// The layer a block works for when blocks are dealt out by blk_first.
__device__ __forceinline__ int sc_layer_of_block(const ScalarParams& sp, int b) {
  int l = 0;
  while (l + 1 < sp.n_layers && b >= sp.blk_first[l + 1]) ++l;
  return l;
}

cudaError_t launch_scalar_init(const ScalarParams& sp, int grid, cudaStream_t stream);
cudaError_t launch_scalar_loop(const ScalarParams& sp, int grid, cudaStream_t stream);
cudaError_t launch_scalar_final(const ScalarParams& sp, int grid, cudaStream_t stream);
cudaError_t launch_scalar_grad(const ScalarParams& sp, int grid, cudaStream_t stream);
cudaError_t launch_scalar_adjoint(const ScalarParams& sp, cudaStream_t stream);
cudaError_t launch_scalar_dw(const ScalarParams& sp, int grid, cudaStream_t stream);
int scalar_grad_threads(int k);   // threads of a block of the gradient pass that take weights

}  // namespace idkm
