// Hard assignment q(w) = argmin_c ||w - c|| (Section 3.1: what the soft quantiser r_tau tends to as tau -> 0): the
// codes and the dequantised weights one ships after training.  One pass over W; the codebook sits in shared memory.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include "idkm_per_device.h"
#include "../../include/idkm.h"

namespace {

constexpr int ASSIGN_BLOCK = 256;
constexpr int ASSIGN_MAX_K = 256;

// Writes the codes and the dequantised weights of one 128-bit group of rows.  (Called by whole warps: shuffles.)
template <int D, int BITS>
__device__ __forceinline__ void assign_store(long long g, long long m, int lane, const int (&bj)[4 / D], const float* cs,
                                             unsigned char* __restrict__ codes, float* __restrict__ Wq) {
  constexpr int VEC = 4 / D, LBITS = VEC * BITS;
  constexpr int NL = LBITS < 8 ? 8 / LBITS : 1;     // lanes that share one byte
  constexpr int NB = LBITS < 8 ? 1 : LBITS / 8;     // bytes a lane (or lane group) writes per trip
  const long long i0 = g * VEC;
  if (codes != nullptr) {
    unsigned int v32 = 0u;
#pragma unroll
    for (int v = 0; v < VEC; ++v)
      if (i0 + v < m) v32 |= (unsigned int)bj[v] << (v * BITS);
    if constexpr (NL > 1) {
      v32 <<= (lane % NL) * LBITS;
#pragma unroll
      for (int o = 1; o < NL; o <<= 1) v32 |= __shfl_xor_sync(0xffffffffu, v32, o);
      if ((lane % NL) == 0 && i0 < m) codes[g / NL] = (unsigned char)v32;
    } else {
      const long long n_bytes = (m * BITS + 7) / 8;
#pragma unroll
      for (int q = 0; q < NB; ++q)
        if (g * NB + q < n_bytes) codes[g * NB + q] = (unsigned char)(v32 >> (8 * q));
    }
  }
  if (Wq != nullptr) {
    if (i0 + VEC <= m) {
      float os[4];
#pragma unroll
      for (int v = 0; v < VEC; ++v)
#pragma unroll
        for (int a = 0; a < D; ++a) os[v * D + a] = cs[bj[v] * D + a];
      reinterpret_cast<float4*>(Wq)[g] = make_float4(os[0], os[1], os[2], os[3]);
    } else {
#pragma unroll
      for (int v = 0; v < VEC; ++v)
        if (i0 + v < m)
#pragma unroll
          for (int a = 0; a < D; ++a) Wq[(i0 + v) * D + a] = cs[bj[v] * D + a];
    }
  }
}

// A lane takes 4 / d consecutive weights per trip -- one 128-bit load, consecutive lanes on consecutive rows -- and
// packs their codes; where that is less than a byte the lanes that share the byte combine by shuffles and the first of
// them writes it, otherwise the lane writes its own bytes.  Every byte is written once, whole.
template <int D, int BITS>
__global__ void __launch_bounds__(ASSIGN_BLOCK) idkm_assign_kernel(const float* __restrict__ W, long long m,
                                                                   const float* __restrict__ C, int k,
                                                                   unsigned char* __restrict__ codes,
                                                                   float* __restrict__ Wq) {
  constexpr int VEC = 4 / D;                        // weights per lane per trip
  __shared__ __align__(16) float cs[ASSIGN_MAX_K * D];
  for (int o = threadIdx.x; o < k * D; o += ASSIGN_BLOCK) cs[o] = C[o];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long groups = (m + VEC - 1) / VEC;             // 128-bit groups of rows
  const long long groups_up = (groups + 31) / 32 * 32;      // whole warps stay in the loop together (shuffles)
  for (long long g = (long long)blockIdx.x * ASSIGN_BLOCK + threadIdx.x; g < groups_up;
       g += (long long)gridDim.x * ASSIGN_BLOCK) {
    const long long i0 = g * VEC;
    float w[VEC][D];
    if (i0 + VEC <= m) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(W) + g);
      const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int v = 0; v < VEC; ++v)
#pragma unroll
        for (int a = 0; a < D; ++a) w[v][a] = xs[v * D + a];
    } else {
#pragma unroll
      for (int v = 0; v < VEC; ++v)
#pragma unroll
        for (int a = 0; a < D; ++a) w[v][a] = (i0 + v < m) ? __ldg(W + (i0 + v) * D + a) : 0.f;
    }
    float bd[VEC];
    int bj[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      bd[v] = 3.0e38f;
      bj[v] = 0;
    }
    for (int j = 0; j < k; ++j) {
      float c[D];
#pragma unroll
      for (int a = 0; a < D; ++a) c[a] = cs[j * D + a];
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        float sq = 0.f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const float df = w[v][a] - c[a];
          sq = fmaf(df, df, sq);
        }
        if (sq < bd[v]) {   // strict: ties keep the lower index
          bd[v] = sq;
          bj[v] = j;
        }
      }
    }
    assign_store<D, BITS>(g, m, lane, bj, cs, codes, Wq);
  }
}

// Larger codebooks.  The distance costs 2 d instructions a pair and keeping the nearest three more; the kernel above is
// bound by issuing them.  Here a pair costs d multiply-adds and one and a bit: the score s_j = |c_j|^2 / 2 - w . c_j orders
// the centroids like the distance up to rounding, and a lane keeps, for each of its four weights, the block of eight centroids
// with the smallest score, and the smallest score of any other block.  Then it settles that block by the distance itself, in
// the arithmetic and with the ties of the kernel above.
// That is the nearest of all k unless another block comes within the rounding of both forms: with u = 2^-24, a score is off
// by at most 6 u (|w| |c| + |c|^2 / 2) and a squared distance, of at most (|w| + |c|)^2, by 8 u of it, together less than
// 20 u (|w| + c_max)^2 <= 40 u (|w|^2 + c_max^2) between two scores; ASSIGN_MARGIN is 64 u (and an absolute term, below which
// numbers are not normal).  Such a weight -- and one with a NaN or an overflow, whose test fails -- is compared with all k
// centroids, by the whole warp.
// What bounds it: the multiply-adds, 8 cycles a pair of a warp at d = 4 (three register operands each, 1.3 cycles).
constexpr float ASSIGN_MARGIN = 64.f * 5.9604645e-8f;
constexpr int ASSIGN_BLK = 8;
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
template <int D>
__device__ __forceinline__ float assign_sq(const float (&w)[D], const float* c) {
  float sq = 0.f;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const float df = w[a] - c[a];
    sq = fmaf(df, df, sq);
  }
  return sq;
}
// The weights of the lanes in `left`, one by one, against all centroids, by the whole warp.
template <int D>
__device__ __forceinline__ void assign_unsure(unsigned left, const float (&w)[D], const float* cs, int k, int lane, int& bj) {
  while (left) {
    const int from = __ffs(left) - 1;
    left &= left - 1;
    float x[D];
#pragma unroll
    for (int a = 0; a < D; ++a) x[a] = __shfl_sync(0xffffffffu, w[a], from);
    unsigned lo = 0xffffffffu;
    int at = 0;
    for (int j = lane; j < k; j += 32) {
      const float sq = assign_sq<D>(x, cs + j * D);
      const unsigned key = sq < 3.0e38f ? __float_as_uint(sq) : 0xffffffffu;   // (squares: ordered like their bits)
      if (key < lo) {
        lo = key;
        at = j;
      }
    }
    const unsigned all = __reduce_min_sync(0xffffffffu, lo);
    const unsigned win = __reduce_min_sync(0xffffffffu, lo == all ? (unsigned)at : 0xffffffffu);
    if (lane == from) bj = all == 0xffffffffu ? 0 : (int)win;
  }
}
template <int D, int BITS>
__global__ void __launch_bounds__(ASSIGN_BLOCK) idkm_assign_score(const float* __restrict__ W, long long m, const float* __restrict__ C,
                                                                  int k, unsigned char* __restrict__ codes, float* __restrict__ Wq) {
  constexpr int VEC = 4 / D, NG = D;   // weights of a 128-bit group, groups of a lane: four weights
  constexpr int KB = ASSIGN_MAX_K / ASSIGN_BLK, BS = ASSIGN_BLK + 1;
  __shared__ __align__(16) float cs[ASSIGN_MAX_K * D];
  __shared__ __align__(16) float half2[ASSIGN_MAX_K];   // |c|^2 / 2
  // the codebook by coordinate, blocks 9 words apart: lanes that read different blocks read different banks
  __shared__ float ct[D][KB * BS];
  __shared__ float s_max;
  const int nblk = (k + ASSIGN_BLK - 1) / ASSIGN_BLK, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = threadIdx.x; j < nblk * ASSIGN_BLK; j += ASSIGN_BLOCK) {
    float q = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const float c = j < k ? C[j * D + a] : 0.f;
      cs[j * D + a] = c;
      ct[a][(j / ASSIGN_BLK) * BS + j % ASSIGN_BLK] = j < k ? c : 2.0e19f;
      q = fmaf(c, c, q);
    }
    half2[j] = j < k ? 0.5f * q : 3.0e38f;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    float q = 0.f;
    bool odd = false;
    for (int j = lane; j < k; j += 32) {
      q = fmaxf(q, half2[j]);
      odd = odd || !(half2[j] < 1e37f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q = fmaxf(q, __shfl_xor_sync(0xffffffffu, q, o));
    odd = __any_sync(0xffffffffu, odd);
    if (lane == 0) s_max = odd ? __int_as_float(0x7fc00000) : 2.f * q;   // (NaN: no weight passes the test)
  }
  __syncthreads();
  const float cmax2 = s_max;
  const long long groups = (m + VEC - 1) / VEC, n_warp = (long long)gridDim.x * (ASSIGN_BLOCK / 32);
  for (long long t = (long long)blockIdx.x * (ASSIGN_BLOCK / 32) + warp; t * (32 * NG) < groups; t += n_warp) {
    const long long g0 = t * (32 * NG) + lane;   // groups g0, g0 + 32, ...
    float w[4][D];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const long long g = g0 + q * 32, i0 = g * VEC;
      float xs[4] = {0.f, 0.f, 0.f, 0.f};
      if (i0 + VEC <= m) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(W) + g);
        xs[0] = x.x; xs[1] = x.y; xs[2] = x.z; xs[3] = x.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (i0 + e / D < m) xs[e] = __ldg(W + i0 * D + e);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) w[q * VEC + e / D][e % D] = xs[e];
    }
    float best[4], second[4], nw[4][D];
    int blk[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      best[v] = second[v] = 3.3e38f;
      blk[v] = 0;
#pragma unroll
      for (int a = 0; a < D; ++a) nw[v][a] = -w[v][a];
    }
#pragma unroll 1
    for (int b = 0; b < nblk; ++b) {
      float c[ASSIGN_BLK * D], h[ASSIGN_BLK];
#pragma unroll
      for (int e = 0; e < ASSIGN_BLK * D; e += 4) {
        const float4 x = *reinterpret_cast<const float4*>(cs + b * (ASSIGN_BLK * D) + e);
        c[e] = x.x; c[e + 1] = x.y; c[e + 2] = x.z; c[e + 3] = x.w;
      }
#pragma unroll
      for (int e = 0; e < ASSIGN_BLK; e += 4) {
        const float4 x = *reinterpret_cast<const float4*>(half2 + b * ASSIGN_BLK + e);
        h[e] = x.x; h[e + 1] = x.y; h[e + 2] = x.z; h[e + 3] = x.w;
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float sc[ASSIGN_BLK];
#pragma unroll
        for (int e = 0; e < ASSIGN_BLK; ++e) {
          sc[e] = h[e];
#pragma unroll
          for (int a = 0; a < D; ++a) sc[e] = fmaf(nw[v][a], c[e * D + a], sc[e]);
        }
        const float lo = min3(min3(sc[0], sc[1], sc[2]), min3(sc[3], sc[4], sc[5]), fminf(sc[6], sc[7]));
        second[v] = fminf(second[v], fmaxf(best[v], lo));
        blk[v] = lo < best[v] ? b : blk[v];
        best[v] = fminf(best[v], lo);
      }
    }
    int bj[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      float w2 = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) w2 = fmaf(w[v][a], w[v][a], w2);
      const bool sure = second[v] - best[v] > fmaf(ASSIGN_MARGIN, w2 + cmax2, 1e-35f) && w2 < 1e37f;
      // the weight's block, by the distance
      float bd = 3.0e38f;
      bj[v] = 0;
#pragma unroll
      for (int e = 0; e < ASSIGN_BLK; ++e) {
        float sq = 0.f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const float df = w[v][a] - ct[a][blk[v] * BS + e];
          sq = fmaf(df, df, sq);
        }
        if (sq < bd) {   // strict: ties keep the lower index (a padding centroid: PAD, never nearer than 3e38)
          bd = sq;
          bj[v] = blk[v] * ASSIGN_BLK + e;
        }
      }
      assign_unsure<D>(__ballot_sync(0xffffffffu, !sure), w[v], cs, k, lane, bj[v]);
    }
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      int o[VEC];
#pragma unroll
      for (int v = 0; v < VEC; ++v) o[v] = bj[q * VEC + v];
      assign_store<D, BITS>(g0 + q * 32, m, lane, o, cs, codes, Wq);
    }
  }
}
// (m = 2.5 M, d = 4: k = 17 31 against 31 us for the kernel above, k = 32 47 against 42, k = 64 81 against 58, k = 256 284 against
// 164; m = 5 M, d = 2: k = 32 55 against 51, k = 256 338 against 219)
constexpr int ASSIGN_SCORE_MIN_K = 32;

// Quadruples of weights, larger codebooks still: the scores on the tensor cores (tcgen05, kind::tf32), a row of the
// accumulator per weight and a column per centroid, so that a thread finds all scores of its weight in its lane of tensor
// memory and only keeps the smallest: one and a bit instructions a pair, and the load.  Each factor is split into two tf32
// terms (hi + lo, rounded; |c|^2 / 2 into three) laid out along k: hi hi, hi lo, lo hi and ones for the constant, 15 of 16
// columns.  What that drops is below 5 u of |w| |c|; the unit's sums are taken to be good to 20 u of
// the terms' magnitudes: with the bounds above less than 66 u (|w|^2 + c_max^2) between two scores, ASSIGN_MMA_MARGIN is 128 u.
// A block is 128 threads with 64 to 256 columns of tensor memory; several share an SM, so that while one waits for its
// products another reads (two at k > 128: a weight and lane then takes 4 cycles a pair and 500 besides, of which the minima are
// two thirds).  Every wait is bounded: if one ran out, the block would compare its weights with all centroids.
constexpr float ASSIGN_MMA_MARGIN = 128.f * 5.9604645e-8f;
constexpr int ASSIGN_MMA_T = 128;
constexpr int ASSIGN_POLLS = 1 << 22;

__device__ __forceinline__ unsigned assign_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// K-major operand without swizzle: core matrices of 8 rows x 16 bytes; ks: bytes between core matrices along k
__device__ __forceinline__ unsigned long long assign_desc(unsigned addr, unsigned ks) {
  return (unsigned long long)((addr >> 4) & 0x3fffu) | ((unsigned long long)(ks >> 4) << 16) | ((unsigned long long)(128u >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ float assign_tf32(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u); }
__device__ __forceinline__ void assign_tmem_ld32(unsigned addr, float (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,"
      "%27,%28,%29,%30,%31}, [%32];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]),
        "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]),
        "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]),
        "=f"(v[30]), "=f"(v[31])
      : "r"(addr)
      : "memory");
}
// the loads issued so far have arrived; v depends on it
__device__ __forceinline__ void assign_tmem_wait(float (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) asm volatile("" : "+f"(v[i]));
}

__global__ void __launch_bounds__(ASSIGN_MMA_T) idkm_assign_mma(const float* __restrict__ W, long long m, const float* __restrict__ C, int k,
                                                                unsigned char* __restrict__ codes, float* __restrict__ Wq, int cols) {
  constexpr int D = 4, K = 4 * D, CH = K / 4;   // columns of the operands, 16-byte chunks of them
  constexpr int KB = ASSIGN_MAX_K / ASSIGN_BLK, BS = ASSIGN_BLK + 1, T = ASSIGN_MMA_T;
  extern __shared__ __align__(128) unsigned char dyn[];
  unsigned char* opB = dyn;                         // [CH][ASSIGN_MAX_K][16]
  unsigned char* opA = dyn + CH * ASSIGN_MAX_K * 16;   // [CH][T][16]
  __shared__ __align__(16) float cs[ASSIGN_MAX_K * D];
  __shared__ float ct[D][KB * BS];   // (see the kernel above)
  __shared__ __align__(8) unsigned long long bar;
  __shared__ unsigned s_tmem;
  __shared__ float s_part[T / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nblk = (k + 31) / 32 * 4;
  float h_max = 0.f;
  for (int j = tid; j < nblk * ASSIGN_BLK; j += T) {
    float c[D], hi[D], lo[D], q = 0.f, v[K];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      c[a] = j < k ? C[j * D + a] : 0.f;
      cs[j * D + a] = c[a];
      ct[a][(j / ASSIGN_BLK) * BS + j % ASSIGN_BLK] = j < k ? c[a] : 2.0e19f;
      q = fmaf(c[a], c[a], q);
      hi[a] = assign_tf32(c[a]);
      lo[a] = assign_tf32(c[a] - hi[a]);
    }
    const float h = j < k ? 0.5f * q : 3.0e38f, h1 = assign_tf32(h), h2 = j < k ? assign_tf32(h - h1) : 0.f;
    h_max = fmaxf(h_max, j < k ? (h < 1e37f ? h : 3.0e38f) : 0.f);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      v[a] = -hi[a];
      v[D + a] = -lo[a];
      v[2 * D + a] = -hi[a];
    }
    v[12] = h1;
    v[13] = h2;
    v[14] = j < k ? assign_tf32((h - h1) - h2) : 0.f;
    v[15] = 0.f;
#pragma unroll
    for (int q4 = 0; q4 < CH; ++q4)
      *reinterpret_cast<float4*>(opB + (q4 * ASSIGN_MAX_K + j) * 16) = make_float4(v[4 * q4], v[4 * q4 + 1], v[4 * q4 + 2], v[4 * q4 + 3]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) h_max = fmaxf(h_max, __shfl_xor_sync(0xffffffffu, h_max, o));
  if (lane == 0) s_part[warp] = h_max;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(assign_smem(&s_tmem)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(assign_smem(&bar)) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *reinterpret_cast<volatile unsigned*>(&s_tmem), mine = tmem + ((unsigned)(warp * 32) << 16);
  h_max = fmaxf(fmaxf(s_part[0], s_part[1]), fmaxf(s_part[2], s_part[3]));
  const float cmax2 = h_max < 1e37f ? 2.f * h_max : __int_as_float(0x7fc00000);   // (NaN: no weight passes the test)
  const unsigned idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(nblk) << 17) | ((unsigned)(T >> 4) << 24);   // tf32 in, fp32 out
  const long long n_tiles = (m + T - 1) / T;
  bool dead = false;   // a wait ran out: nothing more is issued
  unsigned phase = 0;
  float wn[D];
  auto fetch = [&](long long t) {
    const long long row = t * T + tid;
#pragma unroll
    for (int a = 0; a < D; ++a) wn[a] = 0.f;
    if (t < n_tiles && row < m) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(W) + row);
      wn[0] = x.x; wn[1] = x.y; wn[2] = x.z; wn[3] = x.w;
    }
  };
  fetch(blockIdx.x);
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    float w[D], v[K], w2 = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      w[a] = wn[a];
      w2 = fmaf(w[a], w[a], w2);
      const float x = w2 < 1e37f ? w[a] : 0.f;   // (what is not finite stays out of the products)
      v[a] = v[D + a] = assign_tf32(x);
      v[2 * D + a] = assign_tf32(x - v[a]);
    }
    v[12] = v[13] = v[14] = 1.f;
    v[15] = 0.f;
#pragma unroll
    for (int q = 0; q < CH; ++q) *reinterpret_cast<float4*>(opA + (q * T + tid) * 16) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // (the last tile's scores have been read)
    dead = __syncthreads_or(dead ? 1 : 0) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!dead && tid == 0) {
#pragma unroll
      for (int q = 0; q < K / 8; ++q) {
        const unsigned long long da = assign_desc(assign_smem(opA) + q * 2 * (T * 16), T * 16);
        const unsigned long long db = assign_desc(assign_smem(opB) + q * 2 * (ASSIGN_MAX_K * 16), ASSIGN_MAX_K * 16);
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                     "l"(da), "l"(db), "r"(idesc), "r"(q > 0 ? 1u : 0u)
                     : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(assign_smem(&bar)) : "memory");
    }
    __syncwarp();
    fetch(t + gridDim.x);
    if (!dead) {
      unsigned ok = 0;
      for (int i = 0; i < ASSIGN_POLLS && !ok; ++i)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(assign_smem(&bar)), "r"(phase)
                     : "memory");
      phase ^= 1u;
      dead = __any_sync(0xffffffffu, !ok);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    float best = 3.3e38f, second = 3.3e38f;
    int blk = 0;
    if (!dead) {
      float s0[32], s1[32];
      auto scan = [&](const float (&x)[32], int b0) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float lo = min3(min3(x[8 * b], x[8 * b + 1], x[8 * b + 2]), min3(x[8 * b + 3], x[8 * b + 4], x[8 * b + 5]),
                                fminf(x[8 * b + 6], x[8 * b + 7]));
          second = fminf(second, fmaxf(best, lo));
          blk = lo < best ? b0 + b : blk;
          best = fminf(best, lo);
        }
      };
      assign_tmem_ld32(mine, s0);
#pragma unroll 1
      for (int b0 = 0; b0 < nblk; b0 += 8) {   // (the next 32 scores are on their way while 32 are looked at)
        assign_tmem_wait(s0);
        const bool more = b0 + 4 < nblk;
        if (more) assign_tmem_ld32(mine + (unsigned)((b0 + 4) * 8), s1);
        scan(s0, b0);
        if (!more) break;
        assign_tmem_wait(s1);
        if (b0 + 8 < nblk) assign_tmem_ld32(mine + (unsigned)((b0 + 8) * 8), s0);
        scan(s1, b0 + 4);
      }
    }
    const bool sure = !dead && second - best > fmaf(ASSIGN_MMA_MARGIN, w2 + cmax2, 1e-35f) && w2 < 1e37f;
    float bd = 3.0e38f;
    int bj = 0;
#pragma unroll
    for (int e = 0; e < ASSIGN_BLK; ++e) {
      float sq = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float df = w[a] - ct[a][blk * BS + e];
        sq = fmaf(df, df, sq);
      }
      if (sq < bd) {   // strict: ties keep the lower index
        bd = sq;
        bj = blk * ASSIGN_BLK + e;
      }
    }
    const long long row = t * T + tid;
    assign_unsure<D>(__ballot_sync(0xffffffffu, !sure && row < m), w, cs, k, lane, bj);
    if (row < m) {
      if (codes != nullptr) codes[row] = (unsigned char)bj;
      if (Wq != nullptr) reinterpret_cast<float4*>(Wq)[row] = *reinterpret_cast<const float4*>(cs + bj * 4);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}

// Scalar weights, larger codebooks: the codebook is sorted once per block (by counting), a weight finds its place in it by
// bisection.  Rounding keeps the order of the differences and of their squares, so the smallest square is that of one of the
// two neighbours, and the centroids that tie with it follow without gaps: of those the one with the lowest index is taken,
// as the kernel that compares with every centroid does.
template <int BITS>
__global__ void __launch_bounds__(ASSIGN_BLOCK) idkm_assign_search(const float* __restrict__ W, long long m, const float* __restrict__ C,
                                                                   int k, unsigned char* __restrict__ codes, float* __restrict__ Wq) {
  __shared__ __align__(16) float cs[ASSIGN_MAX_K];
  __shared__ float so[ASSIGN_MAX_K];   // sorted, then +inf
  __shared__ short at[ASSIGN_MAX_K];   // and its indices
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  cs[tid] = tid < k ? C[tid] : __int_as_float(0x7f800000);
  __syncthreads();
  const bool real = tid < k && cs[tid] == cs[tid];
  const float mine = real ? cs[tid] : __int_as_float(0x7f800000);   // (a NaN is never the nearest: neither is an infinity)
  int rank = 0;
#pragma unroll 8
  for (int j = 0; j < ASSIGN_MAX_K; ++j) {
    const float c = cs[j], o = c == c ? c : __int_as_float(0x7f800000);
    rank += o < mine || (o == mine && j < tid);
  }
  so[rank] = mine;
  at[rank] = (short)tid;
  __syncthreads();
  const long long groups = (m + 3) / 4, groups_up = (groups + 31) / 32 * 32, n_warp = (long long)gridDim.x * (ASSIGN_BLOCK / 32);
  for (long long t = (long long)blockIdx.x * (ASSIGN_BLOCK / 32) + warp; t * 32 < groups_up; t += n_warp) {
    const long long g = t * 32 + lane, i0 = g * 4;
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    if (i0 + 4 <= m) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(W) + g);
      w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
    } else {
#pragma unroll
      for (int v = 0; v < 4; ++v)
        if (i0 + v < m) w[v] = __ldg(W + i0 + v);
    }
    int pos[4] = {0, 0, 0, 0};   // centroids below the weight, one less than a power of two at most
#pragma unroll
    for (int half = ASSIGN_MAX_K / 2; half > 0; half >>= 1) {
      if (half >= k) continue;
#pragma unroll
      for (int v = 0; v < 4; ++v) pos[v] += so[pos[v] + half - 1] < w[v] ? half : 0;
    }
    int bj[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const float dr = w[v] - so[pos[v]], dl = w[v] - so[pos[v] > 0 ? pos[v] - 1 : 0];
      const float lo = fminf(dr * dr, dl * dl);   // (a square that is NaN loses against any other)
      int best = ASSIGN_MAX_K;
      for (int q = pos[v]; q < ASSIGN_MAX_K; ++q) {
        const float df = w[v] - so[q];
        if (!(df * df == lo)) break;
        best = min(best, (int)at[q]);
      }
      for (int q = pos[v] - 1; q >= 0; --q) {
        const float df = w[v] - so[q];
        if (!(df * df == lo)) break;
        best = min(best, (int)at[q]);
      }
      bj[v] = lo < 3.0e38f ? best : 0;
    }
    assign_store<1, BITS>(g, m, lane, bj, cs, codes, Wq);
  }
}
// (m = 10 M: k = 32 74 against 78 us for the kernel that compares with every centroid, k = 64 131 against 78, k = 256 474 against 90)
constexpr int ASSIGN_SEARCH_MIN_K = 33;
// (m = 2.5 M, d = 4: k = 32 46 against 42 us for the scores on the CUDA cores, k = 64 51 against 58, k = 100 63 against 81, k = 256 106
// against 164; 20 K: 17 against 17.  At d = 2, k = 256, 5 M: 203 against 219, k = 64 81 against 75: not taken)
constexpr int ASSIGN_MMA_MIN_K = 48;


int code_bits(int k) { return k <= 2 ? 1 : (k <= 4 ? 2 : (k <= 16 ? 4 : 8)); }

template <int D, int BITS>
void launch_bits(int grid, int grid_max, cudaStream_t st, const float* W, long long m, const float* C, int k, unsigned char* codes, float* Wq) {
  if constexpr (D == 1 && BITS == 8) {
    if (k >= ASSIGN_SEARCH_MIN_K) {
      idkm_assign_search<BITS><<<grid, ASSIGN_BLOCK, 0, st>>>(W, m, C, k, codes, Wq);
      return;
    }
  }
  if constexpr (D > 1 && BITS == 8) {
    if constexpr (D == 4) {
      if (k >= ASSIGN_MMA_MIN_K) {
        const int cols = k <= 64 ? 64 : (k <= 128 ? 128 : 256), per_sm = cols == 256 ? 2 : 4;
        const int smem = 180 * 1024 / per_sm;   // (no more blocks on an SM than it has tensor memory for)
        static idkm::PerDevice limit;
        const long long tiles = (m + ASSIGN_MMA_T - 1) / ASSIGN_MMA_T;
        const long long most = (long long)(grid_max / 8) * per_sm;
        if (idkm::allow_smem(limit, idkm_assign_mma, 90 * 1024) == cudaSuccess) {   // (otherwise the scores on the CUDA cores)
          idkm_assign_mma<<<(int)(tiles < most ? tiles : most), ASSIGN_MMA_T, smem, st>>>(W, m, C, k, codes, Wq, cols);
          return;
        }
        (void)cudaGetLastError();
      }
    }
    if (k >= ASSIGN_SCORE_MIN_K) {
      idkm_assign_score<D, BITS><<<grid, ASSIGN_BLOCK, 0, st>>>(W, m, C, k, codes, Wq);
      return;
    }
  }
  idkm_assign_kernel<D, BITS><<<grid, ASSIGN_BLOCK, 0, st>>>(W, m, C, k, codes, Wq);
}
template <int D>
cudaError_t launch_assign(int bits, int grid, int grid_max, cudaStream_t st, const float* W, long long m, const float* C, int k,
                          unsigned char* codes, float* Wq) {
  switch (bits) {
    case 1: launch_bits<D, 1>(grid, grid_max, st, W, m, C, k, codes, Wq); break;
    case 2: launch_bits<D, 2>(grid, grid_max, st, W, m, C, k, codes, Wq); break;
    case 4: launch_bits<D, 4>(grid, grid_max, st, W, m, C, k, codes, Wq); break;
    default: launch_bits<D, 8>(grid, grid_max, st, W, m, C, k, codes, Wq); break;
  }
  return cudaGetLastError();
}

}  // namespace

extern "C" int idkm_code_bits(int k) { return (k >= 1 && k <= ASSIGN_MAX_K) ? code_bits(k) : 0; }

extern "C" size_t idkm_codes_bytes(int64_t m, int k) {
  if (m < 1 || k < 1 || k > ASSIGN_MAX_K) return 0;
  return (size_t)((m * code_bits(k) + 7) / 8);
}

extern "C" int idkm_assign(const float* W, int64_t m, int d, const float* C, int k, unsigned char* codes_out,
                           float* Wq_out, void* cuda_stream) {
  if (!W || !C || (!codes_out && !Wq_out)) return IDKM_ERR_NULL;
  if (!(d == 1 || d == 2 || d == 4) || k < 1 || k > ASSIGN_MAX_K) return IDKM_ERR_UNSUPPORTED;
  if (m < 1) return IDKM_ERR_SHAPE;
  if (Wq_out == W) return IDKM_ERR_PARAM;
  if (((uintptr_t)W | (uintptr_t)(Wq_out ? Wq_out : W)) & 15u) return IDKM_ERR_ALIGN;   // vector loads and stores
  const int bits = code_bits(k);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return IDKM_ERR_CUDA;
  const long long groups = ((long long)m * d + 3) / 4;   // one 128-bit group of rows per thread and trip
  long long grid = (groups + ASSIGN_BLOCK - 1) / ASSIGN_BLOCK;
  if (grid > (long long)sms * 8) grid = (long long)sms * 8;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  cudaError_t rc;
  if (d == 1) rc = launch_assign<1>(bits, (int)grid, sms * 8, st, W, m, C, k, codes_out, Wq_out);
  else if (d == 2) rc = launch_assign<2>(bits, (int)grid, sms * 8, st, W, m, C, k, codes_out, Wq_out);
  else rc = launch_assign<4>(bits, (int)grid, sms * 8, st, W, m, C, k, codes_out, Wq_out);
  return rc == cudaSuccess ? IDKM_OK : IDKM_ERR_CUDA;
}
