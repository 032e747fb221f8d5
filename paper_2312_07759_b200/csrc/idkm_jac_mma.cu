// See idkm_jac_mma.cuh.  One block computes 128 x NT tiles of X^T Y over ranges of weights.
//
// What bounds it: producing the operands.  Nothing of X and Y exists in memory; every tile computes its 128 + NT columns of
// them from the weights, the rows' softmax references and normalisers that the codebook-gradient pass left, and its
// centroids: at d = 4 and NT = 256, 96 (weight, centroid) pairs of ~300 instructions per eight weights and lane, two warps
// to a scheduler (48 % of the issue slots, tensor pipe 34 % active), for 32 768 multiply-adds a weight, which three fp16
// products take 1540 cycles a stage for.  Hence the tile as wide as the register file holds its sums, the packed fp32
// instructions, and, where rows and columns of a tile are of the same centroids (k d <= 128), one pass for both operands.
// Measured (adjoint of 50 steps against the fused passes): 4 M x 4, k = 256: 35 ms against 44; 1 M x 2, k = 256: 2.6
// against 11.2; 3 M x 4, k = 16, 30 steps: 0.31 against 1.9 (1.3 with Jacobian tiles on the CUDA cores).
//
// Precision.  X and Y are split into two fp16 terms (22 bits, scaled by powers of two so that the second term stays
// normal): hi hi + hi lo + lo hi; what is dropped is at most 2^-24 of a product and of either sign.  The tensor core adds in
// fp32 and cuts instead of rounding, so an accumulator takes one stage of 64 weights only -- its small terms first --, what
// the cuts take on average is given back (JM_CUT), and the result is added to fp32 sums in registers, which move to an fp64
// partial every JM_FOLD stages; the partials are added in a fixed order.  Error of the adjoint against float64, with the fused
// passes' in brackets, 40 000 weights, 40 steps: d = 4, k = 16 3.2e-7 (2.9e-7), at tau = 0.002 4e-7 (5e-7); k = 64 3.5e-7 (3.4e-7);
// d = 2, k = 64 3.7e-7 (3.3e-7).  With the first term cut to its leading bits and nothing given back it was 5e-7, and 3e-6 at
// tau = 0.002; two stages to an accumulator were no faster and 2 to 5 times less exact.
//
// Roles: a producing warp makes eight weights' share of the stage (a lane holds a centroid, so nothing crosses lanes) and
// writes it in the core-matrix order of the K-major operand, 16 bytes per lane and row of the operand: consecutive lanes
// are consecutive rows, no bank conflicts.  The diagonal sums Dg, d x d numbers a centroid, are added up on the way (as a
// product of their own they took a third of the time for k d^2 useful of (k d)^2 entries).  The first accumulating warp
// issues the products of a stage and commits them to the stage's barrier, which frees its shared memory and hands its half
// of tensor memory over.  Every wait is bounded; if one runs out the layer's status says so.
#include "idkm_jac_mma.cuh"

#include <string.h>

namespace idkm {

// What an accumulator loses by being cut: four steps of the large products leave a quarter, a half, three quarters and all of an
// entry, each cut by half a unit in the last place on average, 0.36 x 2^-23 of itself: 2.5 x 0.36 x 2^-23 of the entry.
constexpr double JM_CUT = 1.0 + 0.9017 / 8388608.0;
constexpr int JM_DFOLD = 32;           // stages after which the diagonal's fp32 sums move to fp64 (one-tile codebooks)
constexpr int JM_RED = 12;             // blocks whose partials one of them adds up (k d <= 64)

// PACK (k d <= 64): the lanes of a warp hold 16 centroids twice, for two sets of eight weights, so a stage takes twice the
// weights; of the product the two diagonal blocks of lanes count, the others are between different weights.
template <int D, int NT, bool PACK>
struct JmCfg {
  static constexpr int LC = PACK ? 16 : 32;               // centroids of a unit of work per eight weights
  static constexpr int MU = JM_M / D / 32, NU = NT / D / 32;
  static constexpr int CPM = MU * LC, CPN = NU * LC;      // centroids of a tile's rows / columns
  static constexpr int SETS = PACK ? 2 : 1;
  static constexpr int ROWS = JM_ROWS * SETS;             // weights per stage
  static constexpr bool BOTH = NT == JM_M;                // rows and columns are of the same centroids
  static constexpr int A_BYTES = JM_M * JM_ROWS * 2, B_BYTES = NT * JM_ROWS * 2;
  static constexpr int STAGE = 2 * A_BYTES + 2 * B_BYTES;
  static constexpr int SET_FLOATS = (D + 2) * 8 + 4;      // (the two sets' broadcasts fall into different banks)
  static constexpr int OFF_DG = 2 * STAGE, OFF_ROW = OFF_DG + 8 * D * D * MU * 32 * 8;
  static constexpr int DYN = OFF_ROW + 8 * SETS * SET_FLOATS * 4;
  static constexpr int XY = PACK ? 64 * 64 : JM_M * NT;   // doubles of a partial: the product's, then the diagonal sums'
  static constexpr int SLOT = XY + D * D * CPM;
  };
constexpr int JM_LAUNCH_REGS = 65536 / JM_THREADS;   // the two kinds of warps redistribute these: 112 + 144, 160 + 96

__device__ __forceinline__ bool jm_wait(unsigned long long* bar, unsigned parity, long long limit /* SM clock ticks */) {
  bool ok = mbar_try_wait(bar, parity);
  if (!ok) {
    const long long t0 = clock64();
    do ok = mbar_try_wait(bar, parity);
    while (!ok && clock64() - t0 < limit);
  }
  return __all_sync(0xffffffffu, ok);   // (by whole warps, which stay together whatever comes of it)
}
__device__ __forceinline__ void jm_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// K-major operand without swizzle: core matrices of 8 rows x 16 bytes; ks: bytes between core matrices along k, 128
// bytes between them along the rows
__device__ __forceinline__ unsigned long long jm_desc(unsigned addr, unsigned ks) {
  return (unsigned long long)((addr >> 4) & 0x3fffu) | ((unsigned long long)(ks >> 4) << 16) | ((unsigned long long)(128u >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ void jm_mma(unsigned tmem, unsigned long long a, unsigned long long b, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 16 columns of this warp's 32 lanes of tensor memory, added to v
__device__ __forceinline__ void jm_tmem_add16(unsigned addr, float* v) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] += __uint_as_float(r[i]);
}

// The largest |w - F_j| the operands are scaled by, a power of two.
__device__ __forceinline__ float jm_range(float wmax, float fmax_) {
  const float r = fmaxf(wmax + fmax_, 1e-30f);
  return exp2f(ceilf(log2f(r)));
}
__device__ __forceinline__ float jm_layer_range(const JacMmaParams& p, int layer, int d) {
  float fm = 0.f;
  for (int i = threadIdx.x & 31; i < p.k * d; i += 32) fm = fmaxf(fm, fabsf(p.F[(size_t)layer * p.k * d + i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fm = fmaxf(fm, __shfl_xor_sync(0xffffffffu, fm, o));
  return jm_range(__int_as_float(p.st[layer].wmax), fm);
}

// A layer's work is dealt to its blocks as one line of (tile, stage) pairs; a block's share touches two tiles at most.  The
// partial of block b and tile t has slot b + t of the layer: consecutive blocks of a tile lie SLOT doubles apart.
struct JmDeal {
  long long n_st, total, blocks;
  __device__ JmDeal(const JacMmaParams& p, int layer, int rows_per_stage) {
    n_st = (p.row_off[layer + 1] - p.row_off[layer] + rows_per_stage - 1) / rows_per_stage;
    total = n_st * p.tiles_m * p.tiles_n;
    blocks = p.unit_first[layer + 1] - p.unit_first[layer];
  }
  __device__ long long first_of(long long b) const { return total * b / blocks; }
  __device__ long long block_of(long long pos) const { return ((pos + 1) * blocks - 1) / total; }
  __device__ size_t slot0(const JacMmaParams& p, int layer) const { return (size_t)p.unit_first[layer] + (size_t)layer * p.tiles_m * p.tiles_n; }
};

// Stop test of an adjoint step, as in the other forms of the iteration.
struct JmStop {
  int it = 0, up = 0, status, done = 0;
  float res = 0.f, prev = 3.0e38f;
  __device__ void test(const JacMmaParams& p, int layer, double num, double den, double u2_limit, bool writer) {
    res = sqrtf((float)(num / fmax(den, 1e-300)));
    ++it;
    if (writer && it <= HIST_CAP) p.hist_adj[(size_t)layer * HIST_CAP + it - 1] = res;
    up = (res > prev) ? up + 1 : 0;
    prev = res;
    if (!(den <= 1e300) || up >= 10 || den > u2_limit) {
      status = ST_DIVERGED;
      done = 1;
    } else if (p.tol > 0.f && res < p.tol) {
      done = 1;
    } else if (p.tol > 0.f && it >= p.max_iter && status == ST_OK) {
      status = ST_MAXITER;
    }
  }
  __device__ void store(LayerState* st) const {
    st->ticket = 0u;
    st->adj_iters = it;
    st->adj_res = res;
    st->adj_up = up;
    st->adj_prev = prev;
    st->adj_done = 1;
    st->status = status;
  }
};

// Splits eight values (four pairs of neighbouring weights) into two fp16 terms and stores them, 16 bytes each.  The first
// term is the value rounded to its 11 leading bits -- an addition and a mask, on the integer pipe, which the producers leave
// idle, instead of a conversion and back -- so the second is exact before its rounding and of either sign: what the products
// leave out, lo lo, averages out.  (Cut instead of rounded, it is up to 2^-20 of a product and always of its sign.)
__device__ __forceinline__ void jm_split_store(const f2 (&v)[4], unsigned char* hi, unsigned char* lo) {
  unsigned ph[4], pl[4];
  const f2 neg = f2_pack(-1.f, -1.f);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float x, y, lx, ly;
    f2_unpack(v[q], x, y);
    const float hx = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u), hy = __uint_as_float((__float_as_uint(y) + 0x1000u) & 0xffffe000u);
    f2_unpack(f2_fma(f2_pack(hx, hy), neg, v[q]), lx, ly);
    const __half2 h2 = __floats2half2_rn(hx, hy), l2 = __floats2half2_rn(lx, ly);
    ph[q] = *reinterpret_cast<const unsigned*>(&h2);
    pl[q] = *reinterpret_cast<const unsigned*>(&l2);
  }
  *reinterpret_cast<uint4*>(hi) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
  *reinterpret_cast<uint4*>(lo) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
}

// Eight weights of one centroid.  rows: [D + 2][8] -- the coordinates, the softmax references and the normalisers of the
// eight weights; nc, nf: minus the centroid, minus its image F.  The eight weights go through every step together, so that
// the special functions' latency is covered within the warp.
// g: one over the distance; at: the attention
// (The coordinates are loaded before anything is stored: the stores of the operands keep later loads behind them.)
template <int D>
__device__ __forceinline__ void jm_load(const float* rows, f2 (&w)[D][4]) {
  const ulonglong2* r2 = reinterpret_cast<const ulonglong2*>(rows);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const ulonglong2 x = r2[a * 2], y = r2[a * 2 + 1];
    w[a][0] = x.x;
    w[a][1] = x.y;
    w[a][2] = y.x;
    w[a][3] = y.y;
  }
}
template <int D>
__device__ __forceinline__ void jm_attention(const float* rows, const f2 (&w)[D][4], const float (&nc)[D], float scale, f2 (&g)[4], f2 (&at)[4]) {
  const ulonglong2* r2 = reinterpret_cast<const ulonglong2*>(rows);
  const ulonglong2 rf0 = r2[D * 2], rf1 = r2[D * 2 + 1], rn0 = r2[D * 2 + 2], rn1 = r2[D * 2 + 3];
  const f2 rf[4] = {rf0.x, rf0.y, rf1.x, rf1.y}, rn[4] = {rn0.x, rn0.y, rn1.x, rn1.y};
  f2 sq[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) sq[q] = f2_pack(1e-30f, 1e-30f);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const f2 c = f2_pack(nc[a], nc[a]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const f2 d = f2_add(w[a][q], c);
      sq[q] = f2_fma(d, d, sq[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float x, y;
    f2_unpack(sq[q], x, y);
    g[q] = f2_pack(rsqrt_approx(x), rsqrt_approx(y));
  }
  const f2 ms = f2_pack(-scale, -scale);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float x, y;
    f2_unpack(f2_fma(ms, f2_mul(sq[q], g[q]), rf[q]), x, y);
    at[q] = f2_mul(f2_pack(ex2_approx(x), ex2_approx(y)), rn[q]);
  }
}
// a coordinate of the eight weights, less what nx is minus of, times g
__device__ __forceinline__ void jm_entries(const f2 (&w)[4], float nx, const f2 (&g)[4], f2 (&v)[4]) {
  const f2 c = f2_pack(nx, nx);
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = f2_mul(f2_add(w[q], c), g[q]);
}
__device__ __forceinline__ void jm_dot(const f2 (&p)[4], const f2 (&n)[4], float& acc) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float px, py, nx, ny;
    f2_unpack(p[q], px, py);
    f2_unpack(n[q], nx, ny);
    acc = fmaf(py, ny, fmaf(px, nx, acc));
  }
}
// X (rows of the tile); with DIAG also the diagonal sums, which are added to dsum in shared memory
template <int D, bool DIAG>
__device__ __forceinline__ void jm_unit_x(const float* rows, const float (&nc)[D], const float (&nf)[D], float scale, float xm, float ym,
                                          double* dsum, int dstep, unsigned char* hi, unsigned char* lo, int coord_bytes) {
  f2 w[D][4], g[4], at[4];
  jm_load<D>(rows, w);
  jm_attention<D>(rows, w, nc, scale, g, at);
  const f2 m2 = f2_pack(xm, xm), y2 = f2_pack(ym, ym);
#pragma unroll
  for (int q = 0; q < 4; ++q) at[q] = f2_mul(at[q], m2);
  if constexpr (DIAG) {   // (only one tile of a row of tiles does it for a weight)
    float dg[D * D];
#pragma unroll
    for (int e = 0; e < D * D; ++e) dg[e] = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const f2 gq = f2_mul(g[q], y2);
      float nx[D], ny[D];
#pragma unroll
      for (int b = 0; b < D; ++b) f2_unpack(f2_mul(f2_add(w[b][q], f2_pack(nc[b], nc[b])), gq), nx[b], ny[b]);
#pragma unroll
      for (int a = 0; a < D; ++a) {
        float px, py;
        f2_unpack(f2_mul(f2_add(w[a][q], f2_pack(nf[a], nf[a])), at[q]), px, py);
#pragma unroll
        for (int b = 0; b < D; ++b) dg[a * D + b] = fmaf(py, ny[b], fmaf(px, nx[b], dg[a * D + b]));
      }
    }
#pragma unroll
    for (int e = 0; e < D * D; ++e) dsum[e * dstep] += (double)dg[e];
  }
#pragma unroll
  for (int a = 0; a < D; ++a) {
    f2 v[4];
    jm_entries(w[a], nf[a], at, v);
    jm_split_store(v, hi + a * coord_bytes, lo + a * coord_bytes);
  }
}
// Y (columns of the tile)
template <int D>
__device__ __forceinline__ void jm_unit_y(const float* rows, const float (&nc)[D], float scale, float ym, unsigned char* hi, unsigned char* lo,
                                          int coord_bytes) {
  f2 w[D][4], g[4], at[4];
  jm_load<D>(rows, w);
  jm_attention<D>(rows, w, nc, scale, g, at);
  const f2 m2 = f2_pack(ym, ym);
#pragma unroll
  for (int q = 0; q < 4; ++q) at[q] = f2_mul(f2_mul(at[q], m2), g[q]);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    f2 v[4];
    jm_entries(w[a], nc[a], at, v);
    jm_split_store(v, hi + a * coord_bytes, lo + a * coord_bytes);
  }
}
// both, and the diagonal sums, of a tile whose rows and columns are of the same centroids
template <int D>
__device__ __forceinline__ void jm_unit_both(const float* rows, const float (&nc)[D], const float (&nf)[D], float scale, float xm, float ym,
                                             float* dg, unsigned char* xhi, unsigned char* xlo, unsigned char* yhi, unsigned char* ylo,
                                             int coord_bytes) {
  f2 w[D][4], g[4], at[4], n[D][4];
  jm_load<D>(rows, w);
  jm_attention<D>(rows, w, nc, scale, g, at);
  const f2 m2 = f2_pack(xm, xm), y2 = f2_pack(ym, ym);
#pragma unroll
  for (int q = 0; q < 4; ++q) g[q] = f2_mul(g[q], y2);
#pragma unroll
  for (int b = 0; b < D; ++b) {
    f2 v[4];
    jm_entries(w[b], nc[b], g, n[b]);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = f2_mul(n[b][q], at[q]);
    jm_split_store(v, yhi + b * coord_bytes, ylo + b * coord_bytes);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) at[q] = f2_mul(at[q], m2);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    f2 v[4];
    jm_entries(w[a], nf[a], at, v);
    jm_split_store(v, xhi + a * coord_bytes, xlo + a * coord_bytes);
#pragma unroll
    for (int b = 0; b < D; ++b) jm_dot(v, n[b], dg[a * D + b]);
  }
}

template <int D, int NT, bool PACK>
__global__ void __launch_bounds__(JM_THREADS, 1) idkm_jac_mma(const __grid_constant__ JacMmaParams p) {
  using Cfg = JmCfg<D, NT, PACK>;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ __align__(8) unsigned long long full[2], done[2], tfree[2];
  __shared__ unsigned s_tmem;
  __shared__ int s_fail, s_flag;
  grid_dependency_sync();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int layer = 0;
  while (layer + 1 < p.n_layers && (int)blockIdx.x >= p.unit_first[layer + 1]) ++layer;
  LayerState* st = p.st + layer;
  if (p.solve_blocks > 0 && (int)blockIdx.x == p.unit_first[layer] && tid < JM_SYNC_WORDS) p.sync[layer * JM_SYNC_WORDS + tid] = 0u;
  if (st->adj_done) return;
  // ---- this block's share: stages lo .. lo + n - 1 of the layer's line, the first nb of them in tile t0 ----
  const JmDeal dl(p, layer, Cfg::ROWS);
  const int bl = (int)blockIdx.x - p.unit_first[layer];
  const long long lo = dl.first_of(bl);
  const int n = (int)(dl.first_of(bl + 1) - lo), t0 = (int)(lo / dl.n_st), st0 = (int)(lo - t0 * dl.n_st);
  const int nb = (int)(dl.n_st - st0 < n ? dl.n_st - st0 : n);
  double* part = p.part + (dl.slot0(p, layer) + bl + t0) * Cfg::SLOT;   // (the second tile's follows)
  const long long rows = p.row_off[layer + 1] - p.row_off[layer];
  const int k = p.k;
  const float range = jm_layer_range(p, layer, D);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(reinterpret_cast<unsigned long long*>(&s_tmem))),
                 "r"(2 * NT)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        mbar_init(&full[i], 8u + (PACK ? (unsigned)p.missing_arrivals : 0u));
        mbar_init(&done[i], 1);
        mbar_init(&tfree[i], 8);
      }
      mbar_init_fence();
      s_fail = 0;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *reinterpret_cast<volatile unsigned*>(&s_tmem);

  if (warp < 8) {
    // ================= accumulating warps: a quarter of the rows, half of the columns each =================
    if constexpr (NT == 128)
      asm volatile("setmaxnreg.dec.sync.aligned.u32 112;");
    else
      asm volatile("setmaxnreg.inc.sync.aligned.u32 160;");
    float acc[NT / 2];
#pragma unroll
    for (int i = 0; i < NT / 2; ++i) acc[i] = 0.f;
    const int half = warp >> 2, quad = warp & 3;
    const unsigned base = tmem + ((unsigned)(quad * 32) << 16) + (unsigned)(half * (NT / 2));
    // a quarter of what stage i left in tensor memory, added to the registers
    auto take = [&](int i, int part4) {
      const int s = i & 1;
      if (part4 == 0) {
        if (!jm_wait(&done[s], (unsigned)((i >> 1) & 1), p.spin_limit)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
#pragma unroll
      for (int q = 0; q < NT / 8; q += 16)
        jm_tmem_add16(base + (unsigned)(s * NT + part4 * (NT / 8) + q), acc + part4 * (NT / 8) + q);
      if (part4 == 3) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) jm_arrive(&tfree[s]);
      }
      return true;
    };
    // after stage i: the sums move on at the end of a run of stages
    auto fold = [&](int i) {
      const int at = i < nb ? i : i - nb, last = i < nb ? nb : n - nb;   // place within the tile's share, its length
      if ((at + 1) % JM_FOLD == 0 || at + 1 == last) {
        double* o = part + (i < nb ? 0 : Cfg::SLOT);
        const bool first = at < JM_FOLD;
        if constexpr (PACK) {   // the two sets' blocks of lanes: this lane's, and the one 16 lanes and 16 columns further
#pragma unroll
          for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int l = 0; l < 16; ++l) {
              const double v = JM_CUT * ((double)acc[b * 32 + l] + (double)__shfl_xor_sync(0xffffffffu, acc[b * 32 + 16 + l], 16));
              double* e = o + ((half * 2 + b) * 16 + l) * 64 + quad * 16 + lane;
              if (lane < 16) *e = first ? v : *e + v;
            }
#pragma unroll
          for (int q = 0; q < NT / 2; ++q) acc[q] = 0.f;
        } else {
#pragma unroll
          for (int q = 0; q < NT / 2; ++q) {
            double* e = o + (size_t)q * 256 + half * 128 + quad * 32 + lane;
            *e = first ? JM_CUT * (double)acc[q] : fma(JM_CUT, (double)acc[q], *e);
            acc[q] = 0.f;
          }
        }
      }};
    bool ok = true;
    if (warp != 0) {
      for (int i = 0; i < n && ok; ++i) {
#pragma unroll
        for (int c = 0; c < 4; ++c) ok = ok && take(i, c);
        if (ok) fold(i);
      }
    } else {
      // This warp also issues the products -- lo hi, hi lo, then hi hi --, three at a time: the tensor core's queue is
      // short, and what the warp has to take of the stage before fits in between.
      const unsigned idesc = (1u << 4) | ((unsigned)(NT >> 3) << 17) | ((unsigned)(JM_M >> 4) << 24);   // fp16 in, fp32 out
      const unsigned sbase = (unsigned)__cvta_generic_to_shared(dyn);
      int issued = 0;
      for (int i = 0; i < n && ok; ++i) {
        const int s = i & 1;
        ok = jm_wait(&full[s], (unsigned)((i >> 1) & 1), p.spin_limit);
        if (ok && i >= 2) ok = jm_wait(&tfree[s], (unsigned)(((i >> 1) - 1) & 1), p.spin_limit);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned a0 = sbase + s * Cfg::STAGE, b0 = a0 + 2 * Cfg::A_BYTES, dst = tmem + (unsigned)(s * NT);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (lane == 0) {
#pragma unroll
            for (int x = c * 3; x < c * 3 + 3; ++x) {
              const int t = x / (JM_ROWS / 16), q = x % (JM_ROWS / 16);
              const unsigned long long da = jm_desc(a0 + (t == 0 ? Cfg::A_BYTES : 0) + q * 2 * (JM_M * 16), JM_M * 16);
              const unsigned long long db = jm_desc(b0 + (t == 1 ? Cfg::B_BYTES : 0) + q * 2 * (NT * 16), NT * 16);
              jm_mma(dst, da, db, idesc, x == 0 ? 0u : 1u);
            }
            if (c == 3)
              asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&done[s])) : "memory");
          }
          __syncwarp();
          issued = i + 1;
          if (i > 0) ok = ok && take(i - 1, c);
        }
        if (ok && i > 0) fold(i - 1);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) ok = ok && take(n - 1, c);
      if (ok) fold(n - 1);
      // (what is in flight ends before tensor memory is given back)
      if (!ok && issued > 0) (void)jm_wait(&done[(issued - 1) & 1], (unsigned)(((issued - 1) >> 1) & 1), p.spin_limit);
    }
    if (!ok && lane == 0) s_fail = 1;
  } else {
    // ================= producing warps: eight weights of every stage (twice eight: PACK) =================
    if constexpr (NT == 128)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
    else
      asm volatile("setmaxnreg.dec.sync.aligned.u32 96;");
    const int pw = warp - 8, cl = PACK ? lane & 15 : lane, set = PACK ? lane >> 4 : 0;
    float cx[Cfg::MU][D], fx[Cfg::MU][D], cy[Cfg::BOTH ? 1 : Cfg::NU][D], dg[Cfg::BOTH ? Cfg::MU : 1][D * D];
    double* dsum = reinterpret_cast<double*>(dyn + Cfg::OFF_DG);   // [8 warps][D * D][MU][32]
    double* dmine = dsum + pw * (D * D * Cfg::MU * 32);
    int mt = 0, nt = 0;
    auto load_tile = [&](int t) {
      mt = t / p.tiles_n;
      nt = t % p.tiles_n;
#pragma unroll
      for (int h = 0; h < Cfg::MU; ++h) {
        const int j = mt * Cfg::CPM + h * Cfg::LC + cl;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          cx[h][a] = -(j < k ? p.C[((size_t)layer * k + j) * D + a] : PAD_COORD);
          fx[h][a] = -(j < k ? p.F[((size_t)layer * k + j) * D + a] : 0.f);
        }
        if constexpr (Cfg::BOTH) {
#pragma unroll
          for (int e = 0; e < D * D; ++e) dg[h][e] = 0.f;
        } else {
#pragma unroll
          for (int e = 0; e < D * D; ++e) dmine[(e * Cfg::MU + h) * 32 + lane] = 0.0;
        }
      }
      if constexpr (!Cfg::BOTH) {
#pragma unroll
        for (int h = 0; h < Cfg::NU; ++h) {
          const int j = nt * Cfg::CPN + h * 32 + lane;
#pragma unroll
          for (int a = 0; a < D; ++a) cy[h][a] = -(j < k ? p.C[((size_t)layer * k + j) * D + a] : PAD_COORD);
        }
      }
    };
    load_tile(t0);
    float* rowsm = reinterpret_cast<float*>(dyn + Cfg::OFF_ROW) + pw * Cfg::SETS * Cfg::SET_FLOATS;   // [D + 2][8] per set
    const float* myrows = rowsm + set * Cfg::SET_FLOATS;
    const long long row0 = p.row_off[layer];
    float4 wn = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 rn = make_float2(0.f, 0.f);
    auto fetch = [&](int i) {
      const int stage = i < nb ? st0 + i : i - nb;
      const long long loc = (long long)stage * Cfg::ROWS + pw * (8 * Cfg::SETS) + lane;
      if (lane < 8 * Cfg::SETS && i < n) {
        const bool ok = loc < rows;
        const long long g = row0 + (ok ? loc : 0);
        if constexpr (D == 4) {
          wn = __ldg(reinterpret_cast<const float4*>(p.W) + g);
        } else {
          const float2 x = __ldg(reinterpret_cast<const float2*>(p.W) + g);
          wn = make_float4(x.x, x.y, 0.f, 0.f);
        }
        rn = __ldg(p.rowstat + g);
        if (!ok) rn.y = 0.f;   // a zero normaliser switches the weight off
      }
    };
    fetch(0);
    const float xm = 16384.f / range, ym = 16384.f;
    bool ok = true;
    for (int i = 0; i < n; ++i) {
      const int s = i & 1;
      if (i == nb) load_tile(t0 + 1);
      // (a warp whose wait ran out makes nothing more, but meets the others at the ends of the tiles)
      if (i >= 2 && ok) ok = jm_wait(&done[s], (unsigned)(((i >> 1) - 1) & 1), p.spin_limit);
      const int at = i < nb ? i : i - nb, last = i < nb ? nb : n - nb;
      if (ok) {
        __syncwarp();
        if (lane < 8 * Cfg::SETS) {
          float* o = rowsm + (lane >> 3) * Cfg::SET_FLOATS + (lane & 7);
          o[0] = wn.x;
          o[8] = wn.y;
          if constexpr (D == 4) {
            o[16] = wn.z;
            o[24] = wn.w;
          }
          o[D * 8] = rn.x;
          o[D * 8 + 8] = rn.y;
        }
        __syncwarp();
        fetch(i + 1);
        unsigned char* A = dyn + s * Cfg::STAGE + pw * (JM_M * 16) + lane * 16;
        unsigned char* B = dyn + s * Cfg::STAGE + 2 * Cfg::A_BYTES + pw * (NT * 16) + lane * 16;
        if constexpr (Cfg::BOTH) {
#pragma unroll
          for (int h = 0; h < Cfg::MU; ++h)
            jm_unit_both<D>(myrows, cx[h], fx[h], p.scale, xm, ym, dg[h], A + h * 512, A + Cfg::A_BYTES + h * 512, B + h * 512,
                            B + Cfg::B_BYTES + h * 512, JM_M / D * 16);
        } else {
          // of the tiles that share these rows of X, one adds this stage to the diagonal sums
          const bool diag = (i < nb ? st0 + i : i - nb) % p.tiles_n == nt;
#pragma unroll
          for (int h = 0; h < Cfg::MU; ++h) {
            unsigned char* o = A + h * 512;
            if (diag)
              jm_unit_x<D, true>(myrows, cx[h], fx[h], p.scale, xm, ym, dmine + h * 32 + lane, Cfg::MU * 32, o, o + Cfg::A_BYTES, JM_M / D * 16);
            else
              jm_unit_x<D, false>(myrows, cx[h], fx[h], p.scale, xm, ym, dmine + h * 32 + lane, Cfg::MU * 32, o, o + Cfg::A_BYTES, JM_M / D * 16);
          }
#pragma unroll
          for (int h = 0; h < Cfg::NU; ++h)
            jm_unit_y<D>(myrows, cy[h], p.scale, ym, B + h * 512, B + Cfg::B_BYTES + h * 512, NT / D * 16);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) jm_arrive(&full[s]);
      }
      if (Cfg::BOTH && ((at + 1) % JM_DFOLD == 0 || at + 1 == last)) {
#pragma unroll
        for (int h = 0; h < (Cfg::BOTH ? Cfg::MU : 0); ++h)
#pragma unroll
          for (int e = 0; e < D * D; ++e) {
            double* o = dmine + (e * Cfg::MU + h) * 32 + lane;
            double v = (double)dg[h][e];
            if constexpr (PACK) v += (double)__shfl_xor_sync(0xffffffffu, dg[h][e], 16);
            *o = at < JM_DFOLD ? v : *o + v;
            dg[h][e] = 0.f;
          }
      }
      if (at + 1 == last) {   // (every producing warp comes here for the same stage)
        asm volatile("bar.sync 1, 256;" ::: "memory");
        double* o = part + (i < nb ? 0 : Cfg::SLOT) + Cfg::XY;
        for (int x = tid - 256; x < D * D * Cfg::CPM; x += 256) {
          const int e = x / Cfg::CPM, c = x % Cfg::CPM;
          double v = 0.0;
#pragma unroll
          for (int w = 0; w < 8; ++w) v += dsum[w * (D * D * Cfg::MU * 32) + (e * Cfg::MU + c / Cfg::LC) * 32 + c % Cfg::LC];
          o[x] = v;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
      }
    }
    if (!ok && lane == 0) s_fail = 1;
  }
  __threadfence();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * NT));
  const bool failed = *reinterpret_cast<volatile int*>(&s_fail) != 0;
  if (failed && tid == 0) {
    st->status = ST_TIMEOUT;
    __threadfence();   // (before this block announces itself: the last block of the layer reads the status)
  }
  if constexpr (PACK) {
    // ================= k d <= 64: the blocks' partials are added in two stages, and the last block runs the iteration ======
    const int units = p.unit_first[layer + 1] - p.unit_first[layer], ng = (units + JM_RED - 1) / JM_RED, grp = bl / JM_RED;
    const int in_group = grp + 1 < ng ? JM_RED : units - grp * JM_RED;
    if (tid == 0) s_flag = atomicAdd(&p.gtickets[p.group_first[layer] + grp], 1u) == (unsigned)(in_group - 1);
    __syncthreads();
    if (!s_flag) return;
    __threadfence();
    double* sum = p.part + (dl.slot0(p, layer) + (size_t)grp * JM_RED) * Cfg::SLOT;
    for (int o = tid; o < Cfg::SLOT; o += JM_THREADS) {
      double s = 0.0;
#pragma unroll
      for (int t = 0; t < JM_RED; ++t)
        if (t < in_group) s += __ldcg(sum + (size_t)t * Cfg::SLOT + o);
      __stcg(sum + o, s);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      p.gtickets[p.group_first[layer] + grp] = 0u;
      s_flag = atomicAdd(&st->ticket, 1u) == (unsigned)(ng - 1);
    }
    __syncthreads();
    if (!s_flag) return;
    __threadfence();
    const int nd = k * D;
    double* J = reinterpret_cast<double*>(dyn);   // [64][65]: J_C^T
    double* ub = J + 64 * 65;                     // [2][4][18]: a quarter per thread of an output, in banks of its own
    double* red = ub + 2 * 72;                    // [2][8][2]
    const double* all = p.part + dl.slot0(p, layer) * Cfg::SLOT;
    for (int o = tid; o < 64 * 64; o += JM_THREADS) {
      const int r = o & 63, q = o >> 6;           // places of the input coordinate (j, a) and the output coordinate (l, b)
      const int j = r % Cfg::CPM, a = r / Cfg::CPM, l = q % Cfg::CPM, b = q / Cfg::CPM;
      double s = 0.0;
#pragma unroll
      for (int t = 0; t < JM_RED + 1; ++t)
        if (t < ng) s -= __ldcg(all + (size_t)t * JM_RED * Cfg::SLOT + o);
      if (j == l)
        for (int t = 0; t < ng; ++t) s += __ldcg(all + (size_t)t * JM_RED * Cfg::SLOT + Cfg::XY + (a * D + b) * Cfg::CPM + j);
      const float S = j < k ? p.S[(size_t)layer * k + j] : 0.f;
      s *= (S >= S_MIN_F) ? p.inv_tau_d / (double)S * ((double)range / 268435456.0) : 0.0;
      J[q * 65 + r] = l < k ? s : 0.0;
    }
    if (tid < 64) {
      const int l = tid % Cfg::CPM, b = tid / Cfg::CPM;
      ub[(tid >> 4) * 18 + (tid & 15)] = l < k ? (double)p.gvec[(size_t)layer * nd + l * D + b] : 0.0;
    }
    __syncthreads();
    if (warp >= 8) return;
    const int q = tid >> 2, pr = tid & 3;         // four threads per output, each with its part of the row in registers
    const double al = (double)p.alpha, be = 1.0 - al;
    JmStop stop;
    stop.status = *reinterpret_cast<volatile int*>(&st->status);
    const int place = (q >> 4) * 18 + (q & 15);
    const double gq = ub[place];
    double row[16], uo = gq, g2 = 0.0;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      row[r] = J[q * 65 + pr * 16 + r];
      const double x = ub[pr * 18 + r];
      g2 = fma(x, x, g2);
    }
    g2 += __shfl_xor_sync(0xffffffffu, g2, 1);
    g2 += __shfl_xor_sync(0xffffffffu, g2, 2);
    const double u2_limit = ADJ_GROWTH_LIMIT * ADJ_GROWTH_LIMIT * g2;
    if (failed || stop.status == ST_TIMEOUT) stop.done = 1;
    while (stop.it < p.max_iter && !stop.done) {
      const double* u = ub + (stop.it & 1) * 72 + pr * 18;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll
      for (int r = 0; r < 16; r += 4) {
        s0 = fma(row[r], u[r], s0);
        s1 = fma(row[r + 1], u[r + 1], s1);
        s2 = fma(row[r + 2], u[r + 2], s2);
        s3 = fma(row[r + 3], u[r + 3], s3);
      }
      double s = (s0 + s1) + (s2 + s3);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      const double un = al * (s + gq) + be * uo;
      if (pr == 0) ub[((stop.it + 1) & 1) * 72 + place] = un;
      double num = (un - uo) * (un - uo), den = un * un;
      uo = un;
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
      }
      double* rd = red + (stop.it & 1) * 16;
      if (lane == 0) {
        rd[warp * 2] = num;
        rd[warp * 2 + 1] = den;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      num = ((rd[0] + rd[2]) + (rd[4] + rd[6])) + ((rd[8] + rd[10]) + (rd[12] + rd[14]));
      den = ((rd[1] + rd[3]) + (rd[5] + rd[7])) + ((rd[9] + rd[11]) + (rd[13] + rd[15]));
      stop.test(p, layer, num, den, u2_limit, tid == 0);
    }
    const int l = q % Cfg::CPM, b = q / Cfg::CPM;
    if (pr == 0 && l < k) p.u[(size_t)layer * nd + l * D + b] = (float)uo;
    if (tid == 0) stop.store(st);
  }
}

// ---- larger codebooks: the iteration by many blocks, eight rows of J_C^T each, kept in shared memory ----
// Blocks of a layer meet at a bounded barrier once per step; the adjoint and the squares of the stop test cross L2.
constexpr int JS_T = 256, JS_ROWS = 8;
template <int D, int NT>
__global__ void __launch_bounds__(JS_T) idkm_jac_solve(const __grid_constant__ JacMmaParams p) {
  using Cfg = JmCfg<D, NT, false>;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ double red[JS_ROWS][2], tot[2];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NB = p.solve_blocks, layer = blockIdx.x / NB, b = blockIdx.x % NB;
  const int kdp = p.tiles_m * JM_M, k = p.k, nd = k * D;
  double* J = reinterpret_cast<double*>(dyn);          // [JS_ROWS][kdp]
  double* u = J + (size_t)JS_ROWS * kdp;               // [kdp], permuted: (M tile, coordinate, centroid of the tile)
  LayerState* st = p.st + layer;
  if (st->adj_done) return;
  const float range = jm_layer_range(p, layer, D);
  const double f0 = p.inv_tau_d * ((double)range / 268435456.0);
  // this warp's output coordinate (l, c) and its place in the permuted order
  const int q = b * JS_ROWS + warp, l = q / D, c = q % D;
  const bool own = q < nd;
  const int place = (l / Cfg::CPM) * JM_M + c * Cfg::CPM + l % Cfg::CPM;
  const JmDeal dl(p, layer, Cfg::ROWS);
  const size_t slot0 = dl.slot0(p, layer);
  const int nt = l / Cfg::CPN, col = c * Cfg::CPN + l % Cfg::CPN;
  const size_t entry = (size_t)(col % (NT / 2)) * 256 + (size_t)(col / (NT / 2)) * 128;
  for (int mt = 0; mt < p.tiles_m; ++mt) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (own) {
      const int t = mt * p.tiles_n + nt;
      const int b0 = (int)dl.block_of(t * dl.n_st), nb = (int)dl.block_of((t + 1) * dl.n_st - 1) - b0 + 1;
      const double* src = p.part + (slot0 + b0 + t) * Cfg::SLOT + entry + lane;
#pragma unroll 8
      for (int x = 0; x < nb; ++x)
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r] -= __ldcg(src + (size_t)x * Cfg::SLOT + 32 * r);
    }
    if (own && l / Cfg::CPM == mt)
      for (int t = mt * p.tiles_n; t < (mt + 1) * p.tiles_n; ++t) {
        const int b0 = (int)dl.block_of(t * dl.n_st), nb = (int)dl.block_of((t + 1) * dl.n_st - 1) - b0 + 1;
        const double* src = p.part + (slot0 + b0 + t) * Cfg::SLOT + Cfg::XY + c * Cfg::CPM + l % Cfg::CPM;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          double v = 0.0;
          for (int x = lane; x < nb; x += 32) v += __ldcg(src + (size_t)x * Cfg::SLOT + a * D * Cfg::CPM);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          const int mrow = a * Cfg::CPM + l % Cfg::CPM;
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (lane + 32 * r == mrow) s[r] += v;
        }
      }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int mrow = lane + 32 * r, j = mt * Cfg::CPM + mrow % Cfg::CPM;
      const float S = j < k ? p.S[(size_t)layer * k + j] : 0.f;
      J[(size_t)warp * kdp + mt * JM_M + mrow] = (S >= S_MIN_F) ? s[r] * (f0 / (double)S) : 0.0;
    }
  }
  const double g = own ? (double)p.gvec[(size_t)layer * nd + q] : 0.0;
  for (int i = tid; i < kdp; i += JS_T) {
    const int mt = i / JM_M, mrow = i % JM_M, j = mt * Cfg::CPM + mrow % Cfg::CPM, a = mrow / Cfg::CPM;
    u[i] = j < k ? (double)p.gvec[((size_t)layer * k + j) * D + a] : 0.0;
  }
  __syncthreads();
  double g2 = 0.0;
  for (int i = lane; i < kdp; i += 32) g2 += u[i] * u[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) g2 += __shfl_xor_sync(0xffffffffu, g2, o);
  const double u2_limit = ADJ_GROWTH_LIMIT * ADJ_GROWTH_LIMIT * g2;
  const double al = (double)p.alpha, be = 1.0 - al;
  JmStop stop;
  stop.status = st->status;
  if (stop.status == ST_TIMEOUT) return;
  unsigned int* sync = p.sync + layer * JM_SYNC_WORDS;
  bool ok = true;
  while (stop.it < p.max_iter && !stop.done) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    const double* row = J + (size_t)warp * kdp;
    for (int i = lane; i < kdp; i += 128) {   // (kdp is a multiple of 128)
      s0 = fma(row[i], u[i], s0);
      s1 = fma(row[i + 32], u[i + 32], s1);
      s2 = fma(row[i + 64], u[i + 64], s2);
      s3 = fma(row[i + 96], u[i + 96], s3);
    }
    double s = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int par = (stop.it + 1) & 1;
    double* out = p.ub + ((size_t)par * p.n_layers + layer) * kdp;
    if (lane == 0) {
      const double uo = own ? u[place] : 0.0, un = own ? al * (s + g) + be * uo : 0.0;
      if (own) __stcg(out + place, un);
      red[warp][0] = (un - uo) * (un - uo);
      red[warp][1] = un * un;
    }
    __syncthreads();
    double* pn = p.pn + ((size_t)par * p.n_layers + layer) * NB * 2;
    if (tid < 2) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < JS_ROWS; ++w) t += red[w][tid];
      __stcg(pn + b * 2 + tid, t);
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
      volatile unsigned int* vs = sync;
      int good = 1;
      __threadfence();
      atomicAdd(&sync[0], 1u);
      const unsigned target = (unsigned)(stop.it + 1) * (unsigned)(NB + p.missing_arrivals);
      const long long t0 = clock64();
      while ((int)(vs[0] - target) < 0) {
        if (vs[1] != 0u || clock64() - t0 > p.spin_limit) {
          atomicExch(&sync[1], 1u);
          good = 0;
          break;
        }
      }
      if (vs[1] != 0u) good = 0;
      __threadfence();
      s_ok = good;
    }
    __syncthreads();
    ok = s_ok != 0;
    if (!ok) break;
    for (int i = tid; i < kdp; i += JS_T) {
      const int mt = i / JM_M, j = mt * Cfg::CPM + (i % JM_M) % Cfg::CPM;
      if (j < k) u[i] = __ldcg(out + i);
    }
    if (warp == 0) {
      double num = 0.0, den = 0.0;
      for (int i = lane; i < NB; i += 32) {
        num += __ldcg(pn + i * 2);
        den += __ldcg(pn + i * 2 + 1);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
      }
      if (lane == 0) {
        tot[0] = num;
        tot[1] = den;
      }
    }
    __syncthreads();
    stop.test(p, layer, tot[0], tot[1], u2_limit, b == 0 && tid == 0);
  }
  if (lane == 0 && own) p.u[(size_t)layer * nd + q] = (float)u[place];
  if (b == 0 && tid == 0) {
    if (!ok) {
      stop.status = ST_TIMEOUT;
    }
    stop.store(st);
  }
}

bool jac_mma_plan(int d, int k, JacMmaPlan* out) {
  if ((d != 2 && d != 4) || k <= 8 || k > 256) return false;
  const int cpm = JM_M / d;
  out->tiles_m = (k + cpm - 1) / cpm;
  if (out->tiles_m == 3) out->tiles_m = 4;   // (column tiles are pairs of row tiles)
  if (out->tiles_m > 4 && (out->tiles_m & 1)) ++out->tiles_m;
  out->nt = out->tiles_m == 1 ? 128 : 256;
  out->tiles_n = out->tiles_m == 1 ? 1 : out->tiles_m / 2;
  out->kdp = out->tiles_m * JM_M;
  return true;
}

static int plan_rows(int d, int k) { return k * d <= 64 ? 2 * JM_ROWS : JM_ROWS; }
int jac_mma_units_max(const JacMmaPlan& pl, int n_layers) { return JM_UNITS + n_layers * pl.tiles_m * pl.tiles_n; }
size_t jac_mma_part_bytes(const JacMmaPlan& pl, int d, int k, int n_layers) {
  const size_t tiles = (size_t)pl.tiles_m * pl.tiles_n;
  const size_t slot = k * d <= 64 ? 64 * 64 + (size_t)d * 64 : (size_t)JM_M * pl.nt + (size_t)d * JM_M;
  return ((size_t)jac_mma_units_max(pl, n_layers) + n_layers * tiles) * slot * sizeof(double);
}

// A layer gets its share of the blocks, at least one per tile (a block's share of the work then touches two tiles at most)
// and no more than it has stages.
int jac_mma_split(const JacMmaPlan& pl, int d, JacMmaParams* p) {
  const int L = p->n_layers, tiles = pl.tiles_m * pl.tiles_n, per = plan_rows(d, p->k);
  const long long m = p->row_off[L];
  int units = 0, groups = 0;
  for (int l = 0; l < L; ++l) {
    const long long rows = p->row_off[l + 1] - p->row_off[l], work = (rows + per - 1) / per * tiles;
    long long n = (long long)JM_UNITS * rows / m;
    if (n < tiles) n = tiles;
    if (n > work) n = work;
    p->unit_first[l] = units;
    p->group_first[l] = groups;
    units += (int)n;
    groups += (int)((n + JM_RED - 1) / JM_RED);
  }
  for (int l = L; l <= MAX_LAYERS; ++l) p->unit_first[l] = units;
  return units;
}
int jac_mma_groups_max(int n_layers) { return (JM_UNITS + n_layers) / JM_RED + n_layers; }   // k d <= 64

template <int D, int NT, bool PACK>
static cudaError_t launch_mma(const JacMmaParams& p, int units, cudaStream_t stream) {
  constexpr int DYN = JmCfg<D, NT, PACK>::DYN;
  static PerDevice shares, limit;
  // (the warps' shares of the registers have to add up)
  cudaError_t rc = shares.once(0, [] {
    cudaFuncAttributes at;
    const cudaError_t got = cudaFuncGetAttributes(&at, idkm_jac_mma<D, NT, PACK>);
    return got != cudaSuccess ? got : (at.numRegs == JM_LAUNCH_REGS ? cudaSuccess : cudaErrorInvalidConfiguration);
  });
  if (rc == cudaSuccess) rc = allow_smem(limit, idkm_jac_mma<D, NT, PACK>, DYN);
  if (rc != cudaSuccess) return rc;
  idkm_jac_mma<D, NT, PACK><<<units, JM_THREADS, DYN, stream>>>(p);
  return cudaGetLastError();
}
cudaError_t launch_jac_mma(int d, const JacMmaPlan& pl, const JacMmaParams& p, int units, cudaStream_t stream) {
  if (p.k * d <= 64) return d == 4 ? launch_mma<4, 128, true>(p, units, stream) : launch_mma<2, 128, true>(p, units, stream);
  if (d == 4) return pl.nt == 128 ? launch_mma<4, 128, false>(p, units, stream) : launch_mma<4, 256, false>(p, units, stream);
  return pl.nt == 128 ? launch_mma<2, 128, false>(p, units, stream) : launch_mma<2, 256, false>(p, units, stream);
}
template <int D, int NT>
static cudaError_t launch_solve(const JacMmaPlan& pl, const JacMmaParams& p, cudaStream_t stream) {
  const int smem = (JS_ROWS + 1) * pl.kdp * 8;
  static PerDevice limit;
  const cudaError_t allowed = allow_smem(limit, idkm_jac_solve<D, NT>, (JS_ROWS + 1) * 1024 * 8);
  if (allowed != cudaSuccess) return allowed;
  void* args[1] = {const_cast<JacMmaParams*>(&p)};
  return cudaLaunchCooperativeKernel((const void*)&idkm_jac_solve<D, NT>, dim3((unsigned)(p.n_layers * p.solve_blocks), 1, 1), dim3(JS_T, 1, 1),
                                     args, (size_t)smem, stream);
}
cudaError_t launch_jac_solve(int d, const JacMmaPlan& pl, const JacMmaParams& p, cudaStream_t stream) {
  if (d == 4) return pl.nt == 128 ? launch_solve<4, 128>(pl, p, stream) : launch_solve<4, 256>(pl, p, stream);
  return pl.nt == 128 ? launch_solve<2, 128>(pl, p, stream) : launch_solve<2, 256>(pl, p, stream);
}

}  // namespace idkm
