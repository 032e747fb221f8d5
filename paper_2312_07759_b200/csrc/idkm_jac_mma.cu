// See idkm_jac_mma.cuh.  One block computes a 128 x NT tile of X^T Y over a range of weights.
//
// What bounds it: the products -- three fp16 products per multiply-add (below) -- and, almost as much, producing the
// operands: nothing of X and Y exists in memory, every tile computes its 128 + NT columns of them from the weights, the
// rows' softmax references and normalisers that the codebook-gradient pass left, and its centroids.  A tile of 128 x 256
// makes 96 (weight, centroid) pairs of work per weight at d = 4 for 32 768 multiply-adds.
//
// Precision.  X and Y are split into two fp16 terms (22 bits, scaled by powers of two so that the second term stays
// normal): hi hi + hi lo + lo hi; what is dropped is 2^-22 of a product, below the 2e-7 of the exponential and the
// reciprocal square root they are made of.  The tensor core adds in fp32 without rounding to nearest, so an accumulator
// takes one stage (64 weights) only -- small terms first -- and is then added to fp32 sums in registers, which move to an
// fp64 partial every 16 K weights; the splits' partials are added in a fixed order.
//
// Roles: a producing warp makes eight weights' share of the stage (a lane holds a centroid, so nothing crosses lanes) and
// writes it in the core-matrix order of the K-major operand, 16 bytes per lane and row of the operand: consecutive lanes
// are consecutive rows, no bank conflicts.  One thread issues the products of a stage and commits them to the stage's
// barrier, which frees its shared memory and hands its half of tensor memory to the accumulating warps.  Every wait is
// bounded; if one runs out the layer's status says so.
#include "idkm_jac_mma.cuh"

#include <string.h>

namespace idkm {

constexpr int JM_POLLS = 1 << 22;

template <int D, int NT>
struct JmCfg {
  static constexpr int CPM = JM_M / D, CPN = NT / D;      // centroids of a tile's rows / columns
  static constexpr int MU = CPM / 32, NU = CPN / 32;      // lane-per-centroid units of work per eight weights
  static constexpr int A_BYTES = JM_M * JM_ROWS * 2, B_BYTES = NT * JM_ROWS * 2;
  static constexpr int STAGE = 2 * A_BYTES + 2 * B_BYTES;
  static constexpr int ROW_FLOATS = D + 2;
  static constexpr int DYN = 2 * STAGE + 8 * 8 * 8 * 4;   // two stages, eight weights per producing warp
};

__device__ __forceinline__ bool jm_wait(unsigned long long* bar, unsigned parity) {
  for (int i = 0; i < JM_POLLS; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
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
__device__ __forceinline__ void jm_tmem_ld16(unsigned addr, float (&v)[16]) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
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

// Where entry ((mt, mrow), column of centroid l, coordinate b) of the product, or of the diagonal tiles, lies in the
// partial of unit 0 of its kind, and how far it is to the next split.
template <int D, int NT>
struct JmIndex {
  using Cfg = JmCfg<D, NT>;
  size_t xy, xy_step, dg, dg_step;
  int ns_n, ns_d;
  __device__ JmIndex(const JacMmaParams& p, int layer, int mt, int l, int b) {
    constexpr size_t TILE = (size_t)JM_M * NT;
    const int tn = p.tiles_m * p.tiles_n;
    ns_n = p.ns_n[layer];
    ns_d = p.ns_d[layer];
    const size_t first = (size_t)p.unit_first[layer];
    const int nt = l / Cfg::CPN, col = b * Cfg::CPN + l % Cfg::CPN;
    xy = (first + (size_t)mt * p.tiles_n + nt) * TILE + (size_t)(col % (NT / 2)) * 256 + (size_t)(col / (NT / 2)) * 128;
    xy_step = (size_t)tn * TILE;
    const int dc = b * Cfg::CPM + l % Cfg::CPM;
    dg = (first + (size_t)tn * ns_n + mt) * TILE + (size_t)(dc % 64) * 256 + (size_t)(dc / 64) * 128;
    dg_step = (size_t)p.tiles_m * TILE;
  }
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

// Eight weights of one centroid: the operand's entries for its D coordinates, split and stored.
// KIND 0: X (rows), 1: Y (columns), 2: n (columns of the diagonal tiles).
template <int D, int KIND>
__device__ __forceinline__ void jm_unit(const float* rows, const float (&c)[D], const float (&f)[D], float scale, float mul, unsigned char* hi,
                                        unsigned char* lo, int coord_bytes) {
  unsigned ph[D][4], pl[D][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float v[2][D];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float* r = rows + (2 * q + h) * 8;
      float w[D];
      if constexpr (D == 4) {
        const float4 x = *reinterpret_cast<const float4*>(r);
        w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
      } else {
        const float2 x = *reinterpret_cast<const float2*>(r);
        w[0] = x.x; w[1] = x.y;
      }
      const float2 rs = *reinterpret_cast<const float2*>(r + 4);
      float df[D], sq = 1e-30f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        df[a] = w[a] - c[a];
        sq = fmaf(df[a], df[a], sq);
      }
      const float ri = rsqrt_approx(sq);
      const float at = ex2_approx(fmaf(-scale, sq * ri, rs.x)) * rs.y;
      const float g = KIND == 0 ? at * mul : (KIND == 1 ? at * ri * mul : ri * mul);
#pragma unroll
      for (int a = 0; a < D; ++a) v[h][a] = (KIND == 0 ? w[a] - f[a] : df[a]) * g;
    }
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const __half2 h2 = __floats2half2_rn(v[0][a], v[1][a]);
      const float2 back = __half22float2(h2);
      const __half2 l2 = __floats2half2_rn(v[0][a] - back.x, v[1][a] - back.y);
      ph[a][q] = *reinterpret_cast<const unsigned*>(&h2);
      pl[a][q] = *reinterpret_cast<const unsigned*>(&l2);
    }
  }
#pragma unroll
  for (int a = 0; a < D; ++a) {
    *reinterpret_cast<uint4*>(hi + a * coord_bytes) = make_uint4(ph[a][0], ph[a][1], ph[a][2], ph[a][3]);
    *reinterpret_cast<uint4*>(lo + a * coord_bytes) = make_uint4(pl[a][0], pl[a][1], pl[a][2], pl[a][3]);
  }
}

template <int D, int NT>
__global__ void __launch_bounds__(JM_THREADS, 1) idkm_jac_mma(const __grid_constant__ JacMmaParams p) {
  using Cfg = JmCfg<D, NT>;
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
  // ---- this unit's tile and rows ----
  const int u0 = (int)blockIdx.x - p.unit_first[layer], tn = p.tiles_m * p.tiles_n;
  const bool diag = u0 >= tn * p.ns_n[layer];
  const int ud = diag ? u0 - tn * p.ns_n[layer] : u0, per = diag ? p.tiles_m : tn, ns = diag ? p.ns_d[layer] : p.ns_n[layer];
  const int split = ud / per, tile = ud % per;
  const int mt = diag ? tile : tile / p.tiles_n, nt = diag ? 0 : tile % p.tiles_n;
  const long long rows = p.row_off[layer + 1] - p.row_off[layer];
  const long long n_st = (rows + JM_ROWS - 1) / JM_ROWS;
  const long long st0 = n_st * split / ns, st1 = n_st * (split + 1) / ns;
  const int n = (int)(st1 - st0);
  const int ncols = diag ? JM_M : NT;
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
        mbar_init(&full[i], 8);
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
    // ================= accumulating warps; the first also issues the products =================
    // (the registers of the two kinds of warps add up to the 128 x 512 of the launch)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
    float acc[NT / 2];
#pragma unroll
    for (int i = 0; i < NT / 2; ++i) acc[i] = 0.f;
    const int half = warp >> 2, quad = warp & 3, cols = ncols / 2;
    const unsigned base = tmem + ((unsigned)(quad * 32) << 16) + (unsigned)(half * cols);
    double* mine = p.part + (size_t)blockIdx.x * (JM_M * NT) + half * 128 + quad * 32 + lane;
    const unsigned idesc = (1u << 4) | ((unsigned)(ncols >> 3) << 17) | ((unsigned)(JM_M >> 4) << 24);   // fp16 in, fp32 out
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(dyn);
    bool first = true, ok = true;
    // products of stage i: all terms of the split, the small ones first; the commit frees the stage's shared memory and
    // hands its half of tensor memory over
    auto issue = [&](int i) {
      const int s = i & 1;
      bool good = jm_wait(&full[s], (unsigned)((i >> 1) & 1));
      if (good && i >= 2) good = jm_wait(&tfree[s], (unsigned)(((i >> 1) - 1) & 1));
      if (!good) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lane == 0) {
        const unsigned a0 = sbase + s * Cfg::STAGE, b0 = a0 + 2 * Cfg::A_BYTES, dst = tmem + (unsigned)(s * NT);
#pragma unroll
        for (int t = 0; t < 3; ++t) {   // lo hi, hi lo, then hi hi
#pragma unroll
          for (int q = 0; q < JM_ROWS / 16; ++q) {
            const unsigned long long da = jm_desc(a0 + (t == 0 ? Cfg::A_BYTES : 0) + q * 2 * (JM_M * 16), JM_M * 16);
            const unsigned long long db = jm_desc(b0 + (t == 1 ? Cfg::B_BYTES : 0) + q * 2 * (NT * 16), NT * 16);
            jm_mma(dst, da, db, idesc, (t == 0 && q == 0) ? 0u : 1u);
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&done[s])) : "memory");
      }
      __syncwarp();
      return true;
    };
    int issued = 0;
    if (warp == 0 && n > 0) {
      ok = issue(0);
      issued = ok ? 1 : 0;
    }
    for (int i = 0; i < n && ok; ++i) {
      const int s = i & 1;
      if (warp == 0 && i + 1 < n) {   // the next stage's products before this one's sums are fetched
        ok = issue(i + 1);
        if (!ok) break;
        issued = i + 2;
      }
      ok = jm_wait(&done[s], (unsigned)((i >> 1) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (ok) {
#pragma unroll
        for (int q = 0; q < NT / 32; ++q) {
          if (q * 16 < cols) {
            float v[16];
            jm_tmem_ld16(base + (unsigned)(s * NT + q * 16), v);
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[q * 16 + e] += v[e];
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) jm_arrive(&tfree[s]);
      if ((i + 1) % JM_FOLD == 0 || i + 1 == n) {
#pragma unroll
        for (int q = 0; q < NT / 2; ++q)
          if (q < cols) {
            double* o = mine + (size_t)q * 256;
            *o = first ? (double)acc[q] : *o + (double)acc[q];
            acc[q] = 0.f;
          }
        first = false;
      }
    }
    if (!ok) {
      if (lane == 0) s_fail = 1;
      // (what is in flight ends before tensor memory is given back)
      if (warp == 0 && issued > 0) (void)jm_wait(&done[(issued - 1) & 1], (unsigned)(((issued - 1) >> 1) & 1));
    }
    if (n == 0) {
      for (int q = 0; q < cols; ++q) mine[(size_t)q * 256] = 0.0;
    }
  } else {
    // ================= producing warps: weights 8 pw .. 8 pw + 7 of every stage =================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    const int pw = warp - 8;
    float cx[Cfg::MU][D], fx[Cfg::MU][D], cy[Cfg::NU][D];
#pragma unroll
    for (int h = 0; h < Cfg::MU; ++h) {
      const int j = mt * Cfg::CPM + h * 32 + lane;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        cx[h][a] = j < k ? p.C[((size_t)layer * k + j) * D + a] : PAD_COORD;
        fx[h][a] = j < k ? p.F[((size_t)layer * k + j) * D + a] : 0.f;
      }
    }
#pragma unroll
    for (int h = 0; h < Cfg::NU; ++h) {
      const int j = (diag ? mt * Cfg::CPM : nt * Cfg::CPN) + h * 32 + lane;
#pragma unroll
      for (int a = 0; a < D; ++a) cy[h][a] = j < k ? p.C[((size_t)layer * k + j) * D + a] : PAD_COORD;
    }
    float* rowsm = reinterpret_cast<float*>(dyn + 2 * Cfg::STAGE) + pw * 64;   // [8][8]: w, reference, normaliser
    const long long row0 = p.row_off[layer];
    float4 wn = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 rn = make_float2(0.f, 0.f);
    auto fetch = [&](int i) {
      const long long loc = (st0 + i) * JM_ROWS + pw * 8 + lane;
      if (lane < 8 && i < n) {
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
    for (int i = 0; i < n && ok; ++i) {
      const int s = i & 1;
      if (i >= 2) ok = jm_wait(&done[s], (unsigned)(((i >> 1) - 1) & 1));
      __syncwarp();
      if (lane < 8) {
        *reinterpret_cast<float4*>(rowsm + lane * 8) = wn;
        *reinterpret_cast<float2*>(rowsm + lane * 8 + 4) = rn;
      }
      __syncwarp();
      fetch(i + 1);
      unsigned char* A = dyn + s * Cfg::STAGE + pw * (JM_M * 16) + lane * 16;
      unsigned char* B = dyn + s * Cfg::STAGE + 2 * Cfg::A_BYTES + pw * (NT * 16) + lane * 16;
      if (ok) {
#pragma unroll
        for (int h = 0; h < Cfg::MU; ++h)
          jm_unit<D, 0>(rowsm, cx[h], fx[h], p.scale, xm, A + h * 512, A + Cfg::A_BYTES + h * 512, Cfg::CPM * 16);
        if (!diag) {
#pragma unroll
          for (int h = 0; h < Cfg::NU; ++h)
            jm_unit<D, 1>(rowsm, cy[h], cy[h], p.scale, ym, B + h * 512, B + Cfg::B_BYTES + h * 512, Cfg::CPN * 16);
        } else {
#pragma unroll
          for (int h = 0; h < Cfg::MU; ++h)
            jm_unit<D, 2>(rowsm, cy[h], cy[h], p.scale, ym, B + h * 512, B + Cfg::B_BYTES + h * 512, Cfg::CPM * 16);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) jm_arrive(&full[s]);
    }
    if (!ok && lane == 0) s_fail = 1;
  }
  __threadfence();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * NT));
  const bool failed = *reinterpret_cast<volatile int*>(&s_fail) != 0;
  if (failed && tid == 0) st->status = ST_TIMEOUT;
  if (p.solve_blocks > 0) return;

  // ================= k d <= 64: the layer's last unit adds the partials and runs the iteration =================
  const int units = p.unit_first[layer + 1] - p.unit_first[layer];
  if (tid == 0) s_flag = atomicAdd(&st->ticket, 1u) == (unsigned)(units - 1);
  __syncthreads();
  if (!s_flag) return;
  __threadfence();
  const int nd = k * D;
  double* J = reinterpret_cast<double*>(dyn);   // [64][65]: J_C^T
  double* ub = J + 64 * 65;                     // [2][64]
  double* gs = ub + 128;                        // [64]
  double* red = gs + 64;                        // [2][8][2]
  for (int o = tid; o < 64 * 64; o += JM_THREADS) {
    const int q = o & 63, r = o >> 6;           // output coordinate (l, b), input coordinate (j, a)
    double s = 0.0;
    if (q < nd && r < nd) {
      const int l = q / D, b = q % D, j = r / D, a = r % D;
      const JmIndex<D, NT> ix(p, layer, 0, l, b);
      const int mrow = a * Cfg::CPM + j;
#pragma unroll 16
      for (int t = 0; t < ix.ns_n; ++t) s -= __ldcg(p.part + ix.xy + t * ix.xy_step + mrow);
      if (j == l)
#pragma unroll 16
        for (int t = 0; t < ix.ns_d; ++t) s += __ldcg(p.part + ix.dg + t * ix.dg_step + mrow);
      const float S = p.S[(size_t)layer * k + j];
      s *= (S >= S_MIN_F) ? p.inv_tau_d / (double)S * ((double)range / 268435456.0) : 0.0;
    }
    J[q * 65 + r] = s;
  }
  if (tid < 64) {
    gs[tid] = tid < nd ? (double)p.gvec[(size_t)layer * nd + tid] : 0.0;
    ub[tid] = gs[tid];
    ub[64 + tid] = 0.0;
  }
  __syncthreads();
  if (warp >= 8) return;
  const int q = tid >> 2, pr = tid & 3;         // four threads per output
  const double al = (double)p.alpha, be = 1.0 - al;
  JmStop stop;
  stop.status = st->status;
  double g2 = 0.0;
  for (int r = 0; r < nd; ++r) g2 += gs[r] * gs[r];
  const double u2_limit = ADJ_GROWTH_LIMIT * ADJ_GROWTH_LIMIT * g2;
  if (failed || stop.status == ST_TIMEOUT) stop.done = 1;
  while (stop.it < p.max_iter && !stop.done) {
    const double* u = ub + (stop.it & 1) * 64;
    double s = 0.0;
#pragma unroll
    for (int r = 0; r < 16; ++r) s = fma(J[q * 65 + pr * 16 + r], u[pr * 16 + r], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    const double uo = u[q], un = q < nd ? al * (s + gs[q]) + be * uo : 0.0;
    if (pr == 0) ub[((stop.it + 1) & 1) * 64 + q] = un;
    double num = pr == 0 ? (un - uo) * (un - uo) : 0.0, den = pr == 0 ? un * un : 0.0;
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
    num = den = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      num += rd[w * 2];
      den += rd[w * 2 + 1];
    }
    stop.test(p, layer, num, den, u2_limit, tid == 0);
  }
  if (pr == 0 && q < nd) p.u[(size_t)layer * nd + q] = (float)ub[(stop.it & 1) * 64 + q];
  if (tid == 0) stop.store(st);
}

// ---- larger codebooks: the iteration by many blocks, eight rows of J_C^T each, kept in shared memory ----
// Blocks of a layer meet at a bounded barrier once per step; the adjoint and the squares of the stop test cross L2.
constexpr int JS_T = 256, JS_ROWS = 8;
template <int D, int NT>
__global__ void __launch_bounds__(JS_T) idkm_jac_solve(const __grid_constant__ JacMmaParams p) {
  using Cfg = JmCfg<D, NT>;
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
  for (int mt = 0; mt < p.tiles_m; ++mt) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (own) {
      const JmIndex<D, NT> ix(p, layer, mt, l, c);
#pragma unroll 4
      for (int t = 0; t < ix.ns_n; ++t)
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r] -= __ldcg(p.part + ix.xy + t * ix.xy_step + lane + 32 * r);
      if (l / Cfg::CPM == mt)
        for (int t = 0; t < ix.ns_d; ++t)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if ((lane + 32 * r) % Cfg::CPM == l % Cfg::CPM) s[r] += __ldcg(p.part + ix.dg + t * ix.dg_step + lane + 32 * r);
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

int jac_mma_units_max(const JacMmaPlan& pl, int n_layers) { return JM_UNITS + n_layers * (pl.tiles_m * pl.tiles_n + pl.tiles_m); }

int jac_mma_split(const JacMmaPlan& pl, JacMmaParams* p) {
  const int L = p->n_layers, tn = pl.tiles_m * pl.tiles_n, td = pl.tiles_m;
  const double cd = pl.nt == 256 ? 0.6 : 1.0;   // a diagonal tile's cost against a product tile's
  const long long m = p->row_off[L];
  int units = 0;
  for (int l = 0; l < L; ++l) {
    const long long rows = p->row_off[l + 1] - p->row_off[l], n_st = (rows + JM_ROWS - 1) / JM_ROWS;
    const double budget = (double)JM_UNITS * (double)rows / (double)m;   // blocks this layer may use
    long long nn = (long long)(budget / ((double)tn + cd * td));
    if (nn < 1) nn = 1;
    long long nd = ((long long)budget - nn * tn) / td;
    if (nd < 1) nd = 1;
    if (nn > n_st) nn = n_st;
    if (nd > n_st) nd = n_st;
    p->unit_first[l] = units;
    p->ns_n[l] = (int)nn;
    p->ns_d[l] = (int)nd;
    units += (int)(nn * tn + nd * td);
  }
  for (int l = L; l <= MAX_LAYERS; ++l) p->unit_first[l] = units;
  return units;
}

template <int D, int NT>
static cudaError_t launch_mma(const JacMmaParams& p, int units, cudaStream_t stream) {
  constexpr int DYN = JmCfg<D, NT>::DYN;
  static bool configured = false;
  if (!configured) {
    const cudaError_t rc = cudaFuncSetAttribute(idkm_jac_mma<D, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, DYN);
    if (rc != cudaSuccess) return rc;
    configured = true;
  }
  idkm_jac_mma<D, NT><<<units, JM_THREADS, DYN, stream>>>(p);
  return cudaGetLastError();
}
cudaError_t launch_jac_mma(int d, const JacMmaPlan& pl, const JacMmaParams& p, int units, cudaStream_t stream) {
  if (d == 4) return pl.nt == 128 ? launch_mma<4, 128>(p, units, stream) : launch_mma<4, 256>(p, units, stream);
  return pl.nt == 128 ? launch_mma<2, 128>(p, units, stream) : launch_mma<2, 256>(p, units, stream);
}
template <int D, int NT>
static cudaError_t launch_solve(const JacMmaPlan& pl, const JacMmaParams& p, cudaStream_t stream) {
  const int smem = (JS_ROWS + 1) * pl.kdp * 8;
  static bool configured = false;
  if (!configured) {
    const cudaError_t rc = cudaFuncSetAttribute(idkm_jac_solve<D, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (JS_ROWS + 1) * 1024 * 8);
    if (rc != cudaSuccess) return rc;
    configured = true;
  }
  void* args[1] = {const_cast<JacMmaParams*>(&p)};
  return cudaLaunchCooperativeKernel((const void*)&idkm_jac_solve<D, NT>, dim3((unsigned)(p.n_layers * p.solve_blocks), 1, 1), dim3(JS_T, 1, 1),
                                     args, (size_t)smem, stream);
}
cudaError_t launch_jac_solve(int d, const JacMmaPlan& pl, const JacMmaParams& p, cudaStream_t stream) {
  if (d == 4) return pl.nt == 128 ? launch_solve<4, 128>(pl, p, stream) : launch_solve<4, 256>(pl, p, stream);
  return pl.nt == 128 ? launch_solve<2, 128>(pl, p, stream) : launch_solve<2, 256>(pl, p, stream);
}

}  // namespace idkm
