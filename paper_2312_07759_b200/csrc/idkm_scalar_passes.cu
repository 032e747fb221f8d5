// The passes around the loop for scalar weights: soft-quantised weights, codebook gradient, adjoint iteration and dL/dW,
// all in the interval form of idkm_scalar.cuh.  A weight costs a search for its interval, one exponential and one
// reciprocal whatever the number of centroids; the adjoint iteration (Section 4.2) does not visit the weights at all.
// Bound by memory and the search's shared-memory lookups.  Measured (soft weights / gradient / dL/dW against the passes over
// pairs): 11.7 M weights, k = 4 38 / 56 / 46 us against 48 / 54 / 56; k = 8 43 / 61 / 49 against 75 / 95 / 101; 16 M, k = 16
// 63 / 80 / 72 against 152 / 234 / 244.  Adjoint iteration of 50 steps, 21 layers, k = 4: 26 us against 104 on a matrix that a
// pass over the weights forms.
#include "idkm_scalar.cuh"

namespace idkm {

constexpr int SP_T = 256;

// Tables of a block, one float array per quantity (neighbouring lanes look up different intervals: arrays of floats keep
// the lookups of up to 32 intervals free of bank conflicts).
struct SpSearch {
  const float* v;   // sorted centroids, padded with +inf to 2 top - 1 entries
  int top;          // first step of the binary search
};
__device__ __forceinline__ int sp_interval(const SpSearch& s, float w) {
  int lo = 0;
  for (int step = s.top; step > 0; step >>= 1) lo += (s.v[lo + step - 1] < w) ? step : 0;
  return lo;   // centroids strictly below w
}
__device__ __forceinline__ SpSearch sp_load_search(float* v /* [512] */, const float* ft, int k) {
  int top = 1;
  while (2 * top <= k) top *= 2;
  for (int i = threadIdx.x; i < 2 * top - 1; i += blockDim.x) v[i] = i < k ? __ldg(ft + FT_V * (k + 1) + i) : __int_as_float(0x7f800000);
  return SpSearch{v, top};
}

// Rows of this block: a contiguous share of its layer, in units of four weights.
struct SpShare {
  int layer;
  long long row0, m, q0, q1;   // first row, rows of the layer, range of 4-weight groups
};
__device__ __forceinline__ SpShare sp_share(const ScalarParams& sp) {
  SpShare s;
  s.layer = sc_layer_of_block(sp, (int)blockIdx.x);
  const int b = (int)blockIdx.x - sp.blk_first[s.layer], NB = sp.blk_first[s.layer + 1] - sp.blk_first[s.layer];
  s.row0 = sp.row_off[s.layer];
  s.m = sp.row_off[s.layer + 1] - s.row0;
  const long long nq = (s.m + 3) / 4;
  s.q0 = nq * b / NB;
  s.q1 = nq * (b + 1) / NB;
  return s;
}

// ---- Wq = A C at the returned centroids (soft quantiser, Section 3.2) ----
__global__ void __launch_bounds__(SP_T) idkm_scalar_final(const __grid_constant__ ScalarParams sp) {
  __shared__ float v[512], te[257], to[257], tr[257], td[257];
  const SpShare sh = sp_share(sp);
  const int k = sp.k, K1 = k + 1;
  const float* ft = sp.p.ftab + (size_t)sh.layer * SC_NFTAB * K1;
  const float slope = (float)(2.0 * 1.4426950408889634 * sp.inv_tau_d);
  grid_dependency_sync();
  const SpSearch se = sp_load_search(v, ft, k);
  for (int i = threadIdx.x; i <= k; i += SP_T) {
    te[i] = ft[FT_E * K1 + i];
    to[i] = ft[FT_O * K1 + i];
    tr[i] = ft[FT_R * K1 + i];
    td[i] = ft[FT_D * K1 + i];
  }
  __syncthreads();
  const float* W = sp.p.W + sh.row0;
  auto one = [&](float w) {
    const int s = sp_interval(se, w);
    float lam, mu;
    sc_lambda(fmaf(w - te[s], slope, to[s]), lam, mu);
    return fmaf(lam, td[s], tr[s]);
  };
  const bool vec = (sh.row0 % 4) == 0;
  for (long long q = sh.q0 + threadIdx.x; q < sh.q1; q += SP_T) {
    const long long r = q * 4;
    if (vec && r + 4 <= sh.m) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(W) + q);
      const float o[4] = {one(x.x), one(x.y), one(x.z), one(x.w)};
      store_wq<4>(sp.p.Wq, sh.row0 + r, o, sp.wq_dtype, true);
    } else {
      for (int i = 0; i < 4; ++i)
        if (r + i < sh.m) {
          const float o[1] = {one(__ldg(W + r + i))};
          store_wq<1>(sp.p.Wq, sh.row0 + r + i, o, sp.wq_dtype, false);
        }
    }
  }
}

// ---- coefficients of dL/dW for an adjoint u (first kw warps; u of this thread's sorted centroid) ----
__device__ __forceinline__ void sp_write_coef(const ScalarParams& sp, int layer, double u, double* ex /* [3][257] */, double* tmp) {
  const int k = sp.k, j = threadIdx.x, kw = (k + 31) >> 5, K1 = k + 1;
  const bool own = j < k;
  const double* t = sp.p.tab + (size_t)layer * SC_NTAB * K1 + j;
  const double a = own ? t[TB_A * K1] : 0.0, ap = (own && j > 0) ? t[TB_A * K1 - 1] : 0.0;
  const double rP = own ? t[TB_RP * K1] : 0.0, rQ = own ? t[TB_RQ * K1] : 0.0, v = own ? t[TB_V * K1] : 0.0;
  const double S = own ? t[TB_S * K1] : 0.0;
  const double us = S > 0.0 ? u / S : 0.0, ka = us * (own ? t[TB_F * K1] : 0.0);
  double x[3] = {us, ka, v}, y[3] = {us, ka, v};
  lin_scan<3, true>(ap, x, k, tmp);
  lin_scan<3, false>(a, y, k, tmp);
  sc_sync(kw);
  if (own)
#pragma unroll
    for (int i = 0; i < 3; ++i) ex[i * 257 + j] = y[i] * rQ;
  sc_sync(kw);
  if (own) {
    float* o = sp.p.ftab + (size_t)layer * SC_NFTAB * K1 + j + 1;
    const double uL = x[0] * rP, kL = x[1] * rP, cL = x[2] * rP, T2 = 2.0 * sp.inv_tau_d;
    float c[5] = {(float)uL, 0.f, 0.f, 0.f, 0.f};
    if (j + 1 < k) {
      const double ref = (double)o[FT_E * K1] - sp.p.tab[(size_t)layer * SC_NTAB * K1 + TB_V * K1 + k];
      const double uR = ex[j + 1], kR = ex[257 + j + 1], cR = ex[2 * 257 + j + 1];
      c[0] = (float)(uL - uR);
      c[1] = (float)uR;
      c[2] = (float)(T2 * (cL - cR));
      c[3] = (float)(T2 * (uL - uR));
      c[4] = (float)(T2 * ((kL - kR) - ref * (uL - uR)));
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) o[(FT_U0 + i) * K1] = c[i];
    if (j == 0) {
#pragma unroll
      for (int i = 0; i < 5; ++i) o[(FT_U0 + i) * K1 - 1] = i == 1 ? (float)ex[0] : 0.f;
    }
  }
}

// ---- direct codebook gradient g = (dWq/dC)^T dL/dWq ----
// Every thread adds G lambda, G mu and G lambda mu of its weights to sums of its own, per interval, in shared memory
// (column = thread: no conflicts); T threads of the block take weights, as many as the sums leave room for.
// One fp32 sum per thread and interval is enough: against float64, with 70 % of the weights in one interval and a gradient of one
// sign, g is off by 3.8e-8 (64 M weights, k = 4: 221 weights a thread), 5e-8 (16 M, 16: 57), 3.3e-8 (20 M, 64) and 6.6e-8 (16 M, 256:
// 3500); with the sums moved to fp64 every 64 weights by 4.9e-8, 3.4e-8, 4.3e-8 and 3.3e-8, at 258 against 231 us (k = 4) and
// 1372 against 948 us (k = 256).
__global__ void __launch_bounds__(1024) idkm_scalar_grad(const __grid_constant__ ScalarParams sp, int T) {
  extern __shared__ __align__(16) float acc[];   // [3 (k + 1)][T]
  __shared__ float v[512], te[257], to[257];
  __shared__ double ex[3 * 257];
  __shared__ double tmp[32];
  __shared__ int s_flag;
  const SpShare sh = sp_share(sp);
  const int k = sp.k, K1 = k + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
  const int plen = 3 * K1;
  const float* ft = sp.p.ftab + (size_t)sh.layer * SC_NFTAB * K1;
  const float slope = (float)(2.0 * 1.4426950408889634 * sp.inv_tau_d);
  for (int i = tid; i < plen * T; i += nt) acc[i] = 0.f;
  grid_dependency_sync();
  const SpSearch se = sp_load_search(v, ft, k);
  for (int i = tid; i <= k; i += nt) {
    te[i] = ft[FT_E * K1 + i];
    to[i] = ft[FT_O * K1 + i];
  }
  __syncthreads();
  const float* W = sp.p.W + sh.row0;
  const float* G = sp.p.G + sh.row0;
  if (tid < T) {
    auto add = [&](int s, float w, float gv) {
      float lam, mu;
      sc_lambda(fmaf(w - te[s], slope, to[s]), lam, mu);
      float* o = acc + (3 * s) * T + tid;
      const float gl = gv * lam;
      o[0] += gl;
      o[T] += gv * mu;
      o[2 * T] += gl * mu;
    };
    auto one = [&](float w, float gv) {
      const int s = sp_interval(se, w);
      if (s < k && v[s] == w) {
        // on a centroid the sub-gradient of |w - c| is 0, the mean of its two sides'
        int s2 = s;
        while (s2 < k && v[s2] == w) ++s2;
        add(s, w, 0.5f * gv);
        add(s2, w, 0.5f * gv);
      } else {
        add(s, w, gv);
      }
    };
    const bool vec = (sh.row0 % 4) == 0;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
    auto fetch = [&](long long q, float4& a, float4& b) {
      const long long r = q * 4;
      if (vec && r + 4 <= sh.m) {
        a = __ldg(reinterpret_cast<const float4*>(W) + q);
        b = __ldg(reinterpret_cast<const float4*>(G) + q);
      } else {
        // rows past the end repeat the first row with a gradient of zero
        a = make_float4(__ldg(W + r), __ldg(W + (r + 1 < sh.m ? r + 1 : r)), __ldg(W + (r + 2 < sh.m ? r + 2 : r)), __ldg(W + (r + 3 < sh.m ? r + 3 : r)));
        b = make_float4(__ldg(G + r), r + 1 < sh.m ? __ldg(G + r + 1) : 0.f, r + 2 < sh.m ? __ldg(G + r + 2) : 0.f, r + 3 < sh.m ? __ldg(G + r + 3) : 0.f);
      }
    };
    long long q = sh.q0 + tid;
    if (q < sh.q1) fetch(q, x, y);
    for (; q < sh.q1; q += T) {
      const float4 cx = x, cy = y;
      if (q + T < sh.q1) fetch(q + T, x, y);
      one(cx.x, cy.x);
      one(cx.y, cy.y);
      one(cx.z, cy.z);
      one(cx.w, cy.w);
    }
  }
  __syncthreads();
  // ---- block sums, then over the layer's blocks (groups of RED_GROUP, then the groups; fixed order) ----
  const int b = (int)blockIdx.x - sp.blk_first[sh.layer], NB = sp.blk_first[sh.layer + 1] - sp.blk_first[sh.layer];
  double* tot = reinterpret_cast<double*>(acc);
  const int ngr = (NB + RED_GROUP - 1) / RED_GROUP;
  double* mine = sp.p.gpart + (size_t)blockIdx.x * plen;
  for (int o = warp; o < plen; o += nt / 32) {
    double s = 0.0;
    for (int i = lane; i < T; i += 32) s += (double)acc[o * T + i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) mine[o] = s;
  }
  if (NB == 1) {
    __syncthreads();
    for (int o = tid; o < plen; o += nt) tot[o] = mine[o];
  } else {
    const int g0 = sp.blk_first[sh.layer] / RED_GROUP + sh.layer;   // first group row / counter of the layer
    const int gr = b / RED_GROUP;
    const int gsize = NB - gr * RED_GROUP < RED_GROUP ? NB - gr * RED_GROUP : RED_GROUP;
    double* rows = sp.p.gpart + (size_t)gridDim.x * plen;            // [groups][plen]
    unsigned int* tick = sp.p.gtick;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_flag = atomicAdd(&tick[g0 + gr], 1u) == (unsigned int)(gsize - 1);
    __syncthreads();
    if (!s_flag) return;
    __threadfence();
    {
      const double* base = sp.p.gpart + (size_t)(sp.blk_first[sh.layer] + gr * RED_GROUP) * plen;
      for (int o = tid; o < plen; o += nt) {
        double x[RED_GROUP], s = 0.0;
#pragma unroll
        for (int i = 0; i < RED_GROUP; ++i) x[i] = i < gsize ? __ldcg(base + (size_t)i * plen + o) : 0.0;
#pragma unroll
        for (int i = 0; i < RED_GROUP; ++i) s += x[i];
        if (ngr > 1) rows[(size_t)(g0 + gr) * plen + o] = s;
        else tot[o] = s;
      }
    }
    if (tid == 0) tick[g0 + gr] = 0u;
    if (ngr > 1) {
      __threadfence();
      __syncthreads();
      if (tid == 0) s_flag = atomicAdd(&sp.p.st[sh.layer].ticket, 1u) == (unsigned int)(ngr - 1);
      __syncthreads();
      if (!s_flag) return;
      __threadfence();
      for (int o = tid; o < plen; o += nt) {
        double s = 0.0;
#pragma unroll 4
        for (int i = 0; i < ngr; ++i) s += __ldcg(rows + (size_t)(g0 + i) * plen + o);
        tot[o] = s;
      }
    }
  }
  __syncthreads();
  const int kw = (k + 31) >> 5;
  if (tid >= kw * 32) return;
  // ---- epilogue: what every centroid receives from the intervals right and left of it ----
  const bool own = tid < k;
  const double* t = sp.p.tab + (size_t)sh.layer * SC_NTAB * K1 + tid;
  const double a = own ? t[TB_A * K1] : 0.0, ap = (own && tid > 0) ? t[TB_A * K1 - 1] : 0.0;
  const double rP = own ? t[TB_RP * K1] : 0.0, rQ = own ? t[TB_RQ * K1] : 0.0, vj = own ? t[TB_V * K1] : 0.0;
  double pc[1] = {vj}, qc[1] = {vj};
  lin_scan<1, true>(ap, pc, k, tmp);
  lin_scan<1, false>(a, qc, k, tmp);
  sc_sync(kw);
  if (own) {
    ex[tid] = pc[0] * rP;          // average of the centroids up to this one
    ex[257 + tid] = qc[0] * rQ;    // ... from this one on
  }
  sc_sync(kw);
  double x[2] = {0.0, 0.0}, y[2] = {0.0, 0.0};
  const double it = sp.inv_tau_d;
  if (own) {
    // interval to the right of v_j: lambda part; interval to its left: mu part
    const double gl = tot[3 * (tid + 1)], gp = tot[3 * (tid + 1) + 2];
    const double cL = ex[tid], cR = tid + 1 < k ? ex[257 + tid + 1] : cL;
    x[0] = (gl + it * ((cL - cR) * gp - cL * gl)) * rP;
    x[1] = it * gl * rP;
    const double gm = tot[3 * tid + 1], gq = tot[3 * tid + 2];
    const double dR = ex[257 + tid], dL = tid > 0 ? ex[tid - 1] : dR;
    y[0] = (gm + it * ((dL - dR) * gq + dR * gm)) * rQ;
    y[1] = -it * gm * rQ;
  }
  lin_scan<2, false>(a, x, k, tmp);
  lin_scan<2, true>(ap, y, k, tmp);
  double r[2] = {0.0, 0.0};
  double g = 0.0;
  if (own) {
    g = (x[0] + vj * x[1]) + (y[0] + vj * y[1]);
    if (!(g == g) || fabs(g) > 1e300) r[0] = 1.0;
    r[1] = g * g;
    const size_t o = (size_t)sh.layer * k + sp.p.perm[(size_t)sh.layer * k + tid];
    sp.p.gvec[o] = (float)g;
    sp.p.u[o] = (float)g;
    if (sp.p.dC) sp.p.dC[o] = (float)g;
  }
  sc_reduce<2>(r, k, tmp);
  sp_write_coef(sp, sh.layer, (double)(float)g, ex, tmp);
  if (tid == 0) {
    LayerState* st = sp.p.st + sh.layer;
    st->ticket = 0u;
    st->adj_done = (r[0] > 0.0) ? 1 : 0;
    st->adj_iters = 0;
    st->adj_res = 0.f;
    st->adj_up = 0;
    st->adj_prev = 3.0e38f;
    st->g_norm = (float)sqrt(r[1]);
    if (r[0] > 0.0) st->status = ST_NONFINITE;
    else if (st->status == ST_DIVERGED) st->status = ST_OK;
  }
}

// ---- the adjoint iteration u <- alpha (J_C^T u + g) + (1 - alpha) u (Section 4.2) on the interval sums ----
// With p_ij = (u_j / S_j) (w_i - F_j), (J_C^T u)_l = (1 / tau) sum_i A_il (p_il - sum_j A_ij p_ij) n_il; every sum over i is
// one of the six sums per interval the loop kernel left (lambda, lambda w, mu, mu w, lambda mu, lambda mu w), so a step is
// six linear recurrences over the centroids.  One block per layer, fp64.
//
// KD > 0 (k <= KD <= 32): one warp.  Lane q first runs the recurrences on the q-th unit vector by itself, which gives the
// k x k matrix J_C^T; lane l then keeps row l and a step is a row times the vector in shared memory.  The stop test of a
// step is taken while the next one is computed (its critical path -- reductions, a division, a square root -- is as long
// as the step's).  KD == 0: one thread per centroid, the recurrences by scans.
template <int KD>
__global__ void __launch_bounds__(KD > 0 ? 32 : 256) idkm_scalar_adjoint(const __grid_constant__ ScalarParams sp) {
  __shared__ double ex[4 * 257];
  __shared__ double tmp[32];
  const int layer = blockIdx.x, k = sp.k, j = threadIdx.x, kw = (k + 31) >> 5, K1 = k + 1;
  if (j >= kw * 32) return;
  grid_dependency_sync();
  LayerState* st = sp.p.st + layer;
  if (st->adj_done) return;
  const bool own = j < k;
  const double* t = sp.p.tab + (size_t)layer * SC_NTAB * K1 + j;
  const double a = own ? t[TB_A * K1] : 0.0, ap = (own && j > 0) ? t[TB_A * K1 - 1] : 0.0;
  const double rP = own ? t[TB_RP * K1] : 0.0, rQ = own ? t[TB_RQ * K1] : 0.0;
  const double S = own ? t[TB_S * K1] : 0.0, F = own ? t[TB_F * K1] : 0.0;
  const double rS = S > 0.0 ? 1.0 / S : 0.0;
  const double L0 = own ? t[TB_L0 * K1] : 0.0, L1 = own ? t[TB_L1 * K1] : 0.0;
  const double M0 = own ? t[TB_M0 * K1] : 0.0, M1 = own ? t[TB_M1 * K1] : 0.0;
  const double X0 = own ? t[TB_X0 * K1] : 0.0, X1 = own ? t[TB_X1 * K1] : 0.0;
  const double Y0 = (own && j > 0) ? t[TB_X0 * K1 - 1] : 0.0, Y1 = (own && j > 0) ? t[TB_X1 * K1 - 1] : 0.0;
  double D1, D0;
  {
    double x[2] = {L1 * rP, L0 * rP}, y[2] = {M1 * rQ, M0 * rQ};
    lin_scan<2, false>(a, x, k, tmp);
    lin_scan<2, true>(ap, y, k, tmp);
    D1 = x[0] - y[0];
    D0 = x[1] - y[1];
  }
  const size_t o = (size_t)layer * k + (own ? sp.p.perm[(size_t)layer * k + j] : 0);
  const double g = own ? (double)sp.p.gvec[o] : 0.0;
  double u = g;
  const double al = (double)sp.alpha, be = 1.0 - al, it_d = sp.inv_tau_d;
  double gg[1] = {g * g};
  sc_reduce<1>(gg, k, tmp);
  const double u2_limit = ADJ_GROWTH_LIMIT * ADJ_GROWTH_LIMIT * gg[0];
  int it = 0, status = st->status, done = 0;
  int up = 0;
  float res = 0.f, prev = 3.0e38f;
  // the stop test of step `it` from |u+ - u|^2 and |u+|^2 (not finite if any entry is not)
  auto stop_test = [&](double num, double den) {
    res = sqrtf((float)(num / fmax(den, 1e-300)));
    ++it;
    if (j == 0 && it <= HIST_CAP) sp.p.hist_adj[(size_t)layer * HIST_CAP + it - 1] = res;
    up = (res > prev) ? up + 1 : 0;
    prev = res;
    if (!(den <= 1e300) || up >= 10 || den > u2_limit) {
      status = ST_DIVERGED;
      done = 1;
    } else if (sp.tol > 0.f && res < sp.tol) {
      done = 1;
    } else if (sp.tol > 0.f && it >= sp.max_iter && status == ST_OK) {
      status = ST_MAXITER;
    }
  };
  if constexpr (KD > 0) {
    __shared__ double cf[16][KD];        // per-centroid coefficients
    __shared__ double sL[2][KD][33];     // left averages of the unit vectors, later right-to-left sums
    __shared__ double JT[KD][KD + 1];
    __shared__ __align__(16) double ub[2][KD];
    if (j < KD) {
      const double c[16] = {a, ap, rP, rQ, rS, rS * F, L0 - X0, L1 - X1, X0, X1, Y0, Y1, M0 - Y0, M1 - Y1, D0, D1};
#pragma unroll
      for (int i = 0; i < 16; ++i) cf[i][j] = c[i];
    }
    __syncwarp();
    if (j < KD) {
      const int q = j;
      // left averages of every centroid (u and u F weighted), going right
      double p0 = 0.0, p1 = 0.0;
      for (int s = 0; s < k; ++s) {
        p0 = fma(cf[1][s], p0, s == q ? cf[4][s] : 0.0);
        p1 = fma(cf[1][s], p1, s == q ? cf[5][s] : 0.0);
        sL[0][s][q] = p0 * cf[2][s];
        sL[1][s][q] = p1 * cf[2][s];
      }
      // going left: right averages q0, q1 and the sums that interval s + 1 sends to the centroids on its left
      double q0 = 0.0, q1 = 0.0, un = 0.0, kn = 0.0, acc = 0.0;
      for (int s = k - 1; s >= 0; --s) {
        q0 = fma(cf[0][s], q0, s == q ? cf[4][s] : 0.0);
        q1 = fma(cf[0][s], q1, s == q ? cf[5][s] : 0.0);
        const double lt = (sL[0][s][q] * cf[7][s] - sL[1][s][q] * cf[6][s] + un * cf[9][s] - kn * cf[8][s]) * cf[2][s];
        acc = fma(cf[0][s], acc, lt);
        un = q0 * cf[3][s];
        kn = q1 * cf[3][s];
        // what interval s sends to the right, waiting for the way back
        const double ul = s > 0 ? sL[0][s - 1][q] : 0.0, kl = s > 0 ? sL[1][s - 1][q] : 0.0;
        const double rt = (ul * cf[11][s] - kl * cf[10][s] + un * cf[13][s] - kn * cf[12][s]) * cf[3][s];
        if (q < k) JT[s][q] = -acc + (s == q ? cf[4][s] * cf[15][s] - cf[5][s] * cf[14][s] : 0.0);
        sL[0][s][q] = rt;   // (entry s is not read again on this way; s - 1 still is)
      }
      double back = 0.0;
      for (int s = 0; s < k; ++s) {
        back = fma(cf[1][s], back, sL[0][s][q]);
        JT[s][q] = al * it_d * (JT[s][q] + back) + (s == q ? be : 0.0);
      }
    }
    __syncwarp();
    double row[KD];
#pragma unroll
    for (int r = 0; r < KD; ++r) row[r] = (own && r < k) ? JT[j][r] : 0.0;
    const double ag = al * g;
    if (j < KD) {
      ub[0][j] = u;
      ub[1][j] = 0.0;
    }
    __syncwarp();
    double num = 0.0, den = 0.0;
    bool pending = false;
    for (int step = 0;; ++step) {
      // u+ of this step, and the stop test of the one before it
      double s0 = ag, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      const double* b = ub[step & 1];
#pragma unroll
      for (int r = 0; r < KD; r += 4) {
        s0 = fma(row[r], b[r], s0);
        if (r + 1 < KD) s1 = fma(row[r + 1], b[r + 1], s1);
        if (r + 2 < KD) s2 = fma(row[r + 2], b[r + 2], s2);
        if (r + 3 < KD) s3 = fma(row[r + 3], b[r + 3], s3);
      }
      const double un = own ? (s0 + s1) + (s2 + s3) : 0.0;
      if (pending) stop_test(num, den);
      if (done || step >= sp.max_iter) break;
      num = (un - u) * (un - u);
      den = un * un;
#pragma unroll
      for (int off = (KD > 16 ? 16 : KD / 2); off > 0; off >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, off);
        den += __shfl_xor_sync(0xffffffffu, den, off);
      }
      if constexpr (KD < 32) {   // (lanes beyond KD hold zeros: everybody takes the first group's sums)
        num = __shfl_sync(0xffffffffu, num, 0);
        den = __shfl_sync(0xffffffffu, den, 0);
      }
      u = un;
      if (j < KD) ub[(step + 1) & 1][j] = un;
      __syncwarp();
      pending = true;
    }
  } else {
    while (it < sp.max_iter && !done) {
      const double us = u * rS, ka = us * F;
      double x[2] = {us, ka}, y[2] = {us, ka};
      lin_scan<2, true>(ap, x, k, tmp);
      lin_scan<2, false>(a, y, k, tmp);
      const double uL = x[0] * rP, kL = x[1] * rP, uR = y[0] * rQ, kR = y[1] * rQ;
      // right averages of the interval to the right, left averages of the interval to the left
      sc_sync(kw);
      if (own) {
        ex[j] = uR;
        ex[257 + j] = kR;
        ex[514 + j] = uL;
        ex[771 + j] = kL;
      }
      sc_sync(kw);
      const double uRn = j + 1 < k ? ex[j + 1] : 0.0, kRn = j + 1 < k ? ex[257 + j + 1] : 0.0;
      const double uLp = (own && j > 0) ? ex[514 + j - 1] : 0.0, kLp = (own && j > 0) ? ex[771 + j - 1] : 0.0;
      double lt[1] = {(uL * (L1 - X1) - kL * (L0 - X0) + uRn * X1 - kRn * X0) * rP};
      double rt[1] = {(uLp * Y1 - kLp * Y0 + uR * (M1 - Y1) - kR * (M0 - Y0)) * rQ};
      lin_scan<1, false>(a, lt, k, tmp);
      lin_scan<1, true>(ap, rt, k, tmp);
      const double jt = it_d * (us * D1 - ka * D0 - lt[0] + rt[0]);
      const double un = own ? al * (jt + g) + be * u : 0.0;
      double r[2] = {(un - u) * (un - u), un * un};
      sc_reduce<2>(r, k, tmp);
      u = un;
      stop_test(r[0], r[1]);
    }
  }
  if (own) {
    sp.p.u[o] = (float)u;
    if (sp.p.dC) sp.p.dC[o] = (float)u;
  }
  sc_sync(kw);
  sp_write_coef(sp, layer, (double)(float)u, ex, tmp);
  if (j == 0) {
    st->adj_iters = it;
    st->adj_res = res;
    st->adj_up = up;
    st->adj_prev = prev;
    st->adj_done = 1;
    st->status = status;
  }
}

// ---- dL/dW = (dWq/dW)^T dWq + (dF/dW)^T u: per weight uR + lambda (uL - uR) - (2 / tau) lambda mu (z_L - z_R) ----
__global__ void __launch_bounds__(SP_T) idkm_scalar_dw(const __grid_constant__ ScalarParams sp) {
  __shared__ float v[512], te[257], to[257], tu[5][257];
  const SpShare sh = sp_share(sp);
  const int k = sp.k, K1 = k + 1;
  const float* ft = sp.p.ftab + (size_t)sh.layer * SC_NFTAB * K1;
  const float slope = (float)(2.0 * 1.4426950408889634 * sp.inv_tau_d);
  grid_dependency_sync();
  const SpSearch se = sp_load_search(v, ft, k);
  for (int i = threadIdx.x; i <= k; i += SP_T) {
    te[i] = ft[FT_E * K1 + i];
    to[i] = ft[FT_O * K1 + i];
#pragma unroll
    for (int q = 0; q < 5; ++q) tu[q][i] = ft[(FT_U0 + q) * K1 + i];
  }
  __syncthreads();
  const float* W = sp.p.W + sh.row0;
  const float* G = sp.p.G + sh.row0;
  float* dW = sp.p.dW + sh.row0;
  auto at = [&](int s, float w, float gv) {
    const float x = w - te[s];
    float lam, mu;
    sc_lambda(fmaf(x, slope, to[s]), lam, mu);
    const float z = fmaf(gv, tu[2][s], fmaf(x, tu[3][s], -tu[4][s]));
    return fmaf(-lam * mu, z, fmaf(lam, tu[0][s], tu[1][s]));
  };
  auto one = [&](float w, float gv) {
    const int s = sp_interval(se, w);
    float r = at(s, w, gv);
    if (s < k && v[s] == w) {   // on a centroid: the mean of the two sides (sub-gradient 0)
      int s2 = s;
      while (s2 < k && v[s2] == w) ++s2;
      r = 0.5f * (r + at(s2, w, gv));
    }
    return r;
  };
  const bool vec = (sh.row0 % 4) == 0;
  for (long long q = sh.q0 + threadIdx.x; q < sh.q1; q += SP_T) {
    const long long r = q * 4;
    if (vec && r + 4 <= sh.m) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(W) + q), y = __ldg(reinterpret_cast<const float4*>(G) + q);
      reinterpret_cast<float4*>(dW)[q] = make_float4(one(x.x, y.x), one(x.y, y.y), one(x.z, y.z), one(x.w, y.w));
    } else {
      for (int i = 0; i < 4; ++i)
        if (r + i < sh.m) dW[r + i] = one(__ldg(W + r + i), __ldg(G + r + i));
    }
  }
}

// Launch that may be scheduled while the stream's previous kernel drains (every kernel here waits for it before its first
// read of what it wrote).
template <typename K, typename... A>
static cudaError_t launch_after(K kernel, int grid, int threads, int smem, cudaStream_t stream, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_scalar_final(const ScalarParams& sp, int grid, cudaStream_t stream) {
  return launch_after(idkm_scalar_final, grid, SP_T, 0, stream, sp);
}
cudaError_t launch_scalar_dw(const ScalarParams& sp, int grid, cudaStream_t stream) {
  return launch_after(idkm_scalar_dw, grid, SP_T, 0, stream, sp);
}
cudaError_t launch_scalar_adjoint(const ScalarParams& sp, cudaStream_t stream) {
  if (sp.k <= 4) return launch_after(idkm_scalar_adjoint<4>, sp.n_layers, 32, 0, stream, sp);
  if (sp.k <= 8) return launch_after(idkm_scalar_adjoint<8>, sp.n_layers, 32, 0, stream, sp);
  if (sp.k <= 16) return launch_after(idkm_scalar_adjoint<16>, sp.n_layers, 32, 0, stream, sp);
  if (sp.k <= 32) return launch_after(idkm_scalar_adjoint<32>, sp.n_layers, 32, 0, stream, sp);
  return launch_after(idkm_scalar_adjoint<0>, sp.n_layers, 256, 0, stream, sp);
}
constexpr int SP_GRAD_BYTES = 200 * 1024;
int scalar_grad_threads(int k) {
  const int T = SP_GRAD_BYTES / (12 * (k + 1)) / 32 * 32;   // k <= 15: 1024 threads; k = 256: 64
  return T > 1024 ? 1024 : T;
}
cudaError_t launch_scalar_grad(const ScalarParams& sp, int grid, cudaStream_t stream) {
  static PerDevice limit;
  const cudaError_t allowed = allow_smem(limit, idkm_scalar_grad, SP_GRAD_BYTES);
  if (allowed != cudaSuccess) return allowed;
  const int T = scalar_grad_threads(sp.k);
  return launch_after(idkm_scalar_grad, grid, T < 256 ? 256 : T, 12 * (sp.k + 1) * T, stream, sp, T);
}

}  // namespace idkm
