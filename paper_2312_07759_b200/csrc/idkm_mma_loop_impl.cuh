// The forward loop's arithmetic on warp-level matrix instructions.
//
// A warp takes eight weights at a time against all centroids: lane (g, t) = (lane / 4, lane % 4) holds the centroids
// g and g + 8 of every 16 and the weights t and t + 4 of the eight, which is how m16n8k8 wants its left operand, the
// attention.  So the column sums -- d + 1 multiply-adds a (weight, centroid) pair, a third of the pair's instructions, and
// d + 1 registers a centroid -- are products A^T [r, r w] whose operands are where they are needed.
//
// Precision: the attention and the right operand are split into two tf32 terms (22 bits); hi hi + hi lo + lo hi.  An
// accumulator takes the products of one set of eight weights, smallest terms first, and is added to fp32 sums (rounded to
// nearest), which move to fp64 sums in shared memory every MML_SPILL sets: the tensor cores' own running sum would be cut,
// not rounded.
#pragma once
#include "idkm_mma_loop.cuh"

namespace idkm {

constexpr int MML_SPILL = 64;

template <int MT>
struct MmlCfg {
  static constexpr int D = 4, KP = MT * 16, NA = D + 1;
  static constexpr int T = MT == 16 ? 256 : (MT == 8 ? 512 : 384), NW = T / 32;
  static constexpr int PLEN = KP * NA + D;
  static constexpr int QG = 4;                   // tiles whose instructions are interleaved by hand
  static constexpr int CDYN = MT * 8 * D * 8;                  // packed centroids
  static constexpr int SDYN = NW * MT * 4 * 32 * 8;            // fp64 sums of every warp
  static constexpr int DYN = CDYN + SDYN;
};

__device__ __forceinline__ void mma_tf32(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// ... with nothing added
__device__ __forceinline__ void mma_tf32_first(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// the 11 leading bits of x, which tf32 holds: cut, or rounded
__device__ __forceinline__ float tf32_cut(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }
__device__ __forceinline__ float tf32_rn(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u); }
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// over the lanes of equal t
__device__ __forceinline__ float mml_min(float v) {
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float mml_sum(float v) {
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int D, int KP, int T>
struct LoopShared {
  float c[KP * D];   // the centroids (padding: far away)
  double tot[KP * (D + 1) + D], part[T];
  double red[T / 32][2];
  float box[T / 32][D][2];
  int cnt[T / 32][2];
  double res;
  int flags[3], ok;   // dead, bad, collapse
};
template <int D, int KP, int T, bool SQ, class Rows>
__device__ __forceinline__ void loop_frame(const MmaLoopParams& mp, LoopShared<D, KP, T>& sh, Rows&& rows) {
  constexpr int NW = T / 32, NA = D + 1, PLEN = KP * NA + D;
  const SmallLoopParams& sp = mp.s;
  float* c_sm = sh.c;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, k = sp.k;
  const int b = (int)blockIdx.x;
  const long long m = sp.row_off[1];
  const float* Wl = sp.W;
  float* Cl = sp.C;
  LayerState* st = sp.st;
  double* gtot = mp.totals;

  int iters = 0, done = 0, status = ST_OK, dead_n = 0;
  int precise = SQ ? 0 : st->precise[0];
  float res_f = 0.f;
  for (int i = tid; i < KP * D; i += T) c_sm[i] = i < k * D ? Cl[i] : PAD_COORD;
  __syncthreads();
  bool ok = true;

  for (int it = 0; it < sp.max_iter; ++it) {
    if (done) break;
    const size_t buf = mp.one_stage ? (size_t)(it & 1) * G : 0;   // (with one barrier the next iteration's partials need a second buffer)
    rows(precise, b, G, m, Wl, sp.partials + (buf + b) * PLEN);
    // ---- everyone has published ----
    const unsigned arrivals = (unsigned)(G + sp.missing_arrivals);
    ok = small_barrier(sp.sync, (unsigned)(mp.one_stage ? it + 1 : 2 * it + 1) * arrivals, sp.spin_limit, &sh.ok);
    if (!ok) break;
    // ---- the layer's totals.  Few partials: every block adds them all, in the same order.  Many: it adds its share of the
    // sums, and after a second barrier reads the rest ----
    const double* base = sp.partials + buf * PLEN;
    if (!mp.one_stage) {
      const int o0 = (int)((long long)PLEN * b / G), o1 = (int)((long long)PLEN * (b + 1) / G);
      if (G >= 16) {
        for (int o = o0 + warp; o < o1; o += NW) {
          double v = 0.0;
          for (int q = lane; q < G; q += 32) v += __ldcg(base + (size_t)q * PLEN + o);
#pragma unroll
          for (int x = 16; x > 0; x >>= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
          if (lane == 0) __stcg(gtot + o, v);
        }
      } else {
        for (int o = o0 + tid; o < o1; o += T) {
          double v = 0.0;
          for (int q = 0; q < G; ++q) v += __ldcg(base + (size_t)q * PLEN + o);
          __stcg(gtot + o, v);
        }
      }
      ok = small_barrier(sp.sync, (unsigned)(2 * it + 2) * arrivals, sp.spin_limit, &sh.ok);
      if (!ok) break;
    }
    if (!mp.one_stage) {
      for (int o = tid; o < PLEN; o += T) sh.tot[o] = __ldcg(gtot + o);
    } else if constexpr (PLEN <= T / 2) {
      constexpr int CH = T / PLEN;
      const int ch = tid / PLEN, o = tid % PLEN;
      if (ch < CH) {
        double v = 0.0;
#pragma unroll 8
        for (int q = ch; q < G; q += CH) v += __ldcg(base + (size_t)q * PLEN + o);
        sh.part[tid] = v;
      }
      __syncthreads();
      if (tid < PLEN) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < CH; ++q) v += sh.part[q * PLEN + tid];
        sh.tot[tid] = v;
      }
    } else {
      for (int o = tid; o < PLEN; o += T) {
        double v = 0.0;
#pragma unroll 8
        for (int q = 0; q < G; ++q) v += __ldcg(base + (size_t)q * PLEN + o);
        sh.tot[o] = v;
      }
    }
    __syncthreads();
    const double* tot = sh.tot;
    // ---- M-step, by every block alike: a thread's entries are of one coordinate ----
    constexpr int NV = (KP * D + T - 1) / T;
    const int a = tid % D;
    const double c0a = (double)c_sm[a], mk = (double)m / (double)k;
    const double ubar = precise ? (tot[KP * NA + a] - (double)m * c0a) / (double)k : 0.0;
    double num = 0.0, den = 0.0;
    int bad = 0, dead = 0;
    float lo = 3.0e38f, hi = -3.0e38f, cn[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int i = tid + v * T, j = i / D;
      if (i < k * D) {
        const double tS = tot[j * NA], tN = tot[j * NA + 1 + a];
        const double s = precise ? mk + tS : tS, cold = (double)c_sm[i];
        const bool alive = (s >= S_MIN);
        const double cnew = alive ? (precise ? c0a + (ubar + tN) / s : tN / s) : cold;
        if (!alive && a == 0) ++dead;
        if (!(s == s) || s > 1e300 || !(cnew == cnew) || fabs(cnew) > 1e300) ++bad;
        num += (cnew - cold) * (cnew - cold);
        den += cnew * cnew;
        cn[v] = (float)cnew;
        lo = fminf(lo, cn[v]);
        hi = fmaxf(hi, cn[v]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    dead = __reduce_add_sync(0xffffffffu, dead);
    bad = __reduce_add_sync(0xffffffffu, bad);
#pragma unroll
    for (int o = 16; o >= D; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __syncthreads();   // (everybody has read the old centroids)
    if (lane < D) {
      sh.box[warp][lane][0] = lo;
      sh.box[warp][lane][1] = hi;
    }
    if (lane == 0) {
      sh.red[warp][0] = num;
      sh.red[warp][1] = den;
      sh.cnt[warp][0] = dead;
      sh.cnt[warp][1] = bad;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (tid + v * T < k * D) c_sm[tid + v * T] = cn[v];
    __syncthreads();
    if (warp == 0) {
      double n2 = lane < NW ? sh.red[lane][0] : 0.0, d2 = lane < NW ? sh.red[lane][1] : 0.0;
      int dd = lane < NW ? sh.cnt[lane][0] : 0, bb = lane < NW ? sh.cnt[lane][1] : 0;
      double ext = 0.0;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        float l2 = lane < NW ? sh.box[lane][c][0] : 3.0e38f, h2 = lane < NW ? sh.box[lane][c][1] : -3.0e38f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          l2 = fminf(l2, __shfl_xor_sync(0xffffffffu, l2, o));
          h2 = fmaxf(h2, __shfl_xor_sync(0xffffffffu, h2, o));
        }
        const double x = (double)h2 - (double)l2;
        ext += x * x;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      }
      dd = __reduce_add_sync(0xffffffffu, dd);
      bb = __reduce_add_sync(0xffffffffu, bb);
      if (lane == 0) {
        sh.res = (double)sqrtf((float)(n2 / fmax(d2, 1e-300)));
        sh.flags[0] = dd;
        sh.flags[1] = bb;
        sh.flags[2] = (!SQ && ext * sp.inv_tau_d * sp.inv_tau_d <= (double)PRECISE_SPAN * (double)PRECISE_SPAN) ? 1 : 0;
      }
    }
    __syncthreads();
    iters = it + 1;
    res_f = (float)sh.res;
    if (b == 0 && tid == 0 && iters <= HIST_CAP) sp.hist[iters - 1] = res_f;
    dead_n = sh.flags[0];
    precise = sh.flags[2];
    if (sh.flags[1] > 0) {
      status = ST_NONFINITE;
      done = iters;
    } else if (sp.tol > 0.f && res_f < sp.tol) {
      done = iters;
      status = ST_OK;
    } else if (sp.tol > 0.f && iters >= sp.max_iter) {
      status = ST_MAXITER;
    }
    __syncthreads();
  }

  if (b == 0) {
    for (int i = tid; i < k * D; i += T) Cl[i] = c_sm[i];
    if (tid == 0) {
      st->fwd_iters = iters;
      st->fwd_res = res_f;
      st->dead = dead_n;
      st->fwd_done = done;
      st->precise[0] = st->precise[1] = precise;
      st->status = ok ? status : ST_TIMEOUT;
      st->ticket = 0u;
    }
  }
}


template <int MT, bool SQ>
__global__ void __launch_bounds__(MmlCfg<MT>::T, 1) idkm_mma_loop(const __grid_constant__ MmaLoopParams mp) {
  using Cfg = MmlCfg<MT>;
  constexpr int D = Cfg::D, QG = Cfg::QG, QD = 2;
  constexpr int T = Cfg::T, NW = Cfg::NW, NA = Cfg::NA, KP = Cfg::KP;
  const SmallLoopParams& sp = mp.s;
  extern __shared__ __align__(16) unsigned char dyn[];
  // minus the centroids, (g, g + 8) side by side: [tile][D / 2][8 g][4] = -(c_g[a], c_g+8[a], c_g[a + 1], c_g+8[a + 1])
  float* cpk = reinterpret_cast<float*>(dyn);
  double* slots = reinterpret_cast<double*>(dyn + Cfg::CDYN);   // [warp][tile][4][32]
  __shared__ LoopShared<D, KP, T> sh;
  __shared__ double wred[NW][D];
  const float* c_sm = sh.c;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int k = sp.k;
  double* myslots = slots + (size_t)warp * (MT * 4 * 32);
  const float inv_tau = (float)sp.inv_tau_d, inv_k = 1.f / (float)k;
  loop_frame<D, KP, T, SQ>(mp, sh, [&](int precise, int b, int NB, long long m, const float* Wl, double* mine) {
    const long long n_set = (m + 7) / 8, step = (long long)NB * NW;
    // ---- packed centroids; of a collapsing layer minus their distance from centroid 0 ----
    for (int i = tid; i < KP * D; i += T) {
      const int j = i / D, a = i % D;
      float v = -c_sm[i];
      if (precise) v = j < k ? (float)((double)c_sm[a] - (double)c_sm[i]) : 0.f;
      cpk[(((j >> 4) * (D / 2) + (a >> 1)) * 8 + (j & 7)) * 4 + (a & 1) * 2 + ((j >> 3) & 1)] = v;
    }
#pragma unroll
    for (int q = 0; q < MT * 4; ++q) myslots[q * 32 + lane] = 0.0;
    __syncthreads();
    f2 acc[MT][2];
#pragma unroll
    for (int q = 0; q < MT; ++q) acc[q][0] = acc[q][1] = f2_pack(0.f, 0.f);
    float us[D];   // sum of the weights (increment form; lanes g = 0)
    double usd[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      us[a] = 0.f;
      usd[a] = 0.0;
    }
    auto spill = [&]() {
#pragma unroll
      for (int q = 0; q < MT; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float x, y;
          f2_unpack(acc[q][h], x, y);
          myslots[(q * 4 + h * 2) * 32 + lane] += (double)x;
          myslots[(q * 4 + h * 2 + 1) * 32 + lane] += (double)y;
          acc[q][h] = f2_pack(0.f, 0.f);
        }
#pragma unroll
      for (int a = 0; a < D; ++a) {
        usd[a] += (double)us[a];
        us[a] = 0.f;
      }
    };
    float c0[D];
#pragma unroll
    for (int a = 0; a < D; ++a) c0[a] = precise ? c_sm[a] : 0.f;
    // the two weights of this lane, and the coordinate that is its entry of the right operand
    float wn[2][D], bn[2];
    bool vn[2];
    auto fetch = [&](long long set) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const long long r = set * 8 + t + 4 * i;
        vn[i] = r < m;
        const long long rr = vn[i] ? r : 0;
        const float4 x = __ldg(reinterpret_cast<const float4*>(Wl) + rr);
        wn[i][0] = x.x; wn[i][1] = x.y; wn[i][2] = x.z; wn[i][3] = x.w;
        bn[i] = (g >= 1 && g <= D) ? __ldg(Wl + rr * D + (g - 1)) : 1.f;   // (column g of the operand: 1, then the coordinates)
      }
    };
    auto load_c = [&](int q, f2 (&c)[D]) {
#pragma unroll
      for (int h = 0; h < D / 2; ++h) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(cpk + ((q * (D / 2) + h) * 8 + g) * 4);
        c[2 * h] = x.x;
        c[2 * h + 1] = x.y;
      }
    };
    // the products of one set: e[tile][weight] against b
    auto products = [&](f2 (&e)[MT][2], const float (&bv)[2]) {
      unsigned bh[2], bl[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float hi = tf32_rn(bv[i]), lo = tf32_rn(bv[i] - hi);
        bh[i] = __float_as_uint(g <= D ? hi : 0.f);
        bl[i] = __float_as_uint(g <= D ? lo : 0.f);
      }
#pragma unroll
      for (int q0 = 0; q0 < MT; q0 += QG) {
        unsigned hx[QG][4], lx[QG][4];   // (g, t), (g + 8, t), (g, t + 4), (g + 8, t + 4)
        float c[QG][4];
#pragma unroll
        for (int q = 0; q < QG; ++q)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float x, y, lo0, lo1;
            f2_unpack(e[q0 + q][i], x, y);
            const float h0 = tf32_cut(x), h1 = tf32_cut(y);
            lo0 = x - h0;
            lo1 = y - h1;
            hx[q][2 * i] = __float_as_uint(h0);
            hx[q][2 * i + 1] = __float_as_uint(h1);
            lx[q][2 * i] = __float_as_uint(lo0);
            lx[q][2 * i + 1] = __float_as_uint(lo1);
          }
#pragma unroll
        for (int q = 0; q < QG; ++q) mma_tf32_first(c[q], lx[q][0], lx[q][1], lx[q][2], lx[q][3], bh[0], bh[1]);
#pragma unroll
        for (int q = 0; q < QG; ++q) mma_tf32(c[q], hx[q][0], hx[q][1], hx[q][2], hx[q][3], bl[0], bl[1]);
#pragma unroll
        for (int q = 0; q < QG; ++q) mma_tf32(c[q], hx[q][0], hx[q][1], hx[q][2], hx[q][3], bh[0], bh[1]);
#pragma unroll
        for (int q = 0; q < QG; ++q) {
          acc[q0 + q][0] = f2_add(acc[q0 + q][0], f2_pack(c[q][0], c[q][1]));
          acc[q0 + q][1] = f2_add(acc[q0 + q][1], f2_pack(c[q][2], c[q][3]));
        }
      }
    };
    long long set = (long long)warp * NB + b;
    if (set < n_set) fetch(set);
    int since = 0;
    for (; set < n_set; set += step) {
      f2 w[2][D], e[MT][2];
      float bw[2];
      bool val[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        val[i] = vn[i];
        bw[i] = bn[i];
#pragma unroll
        for (int a = 0; a < D; ++a) w[i][a] = f2_pack(wn[i][a], wn[i][a]);
      }
      if (precise) {
        // Increment form (see delta_body): with u = w - c_0, delta_j = c_j - c_0 and q_j = D_ij^2 - D_i0^2, the logit
        // differences x_ij = -q_j / (tau (D_ij + D_i0)) and A_ij - 1/k = (t_ij - tbar_i) / (k (1 + tbar_i)),
        // t = exp(x) - 1, to fp32 accuracy relative to delta; the sums are those of A_ij - 1/k and (A_ij - 1/k) u_i.
        float d0sq[2] = {0.f, 0.f}, d0[2], ls[2] = {0.f, 0.f};
        f2 u2[2][D];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
          for (int a = 0; a < D; ++a) {
            const float u = wn[i][a] - c0[a];
            d0sq[i] = fmaf(u, u, d0sq[i]);
            u2[i][a] = f2_pack(2.f * u, 2.f * u);
            if (g == 0 && val[i]) us[a] += wn[i][a];
          }
          d0[i] = sqrt_approx(d0sq[i]);
          float c0g = 0.f;
#pragma unroll
          for (int a = 0; a < D; ++a)
            if (g == a + 1) c0g = c0[a];
          bw[i] -= c0g;
          if (!val[i]) bw[i] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < MT; ++q) {
          f2 c[D];
          load_c(q, c);   // -delta
          f2 dl2 = f2_mul(c[0], c[0]);
#pragma unroll
          for (int a = 1; a < D; ++a) dl2 = f2_fma(c[a], c[a], dl2);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            f2 qq = dl2;
#pragma unroll
            for (int a = 0; a < D; ++a) qq = f2_fma(c[a], u2[i][a], qq);
            float x, y;
            f2_unpack(qq, x, y);
            const float dx = sqrt_approx(fmaxf(d0sq[i] + x, 0.f)), dy = sqrt_approx(fmaxf(d0sq[i] + y, 0.f));
            x = expm1_small(-x * inv_tau * rcp_approx(fmaxf(dx + d0[i], 1e-30f)));
            y = expm1_small(-y * inv_tau * rcp_approx(fmaxf(dy + d0[i], 1e-30f)));
            e[q][i] = f2_pack(x, y);
            ls[i] += x + y;    // (a padding centroid has delta = 0: it adds nothing)
          }
        }
        if (set + step < n_set) fetch(set + step);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float tbar = mml_sum(ls[i]) * inv_k, rr = inv_k * rcp_approx(1.f + tbar), ntr = -tbar * rr;
          const f2 r2 = f2_pack(rr, rr), n2 = f2_pack(ntr, ntr);
#pragma unroll
          for (int q = 0; q < MT; ++q) e[q][i] = f2_fma(e[q][i], r2, n2);
        }
        products(e, bw);
      } else {
        float mn[2] = {3.0e38f, 3.0e38f};
#pragma unroll
        for (int q0 = 0; q0 < MT; q0 += QD) {
          f2 c[QD][D], sq[QD][2];
#pragma unroll
          for (int q = 0; q < QD; ++q) load_c(q0 + q, c[q]);
#pragma unroll
          for (int a = 0; a < D; ++a) {
            f2 d[QD][2];
#pragma unroll
            for (int q = 0; q < QD; ++q)
#pragma unroll
              for (int i = 0; i < 2; ++i) d[q][i] = f2_add(w[i][a], c[q][a]);
#pragma unroll
            for (int q = 0; q < QD; ++q)
#pragma unroll
              for (int i = 0; i < 2; ++i) sq[q][i] = a == 0 ? f2_mul(d[q][i], d[q][i]) : f2_fma(d[q][i], d[q][i], sq[q][i]);
          }
#pragma unroll
          for (int q = 0; q < QD; ++q)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              float x, y;
              f2_unpack(sq[q][i], x, y);
              if constexpr (!SQ) {
                x = sqrt_approx(x);
                y = sqrt_approx(y);
              }
              mn[i] = min3(mn[i], x, y);
              e[q0 + q][i] = f2_pack(x, y);
            }
        }
        if (set + step < n_set) fetch(set + step);
        float mr[2];
        f2 sum[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mr[i] = mml_min(mn[i]) * sp.scale;
          sum[i][0] = sum[i][1] = f2_pack(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < MT; ++q)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float x, y;
            f2_unpack(e[q][i], x, y);
            x = fmaf(-sp.scale, x, mr[i]);
            y = fmaf(-sp.scale, y, mr[i]);
            e[q][i] = f2_pack(ex2_approx(x), ex2_approx(y));
            sum[i][q & 1] = f2_add(sum[i][q & 1], e[q][i]);
          }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float x, y;
          f2_unpack(f2_add(sum[i][0], sum[i][1]), x, y);
          const float rr = rcp_approx(mml_sum(x + y));
          bw[i] = val[i] ? rr * bw[i] : 0.f;
        }
        products(e, bw);
      }
      if (++since == MML_SPILL) {
        spill();
        since = 0;
      }
    }
    spill();
    // ---- this block's partial: warps in index order ----
#pragma unroll
    for (int a = 0; a < D; ++a) {
      double v = g == 0 ? usd[a] : 0.0;
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      if (lane == 0) wred[warp][a] = v;
    }
    __syncthreads();
    // entry (q, h, lane): centroid 16 q + g + 8 (h / 2), column 2 t + h % 2
    for (int x = tid; x < KP * NA; x += T) {
      const int j = x / NA, c = x % NA;
      const double* o = slots + ((j >> 4) * 4 + ((j >> 3) & 1) * 2 + (c & 1)) * 32 + (j & 7) * 4 + (c >> 1);
      double v = 0.0;
#pragma unroll
      for (int wv = 0; wv < NW; ++wv) v += o[(size_t)wv * (MT * 4 * 32)];
      __stcg(mine + x, v);
    }
    if (tid < D) {
      double v = 0.0;
#pragma unroll
      for (int wv = 0; wv < NW; ++wv) v += wred[wv][tid];
      __stcg(mine + KP * NA + tid, v);
    }
  });
}

// ---- the same loop with the sums on the CUDA cores: LPW lanes hold the centroids, KPL each, and take a weight together ----
template <int D, int KPL, int LPW>
struct GrpCfg {
  static constexpr int KP = KPL * LPW, NA = D + 1, T = 512, NW = T / 32;
  static constexpr int PLEN = KP * NA + D, NS = KPL * NA;
  static constexpr int UNROLL = D == 2 ? 2 : 1;  // weights in flight (m = 4 M, d = 4, k = 16: 68.5 against 76 us with 2; d = 2, k = 256: 694 against 680)
  static constexpr int CHUNK = 64;              // weights a thread adds up before its sums move to its slots
  static constexpr int DYN = (NS + D) * T * 4;  // slots: [NS + D][T]
};
template <int D, int KPL, int LPW, bool SQ>
__global__ void __launch_bounds__(GrpCfg<D, KPL, LPW>::T, 1) idkm_group_loop(const __grid_constant__ MmaLoopParams mp) {
  using Cfg = GrpCfg<D, KPL, LPW>;
  constexpr int T = Cfg::T, NW = Cfg::NW, NA = Cfg::NA, KP = Cfg::KP, NS = Cfg::NS, GB = T / LPW;
  const SmallLoopParams& sp = mp.s;
  extern __shared__ __align__(16) unsigned char dyn[];
  float* slots = reinterpret_cast<float*>(dyn);
  __shared__ LoopShared<D, KP, T> sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gl = lane % LPW, grp = tid / LPW;
  const int k = sp.k;
  const float inv_tau = (float)sp.inv_tau_d, inv_k = 1.f / (float)k;
  loop_frame<D, KP, T, SQ>(mp, sh, [&](int precise, int b, int NB, long long m, const float* Wl, double* mine) {
    float c[KPL][D], acc[KPL][NA], us[D];
#pragma unroll
    for (int t = 0; t < KPL; ++t) {
      const int j = gl * KPL + t;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        c[t][a] = sh.c[j * D + a];
        if (precise) c[t][a] = j < k ? (float)((double)sh.c[j * D + a] - (double)sh.c[a]) : 0.f;
      }
#pragma unroll
      for (int a = 0; a < NA; ++a) acc[t][a] = 0.f;
    }
#pragma unroll
    for (int a = 0; a < D; ++a) us[a] = 0.f;
    bool first = true;   // (the slots hold nothing yet)
    auto spill = [&]() {
#pragma unroll
      for (int t = 0; t < KPL; ++t)
#pragma unroll
        for (int a = 0; a < NA; ++a) {
          float* o = slots + (t * NA + a) * T + tid;
          *o = first ? acc[t][a] : *o + acc[t][a];
          acc[t][a] = 0.f;
        }
#pragma unroll
      for (int a = 0; a < D; ++a) {
        float* o = slots + (NS + a) * T + tid;
        *o = first ? us[a] : *o + us[a];
        us[a] = 0.f;
      }
      first = false;
    };
    const long long step = (long long)NB * GB;
    const int trips = (int)((m + step - 1) / step);
    long long r = (long long)b * GB + grp;
    float wn[D];
    auto fetch = [&](long long q) {
      const long long rr = q < m ? q : 0;
      if constexpr (D == 4) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(Wl) + rr);
        wn[0] = x.x; wn[1] = x.y; wn[2] = x.z; wn[3] = x.w;
      } else {
        const float2 x = __ldg(reinterpret_cast<const float2*>(Wl) + rr);
        wn[0] = x.x; wn[1] = x.y;
      }
    };
    fetch(r);
    int since = 0;
    if (!precise) {
#pragma unroll Cfg::UNROLL
      for (int i = 0; i < trips; ++i) {
        float w[D], e[KPL];
#pragma unroll
        for (int a = 0; a < D; ++a) w[a] = wn[a];
        const bool val = r < m;
        r += step;
        fetch(r);
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
          float sq = 0.f;
#pragma unroll
          for (int a = 0; a < D; ++a) {
            const float df = w[a] - c[t][a];
            sq = fmaf(df, df, sq);
          }
          e[t] = SQ ? sq : sqrt_approx(sq);
        }
        const float mref = group_min<LPW>(tree_reduce<KPL, 1>(e)) * sp.scale;
#pragma unroll
        for (int t = 0; t < KPL; ++t) e[t] = ex2_approx(fmaf(-sp.scale, e[t], mref));
        const float gsum = group_sum<LPW>(tree_reduce<KPL, 0>(e));   // (by all lanes, whether their weight exists or not)
        const float rr = val ? rcp_approx(gsum) : 0.f;
        float rw[D];
#pragma unroll
        for (int a = 0; a < D; ++a) rw[a] = rr * w[a];
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
          acc[t][0] = fmaf(e[t], rr, acc[t][0]);
#pragma unroll
          for (int a = 0; a < D; ++a) acc[t][1 + a] = fmaf(e[t], rw[a], acc[t][1 + a]);
        }
        if (++since == Cfg::CHUNK) {
          spill();
          since = 0;
        }
      }
    } else {
      // increment form (see the other kernel); c holds c_j - c_0
      float c0[D];
#pragma unroll
      for (int a = 0; a < D; ++a) c0[a] = sh.c[a];
#pragma unroll 1
      for (int i = 0; i < trips; ++i) {
        float u[D], e[KPL], d0sq = 0.f;
        const bool val = r < m;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          u[a] = wn[a] - c0[a];
          d0sq = fmaf(u[a], u[a], d0sq);
          if (val && gl == 0) us[a] += wn[a];
        }
        r += step;
        fetch(r);
        const float d0 = sqrt_approx(d0sq);
        float ls = 0.f;
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
          float q = 0.f;
#pragma unroll
          for (int a = 0; a < D; ++a) q = fmaf(c[t][a], c[t][a], q);
#pragma unroll
          for (int a = 0; a < D; ++a) q = fmaf(c[t][a], -2.f * u[a], q);          // D_ij^2 - D_i0^2
          const float dij = sqrt_approx(fmaxf(d0sq + q, 0.f));
          e[t] = expm1_small(-q * inv_tau * rcp_approx(fmaxf(dij + d0, 1e-30f)));   // (a padding centroid: 0)
          ls += e[t];
        }
        const float tbar = group_sum<LPW>(ls) * inv_k;
        const float rr = val ? inv_k * rcp_approx(1.f + tbar) : 0.f, ntr = -tbar * rr;
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
          const float aij = fmaf(e[t], rr, ntr);
          acc[t][0] += aij;
#pragma unroll
          for (int a = 0; a < D; ++a) acc[t][1 + a] = fmaf(aij, u[a], acc[t][1 + a]);
        }
        if (++since == Cfg::CHUNK) {
          spill();
          since = 0;
        }
      }
    }
    // ---- this block's partial: a warp takes a row of slots, a lane the threads of its own lane in all warps ----
    spill();
    __syncthreads();
    for (int o = warp; o < NS + D; o += NW) {
      double v = 0.0;
#pragma unroll
      for (int w = 0; w < NW; ++w) v += (double)slots[o * T + w * 32 + lane];
#pragma unroll
      for (int x = LPW; x < 32; x <<= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
      if (o < NS) {
        if (lane < LPW) __stcg(mine + gl * NS + o, v);
      } else if (lane == 0) {
        __stcg(mine + KP * NA + (o - NS), v);
      }
    }
  });
}

template <int D, int KPL, int LPW, bool SQ>
static cudaError_t launch_group_loop(const MmaLoopParams& p, int grid, cudaStream_t stream) {
  using Cfg = GrpCfg<D, KPL, LPW>;
  static PerDevice limit;
  const cudaError_t allowed = allow_smem(limit, idkm_group_loop<D, KPL, LPW, SQ>, Cfg::DYN);
  if (allowed != cudaSuccess) return allowed;
  void* args[1] = {const_cast<MmaLoopParams*>(&p)};
  return cudaLaunchCooperativeKernel((const void*)&idkm_group_loop<D, KPL, LPW, SQ>, dim3((unsigned)grid, 1, 1), dim3(Cfg::T, 1, 1), args,
                                     (size_t)Cfg::DYN, stream);
}
#define IDKM_GRP(D, KPL, LPW, SQ) { &launch_group_loop<D, KPL, LPW, SQ>, KPL * LPW, GrpCfg<D, KPL, LPW>::PLEN }

template <int MT, bool SQ>
static cudaError_t launch_mma_loop(const MmaLoopParams& p, int grid, cudaStream_t stream) {
  using Cfg = MmlCfg<MT>;
  static PerDevice limit;
  const cudaError_t allowed = allow_smem(limit, idkm_mma_loop<MT, SQ>, Cfg::DYN);
  if (allowed != cudaSuccess) return allowed;
  void* args[1] = {const_cast<MmaLoopParams*>(&p)};
  // cooperative launch: refused (instead of hanging at the first barrier) if the grid cannot be co-resident
  return cudaLaunchCooperativeKernel((const void*)&idkm_mma_loop<MT, SQ>, dim3((unsigned)grid, 1, 1), dim3(Cfg::T, 1, 1), args,
                                     (size_t)Cfg::DYN, stream);
}
#define IDKM_MML(MT, SQ) { &launch_mma_loop<MT, SQ>, MT * 16, MmlCfg<MT>::PLEN }

// Which kernel takes a codebook, by time an iteration at 4 K / 64 K / 1 M / 4 M weight-vectors in us (a launch per iteration
// and layout of the group-per-weight step before it in brackets):
//   d = 4, k = 16:  8 x 2 lanes 10.6 / 11.6 / 25 / 69, 16 x 1 10.8 / 12 / 26 / 72, matrix 8.4 / 10.5 / 42 / 140 (14 / 16 / 32 / 83)
//          k = 32:  8 x 4 11.4 / 13.4 / 42 / 131, 16 x 2 10.3 / 12.5 / 41 / 133, matrix 8.9 / 11.5 / 50 / 171 (17 / 18 / 45 / 132)
//          k = 64:  matrix 9.5 / 13.2 / 75 / 265, 8 x 8 12.6 / 15.8 / 74 / 258 (18 / 23 / 80 / 265)
//          k = 128: matrix 12.8 / 17.8 / 115 / 425, 16 x 8 15.3 / 20.7 / 141 / 526 (21 / 29 / 141 / 499)
//          k = 256: matrix 17.6 / 27 / 221 / 845, 8 x 32 17.7 / 28.6 / 254 / 976 (28 / 41 / 246 / 900)
//   d = 2, k = 32:  16 x 2 11.2 / 12.7 / 31 / 90, 8 x 4 9.1 / 10.8 / 32 / 101, matrix 9 / 11 / 45 / 150 (12 / 14 / 36 / 110)
//          k = 64:  16 x 4 11.7 / 14.5 / 52 / 172, 8 x 8 9.6 / 12.2 / 55 / 190, matrix 10 / 13 / 62 / 216 (12 / 17 / 62 / 206)
//          k = 128: 16 x 8 14.1 / 18.1 / 95 / 340, matrix 12.5 / 17.2 / 101 / 363 (15 / 21 / 106 / 375)
//          k = 256: 16 x 16 16.5 / 24.2 / 181 / 680, 8 x 32 13.4 / 22 / 195 / 749, matrix 15.7 / 24 / 199 / 764 (18 / 31 / 192 / 704)
// (a matrix instruction holds the fp32 pipe for 8 cycles -- mma and three packed multiply-adds: 13.7 cycles, alone 8.2 and
// 5.7 -- so at d = 2, where a pair has three sums instead of five, it does not pay)
#define IDKM_LOOP_ROW_2(SQ, LAST) { { nullptr, 0, 0 }, IDKM_GRP(2, 16, 2, SQ), IDKM_GRP(2, 16, 4, SQ), IDKM_GRP(2, 16, 8, SQ), LAST }
#define IDKM_LOOP_ROW_4(SQ) { IDKM_GRP(4, 8, 2, SQ), IDKM_GRP(4, 8, 4, SQ), IDKM_MML(4, SQ), IDKM_MML(8, SQ), IDKM_MML(16, SQ) }

}  // namespace idkm
