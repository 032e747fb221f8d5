// Algorithm 1's whole loop for scalar weights, without a pass over the weights per iteration.
//
// The weights do not change during the loop, so they are summarised once: every layer's value range is cut into coarse
// bins about tau / 6 wide, each with its count and the first four moments of its weights about the bin's centre, and
// lambda(w) -- a logistic function of 2 w / tau inside an interval between centroids -- is summed over a bin by its
// Taylor series (at that width the first dropped term is below 1e-6 of lambda at a bin's very edge, odd, and 1e-8 on
// average; the exponential of the direct path is an approximation to 2e-7).  Far from an interval's even point, where
// lambda or mu is below 2^-96, whole runs of bins are taken from running sums.  A bin that contains a centroid is split
// at it: the moments of the weights below the centroid are the prefix over the fine bins of the coarse bin plus the
// weights of the one fine bin the centroid lies in, which are looked at one by one.  For that the weights' places are
// grouped by fine bin (two bytes per weight).  Everything that is accumulated in an order that can vary is a sum of
// integers, so results are reproducible although the grouping uses atomic counters.
//
// What bounds it.  Building: the grouping pass stores two bytes per weight to scattered places, 67 cycles a warp store
// (110 us per 11.7 M weights on all SMs).  Iterating: the chain of one block a layer, and where the centroids' fine bins hold
// thousands of weights, counting these: up to 16 centroids (sc_iterate) 1.5 us for 4096 weights, k = 4, to 6.0 for 16 M, k = 16;
// more 4.0 (36864, k = 17) to 25 and 92 (16 M, k = 32 and 256).  Measured, loop with the summary against one that
// visits the pairs: 21 layers of a ResNet-18, k = 4, 50 iterations 312 against 1473 us; k = 8, tau = 5e-4, 30 iterations 359
// against 1268; 16 M weights, k = 16, 100 iterations 0.87 against 10.4 ms; 4096 weights, k = 4, tau = 0.05, 30 iterations 71
// against 112.
//
// Layers that bins do not suit -- tau below 1 / 5700 of the weights' range (1 / 2800 in layers beyond the eighth), which an outlier
// is enough for, or thousands of weights in one fine bin -- are evaluated weight by weight by all their blocks (sd_pass): without
// bins an iteration's time does not depend on where the weights lie.  m = 1 M, one weight at 1e5 standard deviations, an iteration
// at k = 4 / 16 / 64 / 256: 17 / 24 / 63 / 63 us; two values for 3/4 of the weights: 19 / 22 / 63.  (Loops over the pairs on such
// weights: 8 / 14 / 37 / 125 us, 16 M weights 27 / 73 / 395 / 1000 against 58 / 78 / 332 / 325.)
//
// Several blocks per layer build the summary (meetings at a bounded barrier), then one block per layer runs the
// iterations: one warp (or a few) per interval between centroids, the M-step by the first warps in fp64.
#include "idkm_scalar.cuh"

namespace idkm {

// Value range -> bins.  Index arithmetic is one fused multiply-add per weight, rounded once.
struct ScGrid {
  double hf, hc;     // widths of fine and coarse bins
  double ctr0;       // centre of coarse bin 0
  double inv_hc, iF; // 1 / hc, 1 / F
  float inv_hf;
  float lo, hi;      // value range, centroids are clamped to it for the choice of a bin
  int fshift, F;     // fine bins per coarse bin: F = 1 << fshift
  int base_f;        // index of the first fine bin
  int nc, nf;
  float eta;         // 2 hc / tau: range of the logistic's argument across a coarse bin
};
constexpr float SC_MAGIC = 12582912.f;   // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits
__device__ __forceinline__ int sc_round_index(float w, float inv_hf) {
  return __float_as_int(fmaf(w, inv_hf, SC_MAGIC)) - 0x4B400000;
}
__device__ __forceinline__ int sc_fine(const ScGrid& g, float w) { return sc_round_index(w, g.inv_hf) - g.base_f; }
// index and place (in 1 / SC_PSCALE of a fine bin, from its centre)
__device__ __forceinline__ int sc_fine_place(const ScGrid& g, float w, int& place) {
  const float f = fmaf(w, g.inv_hf, SC_MAGIC);
  place = __float2int_rn(fmaf(w, g.inv_hf, -(f - SC_MAGIC)) * (float)SC_PSCALE);
  return __float_as_int(f) - 0x4B400000 - g.base_f;
}
__device__ __forceinline__ double sc_center(const ScGrid& g, int c) { return fma((double)c, g.hc, g.ctr0); }

__device__ ScGrid sc_make_grid(float lo, float hi, double tau, long long m, int cap) {
  ScGrid g;
  if (!(lo <= hi)) lo = hi = 0.f;   // no weight besides zeros
  const double amax = fmax(fmax(fabs((double)lo), fabs((double)hi)), 1e-30);
  double range = (double)hi - (double)lo;
  if (!(range > amax * 1e-6)) range = amax * 1e-6;
  const double hmin = amax * (1.0 / 2097152.0);   // indices stay below 2^21 in magnitude
  double hc = 0.17 * tau;
  // (how wide the coarse bins get does not depend on the number of weights)
  const int most = cap;
  if (cap > SC_FINE_BIG) cap = SC_FINE_BIG;
  if (hc < range / (double)(cap - 8)) hc = range / (double)(cap - 8);
  if (hc > range) hc = range;
  if (hc < hmin) hc = hmin;
  // fine bins: about 64 weights each; 16 to a coarse bin (see sc_full) while they hold 8 weights; as many as the
  // workspace holds
  const long long nc0 = (long long)(range / hc) + 5;
  long long want = m / 64 < 512 ? 512 : m / 64;
  if (want < 16 * nc0) want = 16 * nc0 < m / 8 ? 16 * nc0 : (want < m / 8 ? m / 8 : want);
  if (want > most) want = most;
  int f = 0;
  while (f < 12 && hc / (double)(2 << f) >= hmin && (nc0 << (f + 1)) <= want) ++f;
  g.inv_hf = (float)((double)(1 << f) / hc);
  g.hf = 1.0 / (double)g.inv_hf;
  g.fshift = f;
  g.F = 1 << f;
  g.hc = g.hf * (double)g.F;
  g.inv_hc = 1.0 / g.hc;
  g.iF = 1.0 / (double)g.F;
  g.base_f = sc_round_index(lo, g.inv_hf) - 1;
  const int nfn = sc_round_index(hi, g.inv_hf) - g.base_f + 2;
  g.nc = (nfn + g.F - 1) >> f;
  g.nf = g.nc << f;
  g.ctr0 = ((double)g.base_f + 0.5 * (double)(g.F - 1)) * g.hf;
  g.lo = lo;
  g.hi = hi;
  g.eta = (float)(2.0 * g.hc / tau);
  return g;
}

// Barrier among the blocks of one layer: sync[0] arrivals (only grows), sync[1] error word.  Bounded wait.  `stay`: this
// block goes on afterwards (otherwise it only arrives).
__device__ __forceinline__ bool sc_team_barrier(unsigned int* sync, unsigned int target, long long spin_limit, int* s_ok, bool stay) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned int* vs = sync;
    int ok = 1;
    __threadfence();
    atomicAdd(&sync[0], 1u);
    if (stay) {
      const long long t0 = clock64();
      while ((int)(vs[0] - target) < 0) {
        if (vs[1] != 0u || clock64() - t0 > spin_limit) {
          atomicExch(&sync[1], 1u);
          ok = 0;
          break;
        }
      }
      if (vs[1] != 0u) ok = 0;
      __threadfence();
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// Integer powers of a place p (|p| <= 32767): p^2 / 2^14, p^3 / 2^29, p^4 / 2^44, each at most 2^16.
__device__ __forceinline__ void sc_powers(int p, int& p2, int& p3, int& p4) {
  p2 = (p * p + 8192) >> 14;
  p3 = (p2 * p + 16384) >> 15;
  p4 = (int)(((unsigned)p2 * (unsigned)p2 + 32768u) >> 16);
}
constexpr double SC_S1 = 1.0 / (double)SC_PSCALE;
constexpr double SC_S2 = 16384.0 * SC_S1 * SC_S1;
constexpr double SC_S3 = 536870912.0 * SC_S1 * SC_S1 * SC_S1;
constexpr double SC_S4 = 17592186044416.0 * SC_S1 * SC_S1 * SC_S1 * SC_S1;
constexpr int SC_CHUNK = 8192;   // elements whose 32-bit integer sums cannot overflow
// Which powers of the place matter: a fine bin is 1 / F of a coarse bin, so the fourth and third power of a place inside it
// change the interval's sums by less than 1e-8 from F = 64 on, and so does the square in the one bin that is split.  With
// fewer fine bins all four do: 3000 of 4096 weights in a quarter of one coarse bin, F = 8, five iterations from 16 centroids in a
// third of it, centroids against float64: 2e-6 with all powers, 3e-5 without the third and the fourth.
__device__ __forceinline__ bool sc_full(const ScGrid& g) { return g.F < 64; }

// Moments about the coarse bin's centre, in units of the coarse width, of n weights of fine bin kf (0 .. F - 1) whose
// integer sums of powers of the place are s1 .. s4.
__device__ __forceinline__ void sc_shift(const ScGrid& g, double x0, double n, double s1, double s2, double s3, double s4, double (&M)[4]) {
  const double iF = g.iF, iF2 = iF * iF;
  const double d1 = s1 * (SC_S1 * iF), d2 = s2 * (SC_S2 * iF2), d3 = s3 * (SC_S3 * iF2 * iF), d4 = s4 * (SC_S4 * iF2 * iF2);
  M[0] = fma(n, x0, d1);
  M[1] = fma(x0, fma(n, x0, 2.0 * d1), d2);
  M[2] = fma(x0, fma(x0, fma(n, x0, 3.0 * d1), 3.0 * d2), d3);
  M[3] = fma(x0, fma(x0, fma(x0, fma(n, x0, 4.0 * d1), 6.0 * d2), 4.0 * d3), d4);
}
// a fine bin's centre from its coarse bin's, in units of the coarse width
__device__ __forceinline__ double sc_fine_x0(const ScGrid& g, int f) { return ((double)(f & (g.F - 1)) - 0.5 * (double)(g.F - 1)) * g.iF; }

// Coarse records: running count and x sum up to every bin (doubles, nc + 1), then count and moments (floats).
struct ScRec {
  double *cn, *cx;
  float* r;      // [5][stride]
  int stride;
};

__device__ __forceinline__ ScRec sc_global_rec(const ScalarParams& sp, int layer, int cap) {
  ScRec r;
  r.cn = reinterpret_cast<double*>(sp.p.crec + (size_t)sp.fine_off[layer] * SC_REC_BYTES + (size_t)layer * 16);
  r.cx = r.cn + cap + 1;
  r.r = reinterpret_cast<float*>(r.cx + cap + 1);
  r.stride = cap;
  return r;
}

// What the iterations of one layer's block need besides the shared struct.
struct ScLayer {
  const unsigned short* grouped;   // all layers' (16-byte aligned); this layer's weights start at element row0
  long long row0, total;   // ... of `total` in all layers
  const unsigned int* fstart;
  const double* frec;   // [nf][4]: moments of the weights of earlier fine bins of the coarse bin
  ScRec rec;
  int k, twl, wl, lpi;  // 2^twl warps (or lpi lanes) share an interval, 2^wl warps the fine bin of a centroid
  double tau, inv_tau;
  double zone;          // half-width of the zone: SC_ZONE / slope
  float slope;          // 2 log2(e) / tau
};

constexpr int SC_PARTS = 768;   // (centroid, slot) pairs: a slot per warp of an interval and two for its ends
constexpr int SI_K = 16;        // up to this many centroids the iterations are sc_iterate's
constexpr int SI_SLOTS = 52;    // (interval, slot) pairs there
constexpr int SC_BELOW = 272;   // (centroid, warp) pairs of the scan of the centroids' fine bins
struct ScShared {
  ScGrid g;
  ScLayer ly;              // (copy for the functions that are not inlined)
  int ok, bad, flag, steps, done, iters, dead, status;
  // what the evaluations without bins need (here, so that it does not live in registers in the others)
  unsigned int meet;       // barriers of the layer's blocks so far
  const float* W;          // the layer's weights, and this block's share
  long long r0, r1;
  float res;
  long long n0;            // weights that are exactly zero (kept out of the bins)
  float v[257];            // sorted centroids
  int id[256];             // their indices
  float vn[256];
  int idn[256];
  int fb[256], pv[256];    // fine bin and place of every centroid
  double even[257];        // e_s of interval s = 1 .. k - 1
  double bs[SC_BELOW][5];  // twice the sums over a centroid's fine bin below it (sc_bin_below)
  double Ls[SC_PARTS][2];  // sums of lambda (and lambda x) over the interval right of a centroid, per slot
  double Ms[SC_PARTS][2];  // ... of mu over the interval left of it
  double Xs[SC_PARTS][2];  // ... of lambda mu over the interval right of it (last evaluation only)
  alignas(16) double ev[SI_SLOTS][4];  // sc_iterate: per (interval, slot) sums of lambda, lambda x, mu, mu x
  double cnew[256], cold[256];   // the last M-step, for the stop test
  int dead_j[256];
  double qs[256];
  double tmp[32];
  unsigned int scan[SC_WARPS + 1];
  double scan_x[SC_WARPS + 1];
};
constexpr int SC_SH_BYTES = (int)((sizeof(ScShared) + 255) / 256 * 256);
constexpr int SC_BIN_BYTES = (SC_FINE_MOST * 4 > SC_REC_SMEM * SC_REC_BYTES + 16) ? SC_FINE_MOST * 4 : SC_REC_SMEM * SC_REC_BYTES + 16;
// without bins (sd_pass): sums of every thread, of every warp, tables of the search
constexpr int SD_COLS = SC_WARPS * 257 * 4 * 8, SD_WSUM = 8448, SD_BYTES = SD_COLS + SD_WSUM + (512 + 2 * 257) * 4;
constexpr int SC_DYN = SC_SH_BYTES + (SC_BIN_BYTES > SD_BYTES ? SC_BIN_BYTES : SD_BYTES);
constexpr int SC_SMALL_NC = 512;       // layers of up to this many coarse bins leave room for their weights' places
constexpr int SC_SMALL_OFF = (SC_SMALL_NC * SC_REC_BYTES + 16 + 15) / 16 * 16;
static_assert(SC_DYN <= 227 * 1024, "shared memory of the loop kernel");

// exp(x) for x <= 0 in fp64: 2^n times the Taylor polynomial of degree 10 on |f ln 2| <= 0.3466 (remainder below 3e-13
// relative), evaluated by Estrin's scheme: half the latency of the library function, which is on the iteration's chain.
__device__ __forceinline__ double sc_exp(double x) {
  const double y = fmax(x * 1.4426950408889634, -1020.0);
  const double n = rint(y);
  const double t = (y - n) * 0.6931471805599453, t2 = t * t, t4 = t2 * t2;
  const double p01 = 1.0 + t, p23 = fma(t, 1.0 / 6.0, 0.5), p45 = fma(t, 1.0 / 120.0, 1.0 / 24.0);
  const double p67 = fma(t, 1.0 / 5040.0, 1.0 / 720.0), p89 = fma(t, 1.0 / 362880.0, 1.0 / 40320.0);
  const double q0 = fma(t2, p23, p01), q1 = fma(t2, p67, p45), q2 = fma(t2, 1.0 / 3628800.0, p89);
  const double r = fma(t4, fma(t4, q2, q1), q0);
  return r * __hiloint2double((1023 + (int)n) << 20, 0);
}
// 1 / x: fp32 seed and two Newton steps
__device__ __forceinline__ double sc_rcp(double x) {
  double r = (double)rcp_approx((float)x);
  r = r * fma(-x, r, 2.0);
  return r * fma(-x, r, 2.0);
}

// The recurrences over at most 32 centroids, both directions at once, by one warp.  cb[l], cf[l]: products of 2^l
// coefficients a_j going right from, resp. left to, this lane (zero where they run over the end).
template <int LOG>
struct ScScan {
  double cb[LOG > 0 ? LOG : 1], cf[LOG > 0 ? LOG : 1];
};
template <int NX, int LOG>
__device__ __forceinline__ void sc_scan_both(const ScScan<LOG>& c, double (&x)[NX] /* from the right */, double (&y)[NX] /* from the left */) {
#pragma unroll
  for (int l = 0; l < LOG; ++l) {
    double xs[NX], ys[NX];
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      xs[i] = __shfl_down_sync(0xffffffffu, x[i], 1 << l);
      ys[i] = __shfl_up_sync(0xffffffffu, y[i], 1 << l);
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      x[i] = fma(c.cb[l], xs[i], x[i]);
      y[i] = fma(c.cf[l], ys[i], y[i]);
    }
  }
}

// Where a centroid lies among the bins, and the even point of the interval to its right (own threads).
__device__ __forceinline__ void sc_place(ScShared& sh, const ScLayer& ly, int j, float vf, double v, double vx, double ratio) {
  if (j + 1 < ly.k) sh.even[j + 1] = 0.5 * (v + vx) - 0.5 * ly.tau * (double)logf((float)ratio);
  const ScGrid& g = sh.g;
  int place;
  const int fi = sc_fine_place(g, fminf(fmaxf(vf, g.lo), g.hi), place);
  // one beyond the ends of the scale where the centroid lies outside the weights' range
  if (vf > g.hi) place = 40000;
  if (vf < g.lo) place = -40000;
  sh.fb[j] = fi;
  sh.pv[j] = place;
}

// Interval tables of the sorted centroids: a_j, 1 / P_j, 1 / Q_j of this thread's centroid, e_s, bins.  One warp, k <= 32.
template <int LOG>
__device__ __forceinline__ void sc_tables_warp(ScShared& sh, const ScLayer& ly, float vf, ScScan<LOG>& sc, double& rP, double& rQ) {
  const int j = threadIdx.x, k = ly.k;
  const bool own = j < k;
  const double v = (double)vf, vx = (double)__shfl_down_sync(0xffffffffu, vf, 1);
  const double a = j + 1 < k ? sc_exp((v - vx) * ly.inv_tau) : 0.0;
  sc.cb[0] = a;
  const double al = __shfl_up_sync(0xffffffffu, a, 1);
  sc.cf[0] = (j > 0 && own) ? al : 0.0;
  double P = 1.0, Q = 1.0;
#pragma unroll
  for (int l = 0; l < LOG; ++l) {
    const double qs = __shfl_down_sync(0xffffffffu, Q, 1 << l), ps = __shfl_up_sync(0xffffffffu, P, 1 << l);
    Q = fma(sc.cb[l], qs, Q);
    P = fma(sc.cf[l], ps, P);
    if (l + 1 < LOG) {
      sc.cb[l + 1] = sc.cb[l] * __shfl_down_sync(0xffffffffu, sc.cb[l], 1 << l);
      sc.cf[l + 1] = sc.cf[l] * __shfl_up_sync(0xffffffffu, sc.cf[l], 1 << l);
    }
  }
  const double Qn = __shfl_down_sync(0xffffffffu, Q, 1);
  rP = own ? sc_rcp(P) : 0.0;
  rQ = own ? sc_rcp(Q) : 0.0;
  if (own) sc_place(sh, ly, j, vf, v, vx, Qn * rP);
}
// The same for up to 256 centroids, by the first kw warps.
__device__ __forceinline__ void sc_tables_block(ScShared& sh, const ScLayer& ly, double& a, double& ap, double& rP, double& rQ) {
  const int j = threadIdx.x, k = ly.k, kw = (k + 31) >> 5;
  const bool own = j < k;
  const double v = own ? (double)sh.v[j] : 0.0;
  const double vx = (own && j + 1 < k) ? (double)sh.v[j + 1] : v;
  a = (own && j + 1 < k) ? sc_exp((v - vx) * ly.inv_tau) : 0.0;
  ap = __shfl_up_sync(0xffffffffu, a, 1);
  if ((j & 31) == 0) ap = (own && j > 0) ? sc_exp(((double)sh.v[j - 1] - v) * ly.inv_tau) : 0.0;
  if (!own) ap = 0.0;
  double x[1] = {own ? 1.0 : 0.0}, y[1] = {own ? 1.0 : 0.0};
  lin_scan<1, true>(ap, x, k, sh.tmp);
  lin_scan<1, false>(a, y, k, sh.tmp);
  sc_sync(kw);
  if (own) sh.qs[j] = y[0];
  sc_sync(kw);
  rP = own ? sc_rcp(x[0]) : 0.0;
  rQ = own ? sc_rcp(y[0]) : 0.0;
  if (own) sc_place(sh, ly, j, sh.v[j], v, vx, j + 1 < k ? sh.qs[j + 1] * rP : 1.0);
}

// Sorts the k centroids in vn / idn into v / id (first kw warps; NaN sorts last).
__device__ __forceinline__ void sc_sort(ScShared& sh, int k) {
  const int j = threadIdx.x, kw = (k + 31) >> 5;
  if (j < k) {
    const float x = sh.vn[j];
    const float key = (x == x) ? x : __int_as_float(0x7f800000);
    int r = 0;
    for (int i = 0; i < k; ++i) {
      const float y = sh.vn[i];
      const float ky = (y == y) ? y : __int_as_float(0x7f800000);
      r += (ky < key || (ky == key && i < j)) ? 1 : 0;
    }
    sh.v[r] = x;
    sh.id[r] = sh.idn[j];
  }
  sc_sync(kw);
}

// Eight places starting at element e (a multiple of 8); past the last of `total` elements zeros.
__device__ __forceinline__ uint4 sc_load8(const unsigned short* grouped, long long e, long long total) {
  if (e + 8 <= total) return *reinterpret_cast<const uint4*>(grouped + e);
  unsigned int x[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (e + i < total) x[i >> 1] |= (unsigned int)grouped[e + i] << (16 * (i & 1));
  return make_uint4(x[0], x[1], x[2], x[3]);
}

// A fine bin as a warp of the last evaluation sees it: up to SC_HEAD of its weights in registers.
constexpr int SC_HEAD = 248;
struct ScBin {
  int groups;             // of 32 weights in pe
  int pe[8];              // places (40001: no weight)
  long long t0, t1;       // the rest, as elements of `grouped` (t0 is a multiple of 8)
};
// (n warps share a bin: this one takes share `sub`, boundaries at multiples of 8)
__device__ __forceinline__ void sc_bin_load(const ScLayer& ly, unsigned int e0, unsigned int e1, int sub, int n, ScBin& bn) {
  const int lane = threadIdx.x & 31;
  long long A0 = ly.row0 + e0, A1 = ly.row0 + e1;
  if (n > 1) {
    const long long len = A1 - A0, b = A0, e = A1;
    A0 = sub == 0 ? b : ((b + len * sub / n) & ~7LL);
    A1 = sub == n - 1 ? e : ((b + len * (sub + 1) / n) & ~7LL);
    if (A0 < b) A0 = b;
    if (A1 < A0) A1 = A0;
  }
  long long h = (A0 + SC_HEAD) & ~7LL;
  if (h > A1) h = A1;
  bn.t0 = h;
  bn.t1 = A1;
  bn.groups = (int)(h - A0 + 31) >> 5;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long e = A0 + 32 * i + lane;
    bn.pe[i] = e < h ? (int)ly.grouped[e] - 32768 : 40001;
  }
}
// Sums over the bin's weights that lie below place pv, weights at pv itself counting half: twice the count and twice the
// sums of the powers of the place.  Result in every lane.  `full`: see sc_full.  This part: the weights that are not in
// registers, eight places per load, two loads in flight beyond the one being counted, in stretches whose 32-bit sums
// cannot overflow.
__device__ __noinline__ void sc_bin_below_rest(const ScLayer& ly, long long t0, long long t1, int pv, bool full, double* s) {
  const int lane = threadIdx.x & 31;
  for (long long tb = t0; tb < t1; tb += SC_CHUNK) {
    const long long te = tb + SC_CHUNK < t1 ? tb + SC_CHUNK : t1;
    int c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
    long long e = tb + 8 * lane;
    uint4 x = e < te ? sc_load8(ly.grouped, e, ly.total) : make_uint4(0u, 0u, 0u, 0u);
    uint4 x1 = e + 256 < te ? sc_load8(ly.grouped, e + 256, ly.total) : make_uint4(0u, 0u, 0u, 0u);
    for (; e < te; e += 256) {
      const uint4 x2 = e + 512 < te ? sc_load8(ly.grouped, e + 512, ly.total) : make_uint4(0u, 0u, 0u, 0u);
      const unsigned int xs[4] = {x.x, x.y, x.z, x.w};
      const int left = (int)(te - e);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int p = i < left ? (int)((i & 1) ? xs[i >> 1] >> 16 : xs[i >> 1] & 0xffffu) - 32768 : 40001;
        const int w = p < pv ? 2 : (p == pv ? 1 : 0);
        c0 += w;
        c1 += w ? w * p : 0;
        if (full && w) {
          int p2, p3, p4;
          sc_powers(p, p2, p3, p4);
          c2 += w * p2;
          c3 += w * p3;
          c4 += w * p4;
        }
      }
      x = x1;
      x1 = x2;
    }
    s[0] += (double)__reduce_add_sync(0xffffffffu, c0);
    s[1] += (double)__reduce_add_sync(0xffffffffu, c1);
    if (full) {
      s[2] += (double)__reduce_add_sync(0xffffffffu, c2);
      s[3] += (double)__reduce_add_sync(0xffffffffu, c3);
      s[4] += (double)__reduce_add_sync(0xffffffffu, c4);
    }
  }
}
__device__ __forceinline__ void sc_bin_below(const ScLayer& ly, const ScBin& bn, int pv, bool full, double (&s)[5]) {
  int lt = 0, eq = 0, s1 = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (i >= bn.groups) break;
    const int p = bn.pe[i];
    if (p < pv) {
      ++lt;
      s1 += p;
    }
    eq += p == pv ? 1 : 0;
  }
  s[0] = (double)__reduce_add_sync(0xffffffffu, 2 * lt + eq);
  s[1] = (double)__reduce_add_sync(0xffffffffu, 2 * s1 + eq * pv);
  s[2] = s[3] = s[4] = 0.0;
  if (full) {
    int q2 = 0, q3 = 0, q4 = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i >= bn.groups) break;
      const int p = bn.pe[i], w = p < pv ? 2 : (p == pv ? 1 : 0);
      int p2, p3, p4;
      sc_powers(w ? p : 0, p2, p3, p4);
      q2 += w * p2;
      q3 += w * p3;
      q4 += w * p4;
    }
    s[2] = (double)__reduce_add_sync(0xffffffffu, q2);
    s[3] = (double)__reduce_add_sync(0xffffffffu, q3);
    s[4] = (double)__reduce_add_sync(0xffffffffu, q4);
  }
  if (bn.t0 < bn.t1) {   // (through a copy: what is handed to a function by address would live in memory everywhere)
    double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    sc_bin_below_rest(ly, bn.t0, bn.t1, pv, full, t);
#pragma unroll
    for (int i = 0; i < 5; ++i) s[i] += t[i];
  }
}

struct ScCoef {   // Taylor coefficients of a bin: lambda, mu and phi = lambda mu at its centre and derivatives
  float lam, mu, phi, del, d3, d4;
};
__device__ __forceinline__ ScCoef sc_coef(float z) {
  ScCoef c;
  sc_lambda(z, c.lam, c.mu);
  c.phi = c.lam * c.mu;
  c.del = c.lam - c.mu;
  c.d3 = fmaf(-6.f, c.phi, 1.f);
  c.d4 = c.del * fmaf(-12.f, c.phi, 1.f);
  return c;
}
// Sums over n weights with moments m1 .. m4 about the bin centre, which lies at x0 from the origin of the x sums.
// (mu' = phi, mu'' = phi del, mu''' = phi d3, mu'''' = phi d4; lambda = 1 - mu)
template <bool EXTRA, typename T>
__device__ __forceinline__ void sc_bin_sums(const ScCoef& c, float eta, T n, T m1, T m2, T m3, T m4, double x0, double hc, double (&acc)[6]) {
  const float e2 = 0.5f * eta * eta, e3 = e2 * eta * (1.f / 3.f), e4 = e3 * eta * 0.25f;
  const T corr = (T)c.phi * ((T)eta * m1 + (T)(e2 * c.del) * m2 + (T)(e3 * c.d3) * m3 + (T)(e4 * c.d4) * m4);
  const T cort = (T)c.phi * ((T)eta * m2 + (T)(e2 * c.del) * m3 + (T)(e3 * c.d3) * m4);
  const double sl = (double)(n * (T)c.lam - corr), sm = (double)(n * (T)c.mu + corr);
  acc[0] += sl;
  acc[2] += sm;
  acc[1] += fma(x0, sl, hc * (double)((T)c.lam * m1 - cort));
  acc[3] += fma(x0, sm, hc * (double)((T)c.mu * m1 + cort));
  if (EXTRA) {
    const float d5 = fmaf(-12.f, c.phi, 1.f) * c.d3 - 12.f * c.phi * c.del * c.del;
    const T sp = (T)c.phi * (n + (T)(eta * c.del) * m1 + (T)(e2 * c.d3) * m2 + (T)(e3 * c.d4) * m3 + (T)(e4 * d5) * m4);
    const T tp = (T)c.phi * (m1 + (T)(eta * c.del) * m2 + (T)(e2 * c.d3) * m3 + (T)(e3 * c.d4) * m4);
    acc[4] += (double)sp;
    acc[5] += fma(x0, (double)sp, hc * (double)tp);
  }
}

constexpr double SC_ZONE = 96.0;   // |z| beyond which lambda resp. mu (below 2^-96) is taken as zero for whole bins

// The weights that are exactly zero; on a centroid half of them belong to either side.
__device__ __noinline__ void sc_zeros(const ScShared& sh, int s, double even, double v0, double* acc) {
  const float vl = sh.v[s - 1], vr = sh.v[s];
  const double share = (vl < 0.f && vr > 0.f) ? 1.0 : (((vl == 0.f && vr > 0.f) || (vl < 0.f && vr == 0.f)) ? 0.5 : 0.0);
  float lam, mu;
  sc_lambda((float)(-even * (double)sh.ly.slope), lam, mu);
  const double n = share * (double)sh.n0, nl = n * (double)lam, nm = n * (double)mu, nx = n * (double)(lam * mu);
  acc[0] += nl;
  acc[1] -= nl * v0;
  acc[2] += nm;
  acc[3] -= nm * v0;
  acc[4] += nx;
  acc[5] -= nx * v0;
}

// Stop test of the M-step before (Algorithm 1's rule), by one warp while the others evaluate.
__device__ __noinline__ void sc_stop_test(ScShared& sh, const ScalarParams& sp, int layer, int test) {
  const int lane = threadIdx.x & 31, k = sp.k;
  double num = 0.0, den = 0.0;
  int dead = 0;
  for (int j = lane; j < k; j += 32) {
    const double c = sh.cnew[j], d = c - sh.cold[j];
    num = fma(d, d, num);
    den = fma(c, c, den);
    dead += sh.dead_j[j];
  }
  const bool bad = __any_sync(0xffffffffu, dead < 0 || dead > 0x8000);
  dead = __reduce_add_sync(0xffffffffu, dead & 0x7fff);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
  }
  if (lane == 0) {
    const float res = sqrtf((float)(num / fmax(den, 1e-300)));
    sh.iters = test;
    sh.res = res;
    sh.dead = dead;
    if (test <= HIST_CAP && (int)blockIdx.x == sp.blk_first[layer]) sp.p.hist_fwd[(size_t)layer * HIST_CAP + test - 1] = res;
    if (bad) {
      sh.status = ST_NONFINITE;
      sh.done = test;
    } else if (sp.tol > 0.f && res < sp.tol) {
      sh.done = test;
      sh.status = ST_OK;
    } else if (sp.tol > 0.f && test >= sp.max_iter) {
      sh.status = ST_MAXITER;
    }
  }
  }

// First half of an evaluation: the weights of every centroid's fine bin below it.  Up to 16 centroids (the last evaluation only:
// the others are sc_iterate's): a warp (or two) each.  More: eight lanes each, eight places per load.
__device__ __forceinline__ void sc_scan_warps(ScShared& sh, const ScLayer& ly, bool full) {
  const int lane = threadIdx.x & 31, t = threadIdx.x >> 5;
  if (t >= ly.k << ly.wl) return;
  const int j = t >> ly.wl, sub = t & ((1 << ly.wl) - 1);
  const int f = sh.fb[j];
  ScBin bn;
  sc_bin_load(ly, ly.fstart[f], ly.fstart[f + 1], sub, 1 << ly.wl, bn);
  double s[5];
  sc_bin_below(sh.ly, bn, sh.pv[j], full, s);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 5; ++i) sh.bs[t][i] = s[i];
  }
}
__device__ __noinline__ void sc_scan_quarters(ScShared& sh, bool full) {
  const ScLayer& ly = sh.ly;
  const int ql = threadIdx.x & 7;
  const unsigned int qmask = 0xffu << (threadIdx.x & 24);
  const int k = ly.k;
  int j = threadIdx.x >> 3;
  long long A0 = 0, A1 = 0, B0 = 0, B1 = 0;
  auto range = [&](int i, long long& a0, long long& a1) {
    a0 = a1 = 0;
    if (i < k) {
      const int f = sh.fb[i];
      a0 = ly.row0 + ly.fstart[f];
      a1 = ly.row0 + ly.fstart[f + 1];
    }
  };
  auto load = [&](long long e, long long a1) { return e < a1 ? sc_load8(ly.grouped, e, ly.total) : make_uint4(0u, 0u, 0u, 0u); };
  range(j, A0, A1);
  uint4 x0 = load((A0 & ~7LL) + 8 * ql, A1), x1 = load((A0 & ~7LL) + 8 * ql + 64, A1);
  for (; j < k; j += SC_T / 8) {
    range(j + SC_T / 8, B0, B1);   // (the next centroid's bin: its first loads go out before this one is counted)
    const uint4 n0 = load((B0 & ~7LL) + 8 * ql, B1), n1 = load((B0 & ~7LL) + 8 * ql + 64, B1);
    const int pv = sh.pv[j];
    long long c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
    long long e = (A0 & ~7LL) + 8 * ql;
    while (e < A1) {
      int s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0;   // (eight places: no overflow)
      const unsigned int xs[4] = {x0.x, x0.y, x0.z, x0.w};
      const int lo = (int)(A0 - e), hi = (int)(A1 - e < 8 ? A1 - e : 8);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int p = (int)((q & 1) ? xs[q >> 1] >> 16 : xs[q >> 1] & 0xffffu) - 32768;
        const int w = (q >= lo && q < hi) ? (p < pv ? 2 : (p == pv ? 1 : 0)) : 0;
        s0 += w;
        s1 += w * p;
        if (full) {
          int p2, p3, p4;
          sc_powers(p, p2, p3, p4);
          s2 += w * p2;
          s3 += w * p3;
          s4 += w * p4;
        }
      }
      c0 += s0;
      c1 += s1;
      c2 += s2;
      c3 += s3;
      c4 += s4;
      e += 64;
      x0 = x1;
      x1 = load(e + 64, A1);
    }
    long long c[5] = {c0, c1, c2, c3, c4};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      if (i >= 2 && !full) break;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) c[i] += __shfl_xor_sync(qmask, c[i], o);
    }
    if (ql == 0) {
#pragma unroll
      for (int i = 0; i < 5; ++i) sh.bs[j][i] = (double)c[i];
    }
    A0 = B0;
    A1 = B1;
    x0 = n0;
    x1 = n1;
  }
}

// Second half: every interval's sums.  Its two ends by two neighbouring threads (the block's last ones), the whole bins
// between them by 2^twl warps; each leaves its share in a slot of Ls, Ms (and Xs).
template <bool EXTRA>
__device__ __forceinline__ void sc_sum_intervals(ScShared& sh, const ScLayer& ly, bool full) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const ScGrid& g = sh.g;
  const int k = ly.k, tw = 1 << ly.twl, slots = tw + 2;
  const double v0 = (double)sh.v[0];
  if (k == 1) {
    // one centroid: every weight counts on its left, with attention 1
    if (threadIdx.x == 0) {
      const double n = ly.rec.cn[g.nc] + (double)sh.n0;
      sh.Ms[0][0] = n;
      sh.Ms[0][1] = ly.rec.cx[g.nc] - v0 * n;
    }
    return;
  }
  // ---- the ends: two neighbouring threads per interval, counted from the block's last; a second set of threads (of the
  // warps before them, for few intervals) takes the runs of whole bins outside the zone, the outer intervals and zeros ----
  const int ew = (2 * (k - 1) + 31) & ~31;   // threads of one set, whole warps
  for (int base = 0; base < 2 * ew; base += SC_T) {
    const int e0 = base + SC_T - 1 - (int)threadIdx.x;
    if (e0 - (e0 & 31) >= 2 * ew) continue;
    const bool runs = e0 >= ew;
    const int e = runs ? e0 - ew : e0;                  // 2 (s - 1) + (0: right end, 1: left end)
    const bool mine = e < 2 * (k - 1), left = e & 1;
    const int s = mine ? (e >> 1) + 1 : 1, j = left ? s - 1 : s;
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int fl = sh.fb[s - 1], fr = sh.fb[s], cl = fl >> g.fshift, cr = fr >> g.fshift;
    const int f = left ? fl : fr, c = left ? cl : cr;
    const double even = sh.even[s], ctr = sc_center(g, c);
    if (mine) {
      // weights of the coarse bin below the centroid: earlier fine bins, and those of its own
      const double2 q0 = *reinterpret_cast<const double2*>(ly.frec + (size_t)f * 4);
      const double2 q1 = *reinterpret_cast<const double2*>(ly.frec + (size_t)f * 4 + 2);
      const double nb = ly.rec.cn[c];
      double b[5] = {sh.bs[j << ly.wl][0], sh.bs[j << ly.wl][1], 0.0, 0.0, 0.0};
      if (full) {
        b[2] = sh.bs[j << ly.wl][2];
        b[3] = sh.bs[j << ly.wl][3];
        b[4] = sh.bs[j << ly.wl][4];
      }
      if (ly.wl) {
#pragma unroll
        for (int i = 0; i < 5; ++i) b[i] += (full || i < 2) ? sh.bs[(j << 1) + 1][i] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < 5; ++i) b[i] *= 0.5;
      double M[4];
      sc_shift(g, sc_fine_x0(g, f), b[0], b[1], b[2], b[3], b[4], M);
      double n = b[0] + ((double)ly.fstart[f] - nb);
      M[0] += q0.x;
      M[1] += q0.y;
      M[2] += q1.x;
      M[3] += q1.y;
      if (!runs) {
        const ScCoef co = sc_coef((float)((ctr - even) * (double)ly.slope));
        if (left) {   // the piece above the left end: the whole bin (unless the right end lies in it) minus what is below
          const bool whole = cl != cr;
          n = (whole ? (double)ly.rec.r[cl] : 0.0) - n;
#pragma unroll
          for (int i = 0; i < 4; ++i) M[i] = (whole ? (double)ly.rec.r[(i + 1) * ly.rec.stride + cl] : 0.0) - M[i];
        }
        sc_bin_sums<EXTRA, double>(co, g.eta, n, M[0], M[1], M[2], M[3], ctr - v0, g.hc, acc);
      } else {
        if (left ? (s == 1) : (s == k - 1)) {
          // the outer interval beyond this end: every weight there, and the zeros
          double nn = n + nb, xx = fma(ctr, n, fma(g.hc, M[0], ly.rec.cx[c]));
          if (!left) {
            nn = ly.rec.cn[g.nc] - nn;
            xx = ly.rec.cx[g.nc] - xx;
          }
          if (sh.n0 > 0) {
            const float v = left ? sh.v[0] : -sh.v[k - 1];
            nn += (v > 0.f ? 1.0 : (v == 0.f ? 0.5 : 0.0)) * (double)sh.n0;
          }
          double* o = left ? sh.Ms[0] : sh.Ls[(k - 1) * slots];
          o[0] = nn;
          o[1] = xx - v0 * nn;
        }
        if (cr - cl >= 2) {
          // whole bins on this side of the zone: lambda = 1 left of it, mu = 1 right of it
          int lo = cl + 1, hi = cr;
          if (left) {
            const int z = __double2int_rd((even - ly.zone - g.ctr0) * g.inv_hc);
            hi = z < lo ? lo : (z < cr ? z : cr);
          } else {
            const int z = __double2int_ru((even + ly.zone - g.ctr0) * g.inv_hc) + 1;
            lo = z < lo ? lo : (z < cr ? z : cr);
          }
          const double nn = ly.rec.cn[hi] - ly.rec.cn[lo], xx = ly.rec.cx[hi] - ly.rec.cx[lo] - v0 * nn;
          acc[0] = left ? nn : 0.0;
          acc[1] = left ? xx : 0.0;
          acc[2] = left ? 0.0 : nn;
          acc[3] = left ? 0.0 : xx;
        }
        if (left && sh.n0 > 0) {
          double t6[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
          sc_zeros(sh, s, even, v0, t6);
#pragma unroll
          for (int i = 0; i < 6; ++i) acc[i] += t6[i];
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < (EXTRA ? 6 : 4); ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 1);
    if (mine && left) {
      const int q = tw + (runs ? 1 : 0);
      double *lo = sh.Ls[(s - 1) * slots + q], *mo = sh.Ms[s * slots + q], *xo = sh.Xs[(s - 1) * slots + q];
      lo[0] = acc[0];
      lo[1] = acc[1];
      mo[0] = acc[2];
      mo[1] = acc[3];
      if (EXTRA) {
        xo[0] = acc[4];
        xo[1] = acc[5];
      }
    }
  }
  // ---- whole bins between the ends, inside the zone where neither lambda nor mu vanishes ----
  // up to 16 intervals: 2^twl warps each; up to 32: half a warp; more: eight lanes (an interval holds few bins then)
  const int lpi = ly.lpi, per = lpi < 32 ? 32 / lpi : 1;
  for (int t0 = warp * per; t0 < (k - 1) << ly.twl; t0 += SC_WARPS * per) {
    const int t = t0 + lane / lpi;
    const bool on = t < (k - 1) << ly.twl;
    const int s = on ? (t >> ly.twl) + 1 : 1, sub = t & (tw - 1), l = lane & (lpi - 1);
    const int cl = sh.fb[s - 1] >> g.fshift, cr = sh.fb[s] >> g.fshift;
    const double even = sh.even[s];
    int b0 = __double2int_rd((even - ly.zone - g.ctr0) * g.inv_hc), b1 = __double2int_ru((even + ly.zone - g.ctr0) * g.inv_hc);
    if (b0 < cl + 1) b0 = cl + 1;
    if (b1 > cr - 1) b1 = cr - 1;
    if (!on) b1 = b0 - 1;
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = b0 + sub * 32 + l; b <= b1; b += lpi * tw) {
      const float n = ly.rec.r[b];
      const double ctr = sc_center(g, b);
      const ScCoef c = sc_coef((float)((ctr - even) * (double)ly.slope));
      sc_bin_sums<EXTRA, float>(c, g.eta, n, ly.rec.r[ly.rec.stride + b], ly.rec.r[2 * ly.rec.stride + b], ly.rec.r[3 * ly.rec.stride + b],
                                ly.rec.r[4 * ly.rec.stride + b], ctr - v0, g.hc, acc);
    }
    __syncwarp();
    double* lo = sh.Ls[(s - 1) * slots + sub];
    double* mo = sh.Ms[s * slots + sub];
    if (lpi == 32) {
      // four sums over the warp: the first two levels also deal the sums out, so that lanes 0, 8, 16, 24 end with one each
      const bool h4 = lane & 16, h3 = lane & 8;
      double p = h4 ? acc[2] : acc[0], q = h4 ? acc[3] : acc[1];
      p += __shfl_xor_sync(0xffffffffu, h4 ? acc[0] : acc[2], 16);
      q += __shfl_xor_sync(0xffffffffu, h4 ? acc[1] : acc[3], 16);
      double r = h3 ? q : p;
      r += __shfl_xor_sync(0xffffffffu, h3 ? p : q, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if ((lane & 7) == 0) (h4 ? mo : lo)[h3 ? 1 : 0] = r;
    } else {
      // the same within groups of at least eight lanes: lanes 0, 2, 4, 6 of a group end with one each
      const bool h2 = lane & 4, h1 = lane & 2;
      double p = h2 ? acc[2] : acc[0], q = h2 ? acc[3] : acc[1];
      p += __shfl_xor_sync(0xffffffffu, h2 ? acc[0] : acc[2], 4);
      q += __shfl_xor_sync(0xffffffffu, h2 ? acc[1] : acc[3], 4);
      double r = h1 ? q : p;
      r += __shfl_xor_sync(0xffffffffu, h1 ? p : q, 2);
      r += __shfl_xor_sync(0xffffffffu, r, 1);
      if (lpi == 16) r += __shfl_xor_sync(0xffffffffu, r, 8);
      if (on && (l & 1) == 0 && l < 8) (h2 ? mo : lo)[h1 ? 1 : 0] = r;
    }
    if (EXTRA) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (o < lpi) {
          acc[4] += __shfl_xor_sync(0xffffffffu, acc[4], o);
          acc[5] += __shfl_xor_sync(0xffffffffu, acc[5], o);
        }
      if (on && l == 0) {
        sh.Xs[(s - 1) * slots + sub][0] = acc[4];
        sh.Xs[(s - 1) * slots + sub][1] = acc[5];
      }
    }
  }
}

// Both halves; the last warp first runs the stop test of the M-step before (`test` = its number, 0: none).
template <bool EXTRA, bool WARPS>
__device__ __forceinline__ void sc_evaluate(ScShared& sh, const ScLayer& ly, const ScalarParams& sp, int layer, int test) {
  const bool full = sc_full(sh.g);
  if (test > 0 && threadIdx.x >= SC_T - 32) sc_stop_test(sh, sp, layer, test);
  if constexpr (WARPS) sc_scan_warps(sh, ly, full);
  else sc_scan_quarters(sh, full);
  __syncthreads();
  sc_sum_intervals<EXTRA>(sh, ly, full);
}

// Sums a centroid sees on one of its sides (all slots; entries without a task stay zero).
__device__ __forceinline__ void sc_gather(const double (*a)[2], int j, int twl, double& s0, double& s1) {
  const int slots = (1 << twl) + 2;
  s0 = s1 = 0.0;
#pragma unroll
  for (int q = 0; q < 6; ++q)
    if (q < slots) {
      s0 += a[j * slots + q][0];
      s1 += a[j * slots + q][1];
    }
}

// ---- layers whose bins would not pay: the sums of an evaluation from the weights themselves ----
// Where tau is far below the weights' range (bins as wide as the workspace allows are then too wide for the series, and
// places of 16 bits in them too coarse), or very many weights share a few values (the bin of a centroid is looked at weight by
// weight by one or two warps), every evaluation is a pass over the weights by all blocks of the layer.  A weight costs a search
// for its interval, an exponential and a reciprocal whatever the number of centroids, and four additions in shared memory, so
// the time does not depend on where the weights lie.
constexpr float SC_ETA_MAX = 0.35f;          // coarse bins of 0.17 tau and their rounding
constexpr unsigned int SC_CROWD = 4096;      // weights of a fine bin, besides 1 / 256 of the layer's
// Up to SD_OWN_K centroids every thread has fp32 sums of its own for every interval (as many threads take weights as there is
// room for); more have fp64 sums for every warp, to which the lanes that have weights of the same interval add one after the
// other, or, where few intervals have many, after a sum over the warp.  (m = 1 M, an iteration, own sums against the warp's:
// k = 64 58 against 85 us, k = 256 248 against 63.)
constexpr int SD_OWN_K = 100;
__device__ __forceinline__ int sd_threads(int k) {
  if (k > SD_OWN_K) return SC_T;
  const int t = (SD_COLS / (16 * (k + 1))) & ~31;
  return t > SC_T ? SC_T : t;
}
struct SdView {
  float4* own;        // [k + 1][threads]: by interval, sums of lambda, lambda x, mu, mu x
  double* wsum;       // [warps][4 (k + 1)] the same of a warp
  float *v, *te, *to; // sorted centroids, even points and what their rounding adds to the exponent
};
__device__ __forceinline__ SdView sd_view(int k) {
  extern __shared__ __align__(16) unsigned char smem_all[];
  SdView d;
  d.own = reinterpret_cast<float4*>(smem_all + SC_SH_BYTES);
  d.wsum = reinterpret_cast<double*>(smem_all + SC_SH_BYTES + (k <= SD_OWN_K ? SD_COLS : 0));
  d.v = reinterpret_cast<float*>(smem_all + SC_SH_BYTES + SD_COLS + SD_WSUM);
  d.te = d.v + 512;
  d.to = d.te + 257;
  return d;
}
// A warp's fp32 sums move to its fp64 sums and start at zero again.  A thread adds at most SD_FOLD terms to one between two such
// calls (a longer fp32 sum loses the many terms below half its last place, see PassCfg).  A lane takes an interval, or several
// lanes share one: few conversions a lane.  Each starts from a thread of its own: the lanes read different banks.
constexpr int SD_FOLD = 64;
__device__ __forceinline__ void sd_fold(const SdView& d, int T, int k, double* wsum, bool first) {
  const int tid = threadIdx.x, lane = tid & 31, n = k + 1, P = n < 32 ? 32 / n : 1, c = n < 32 ? lane / n : 0;
  __syncwarp();
  for (int s0 = 0; s0 < n; s0 += 32) {   // (one round where lanes share)
    const int s = n < 32 ? lane % n : s0 + lane, N = (31 - c) / P + 1;
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    if (c < P && s < n) {
      const float4* col = d.own + (size_t)s * T + (tid - lane) + c;
      int j = s % N;
#pragma unroll 4
      for (int i = 0; i < N; ++i) {
        const float4 y = col[P * j];
        x[0] += (double)y.x;
        x[1] += (double)y.y;
        x[2] += (double)y.z;
        x[3] += (double)y.w;
        j = j + 1 == N ? 0 : j + 1;
      }
    }
    double t[4] = {x[0], x[1], x[2], x[3]};
    for (int q = 1; q < P; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) t[i] += __shfl_sync(0xffffffffu, x[i], s + q * n);
    if (c == 0 && s < n)
#pragma unroll
      for (int i = 0; i < 4; ++i) wsum[s * 4 + i] = first ? t[i] : wsum[s * 4 + i] + t[i];
  }
  __syncwarp();
  for (int i = 0; i < n; ++i) d.own[(size_t)i * T + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
}
// MODE 0: sums of lambda and mu; 1: the same, a weight on a centroid counting half on either side (sub-gradient 0 of its
// distance); 2: of lambda mu in place of lambda.  x: from the interval's left centroid.
template <int MODE, bool OWN>
__device__ __noinline__ void sd_pass(const float* __restrict__ Wl, long long r0, long long r1, int k, float slope) {
  const SdView d = sd_view(k);
  const int tid = threadIdx.x, lane = tid & 31, T = OWN ? sd_threads(k) : SC_T;
  if (OWN && tid >= T) {   // (whole warps)
    __syncthreads();
    return;
  }
  double* wsum = d.wsum + (size_t)(tid >> 5) * 4 * (k + 1);
  if (OWN) {
    for (int s = 0; s <= k; ++s) d.own[(size_t)s * T + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    for (int e = lane; e < 4 * (k + 1); e += 32) wsum[e] = 0.0;
    __syncwarp();
  }
  int top = 1;
  while (2 * top <= k) top *= 2;
  // what a weight adds to its interval (outside the centroids lambda resp. mu is 1)
  auto terms = [&](int s, float w, float g) {
    const float x = w - d.v[s > 0 ? s - 1 : 0];
    float lam, mu;
    sc_lambda(fmaf(w - d.te[s], slope, d.to[s]), lam, mu);
    const bool in = s > 0 && s < k;
    if (MODE == 2) {
      lam = in ? g * lam * mu : 0.f;
      mu = 0.f;
    } else {
      lam = in ? g * lam : (s > 0 ? g : 0.f);
      mu = in ? g * mu : (s < k ? g : 0.f);
    }
    return make_float4(lam, lam * x, mu, mu * x);
  };
  auto add = [&](int s, const float4& y, bool real) {   // (by whole warps)
    if (OWN) {
      if (!real) return;
      float4* c = d.own + (size_t)s * T + tid;
      float4 x = *c;
      x.x += y.x;
      x.y += y.y;
      x.z += y.z;
      x.w += y.w;
      *c = x;
    } else {
      const unsigned int same = __match_any_sync(0xffffffffu, real ? s : -1);
      const int turn = real ? __popc(same & ((1u << lane) - 1u)) : -1;
      const int turns = __reduce_max_sync(0xffffffffu, turn);
      const unsigned int firsts = __ballot_sync(0xffffffffu, turn == 0);
      if (2 * __popc(firsts) <= turns) {
        for (unsigned int left = firsts; left; left &= left - 1) {
          const int lead = __ffs(left) - 1, sl = __shfl_sync(0xffffffffu, s, lead);
          const bool mine = real && s == sl;
          float x[4] = {mine ? y.x : 0.f, mine ? y.y : 0.f, mine ? y.z : 0.f, mine ? y.w : 0.f};
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], o);
          if (lane < 4) wsum[4 * sl + lane] += (double)(lane == 0 ? x[0] : (lane == 1 ? x[1] : (lane == 2 ? x[2] : x[3])));
        }
        __syncwarp();
        return;
      }
      double2* c = reinterpret_cast<double2*>(wsum + 4 * s);
      for (int t = 0; t <= turns; ++t) {
        if (t == turn) {
          double2 a = c[0], b = c[1];
          a.x += (double)y.x;
          a.y += (double)y.y;
          b.x += (double)y.z;
          b.y += (double)y.w;
          c[0] = a;
          c[1] = b;
        }
        __syncwarp();
      }
    }
  };
  constexpr int U = OWN ? 8 : 4;
  static_assert(SD_FOLD % U == 0, "");
  const long long step = (long long)T * U;
  long long r = r0 + tid;
  float wn[U];
  auto fetch = [&](long long q) {
#pragma unroll
    for (int i = 0; i < U; ++i) wn[i] = q + i * T < r1 ? __ldg(Wl + q + i * T) : 0.f;
  };
  fetch(r);
  bool first = true;
  int since = 0;
  for (long long q = r0; q < r1; q += step, r += step) {   // (the same trips for all threads)
    float w[U];
    float4 y[U];
    int s[U];
    bool real[U], on[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      w[i] = wn[i];
      s[i] = 0;
      real[i] = r + i * T < r1;
    }
    fetch(r + step);
    for (int h = top; h > 0; h >>= 1)
#pragma unroll
      for (int i = 0; i < U; ++i) s[i] += d.v[s[i] + h - 1] < w[i] ? h : 0;
#pragma unroll
    for (int i = 0; i < U; ++i) {
      on[i] = MODE > 0 && real[i] && s[i] < k && d.v[s[i] < k ? s[i] : 0] == w[i];
      y[i] = terms(s[i], w[i], on[i] ? 0.5f : 1.f);
    }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      add(s[i], y[i], real[i]);
      if (MODE > 0 && __any_sync(0xffffffffu, on[i])) {
        int s2 = s[i];
        while (on[i] && s2 < k && d.v[s2] == w[i]) ++s2;
        add(s2, terms(s2, w[i], 0.5f), on[i]);
      }
    }
    if (OWN && (since += U) == SD_FOLD) {
      sd_fold(d, T, k, wsum, first);
      first = false;
      since = 0;
    }
  }
  if (OWN && (first || since > 0)) sd_fold(d, T, k, wsum, first);
  __syncthreads();
}
// One evaluation, by all threads of a block of the layer.  A block that is the layer's only one leaves the sums where the M-step
// looks for them; several leave a row of SD_SUMS each: 4 (k + 1) by interval and kind, then 2 (k + 1) of lambda mu.
__device__ __forceinline__ void sd_place(ScShared& sh, int k, int o, double x) {
  const int n = 4 * (k + 1);
  if (o < n) {
    const int s = o >> 2, c = o & 3;   // interval s: lambda for the centroid on its left, mu for the one on its right
    if (c < 2) {
      if (s > 0) sh.Ls[(s - 1) * 3][c] = x;
    } else if (s < k) {
      sh.Ms[s * 3][c - 2] = x;
    }
  } else {
    const int s = (o - n) >> 1;
    if (s > 0) sh.Xs[(s - 1) * 3][o & 1] = x;
  }
}
template <int MODE>
__device__ __forceinline__ void sd_one(ScShared& sh, int k, float slope, double* row) {
  if (k <= SD_OWN_K) sd_pass<MODE, true>(sh.W, sh.r0, sh.r1, k, slope);
  else sd_pass<MODE, false>(sh.W, sh.r0, sh.r1, k, slope);
  const SdView d = sd_view(k);
  const int n4 = 4 * (k + 1), warps = sd_threads(k) / 32;
  for (int i = threadIdx.x; i < (MODE == 2 ? n4 / 2 : n4); i += SC_T) {
    const int e = MODE == 2 ? (i >> 1) * 4 + (i & 1) : i, o = MODE == 2 ? n4 + i : i;
    double s[2] = {0.0, 0.0};
#pragma unroll
    for (int w = 0; w < SC_WARPS; ++w) s[w & 1] += w < warps ? d.wsum[(size_t)w * n4 + e] : 0.0;
    if (row) __stcg(row + o, s[0] + s[1]);
    else sd_place(sh, k, o, s[0] + s[1]);
  }
  __syncthreads();
}
__device__ __forceinline__ void sd_evaluate(ScShared& sh, int k, float slope, bool last, double* row) {
  if (!last) {
    sd_one<0>(sh, k, slope, row);
  } else {
    sd_one<1>(sh, k, slope, row);
    sd_one<2>(sh, k, slope, row);
  }
}
// Sums of all blocks of the layer, which all call (the last warp runs the stop test of the M-step before first, as in
// sc_evaluate), in the same order in every one of them: slot 0 of Ls, Ms (and, in the last evaluation, Xs); x sums from v_0.  Few
// rows: every block adds them all up, and the next evaluation's go to a second buffer.  Many: it adds up its share of the sums, and
// reads the others' after a second barrier.
constexpr long long SD_ONE_STAGE = 1 << 20;   // doubles that all blocks together may read (8 MB)
__device__ __noinline__ bool sd_sums(ScShared& sh, const ScalarParams& sp, int layer, bool last, int test) {
  const SdView d = sd_view(sp.k);
  if (test > 0 && threadIdx.x >= SC_T - 32) sc_stop_test(sh, sp, layer, test);
  const int tid = threadIdx.x, k = sp.k, NB = sp.blk_first[layer + 1] - sp.blk_first[layer], b = (int)blockIdx.x - sp.blk_first[layer];
  const bool alone = NB == 1 && sp.missing_arrivals == 0;
  const float slope = sh.ly.slope;
  const unsigned int meet = sh.meet;
  for (int i = tid; i < 512; i += SC_T) d.v[i] = i < k ? sh.v[i] : __int_as_float(0x7f800000);
  for (int i = tid; i <= k; i += SC_T) {
    const double even = i > 0 && i < k ? sh.even[i] : 0.0;
    const float e = (float)even;
    d.te[i] = e;
    d.to[i] = (float)(((double)e - even) * (double)slope);
  }
  __syncthreads();
  if (alone) {
    sd_evaluate(sh, k, slope, last, nullptr);
  } else {
    const int R = SD_SUMS(k), n = last ? R : 4 * (k + 1);
    const bool one_stage = k <= SD_TWO_ROWS_K && (long long)NB * NB * 4 * k <= SD_ONE_STAGE;
    const unsigned int arrivals = (unsigned int)(NB + sp.missing_arrivals);
    unsigned int* sync = sp.p.sync + (size_t)layer * SC_SYNC_WORDS;
    // rows: [blocks][R], then (one stage) as many again, or the layers' totals, [layers][R]
    const size_t all = (size_t)gridDim.x * R;
    double* rows = sp.p.gpart + (size_t)sp.blk_first[layer] * R + ((one_stage && (meet & 1u)) ? all : 0);
    sd_evaluate(sh, k, slope, last, rows + (size_t)b * R);
    if (!sc_team_barrier(sync, (meet + 1) * arrivals, sp.spin_limit, &sh.ok, true)) return false;
    const double* from = rows;
    int n_rows = NB;
    if (!one_stage) {
      double* tot = sp.p.gpart + all + (size_t)layer * R;
      const int o0 = (int)((long long)n * b / NB), o1 = (int)((long long)n * (b + 1) / NB);
      for (int o = o0 + (tid >> 5); o < o1; o += SC_WARPS) {
        double s = 0.0;
        for (int q = tid & 31; q < NB; q += 32) s += __ldcg(rows + (size_t)q * R + o);
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
        if ((tid & 31) == 0) __stcg(tot + o, s);
      }
      if (!sc_team_barrier(sync, (meet + 2) * arrivals, sp.spin_limit, &sh.ok, true)) return false;
      from = tot;
      n_rows = 1;
    }
    if (tid == 0) sh.meet = meet + (one_stage ? 1u : 2u);   // (read again after the next barriers of the block)
    // few sums: several threads each
    const int per = (n >= SC_T || n_rows == 1) ? 1 : SC_T / n;
    double* part = reinterpret_cast<double*>(d.own);   // (what it holds has been read)
    for (int o = tid; o < n * per; o += SC_T) {
      const int e = o % n, c = o / n;
      double s = 0.0;
#pragma unroll 8
      for (int q = c; q < n_rows; q += per) s += __ldcg(from + (size_t)q * R + e);
      if (per == 1) sd_place(sh, k, e, s);
      else part[o] = s;
    }
    __syncthreads();
    if (per > 1 && tid < n) {
      double s = 0.0;
      for (int c = 0; c < per; ++c) s += part[c * n + tid];
      sd_place(sh, k, tid, s);
    }
    __syncthreads();
  }
  for (int j = tid; j < k; j += SC_T) {
    const double right = (double)sh.v[j] - (double)sh.v[0], left = j > 0 ? (double)sh.v[j - 1] - (double)sh.v[0] : 0.0;
    sh.Ls[j * 3][1] = fma(right, sh.Ls[j * 3][0], sh.Ls[j * 3][1]);
    sh.Ms[j * 3][1] = fma(left, sh.Ms[j * 3][0], sh.Ms[j * 3][1]);
    if (last) sh.Xs[j * 3][1] = fma(right, sh.Xs[j * 3][0], sh.Xs[j * 3][1]);
  }
  __syncthreads();
  return true;
}

// ---- the iterations of up to SI_K centroids ----
// What bounds an iteration is the latency of its chain, instruction by instruction.  So its parts overlap: the first warp takes
// the M-step and publishes the centroids (meeting B1), then the even points and places (B2); a warp per centroid counts its
// fine bin between the two and afterwards takes the ends of the two intervals the centroid borders; other warps have the
// whole bins of an interval; at the third meeting (A) the first warp has all sums.  What a warp does is the same in every
// iteration, and a centroid's fine bin (up to SI_HEAD of its places, and its record) stays in its warp's registers, unless the
// warp has two centroids (16 of them).  Nothing in the loop may live in local memory: with the shared memory the block takes the L1 cache holds none of it, and every access
// is a trip to L2; and a load whose value is used before the next one is issued is one more such trip.  Cycles an iteration, in
// brackets the loop in which the whole block goes through counts, ends and M-step one after the other: 4096 weights, k = 4 3000
// (5500); 36864, k = 8 3800 (6700), k = 15 and 16 5400 and 5600; 2.4 M, k = 4 3600 (8000), k = 8 at tau = 5e-4 6900; 16 M, k = 4
// 6400, k = 16 11800 (24000 with half as many fine bins): there the centroids' bins hold 2000 weights and more.  Under ncu 36864
// weights, k = 16: issue slots 36 % busy, a warp waits at the meetings for 2.5 cycles of every instruction issued, for fixed
// latencies 2.1, for shared memory 1.5; no access to local memory.
constexpr int SI_WORDS = 8, SI_HEAD = 64 * SI_WORDS;
constexpr int SI_A = 2, SI_B1 = 3, SI_B2 = 4;   // hardware barriers
__device__ __forceinline__ void si_arrive(int id) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(SC_T) : "memory"); }
__device__ __forceinline__ void si_meet(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(SC_T) : "memory"); }
// (interval, slot) pairs of an interval: warps that share its whole bins, then its left and its right end
template <int LOG>
__host__ __device__ constexpr int si_slots() { return LOG <= 2 ? 5 : (LOG == 3 ? 4 : 3); }

struct SiBin {
  int f;                      // fine bin, -1: none
  unsigned int e0, e1;        // its elements
  unsigned int w[SI_WORDS];   // 64 places each, two a lane; 0 (which no weight's place is) where there is none
  double m[4];                // moments of the weights of earlier fine bins of the coarse bin
};
// (places start at a multiple of 8 elements of `grouped`)
__device__ __forceinline__ long long si_base(const ScLayer& ly, const SiBin& bn) { return (ly.row0 + bn.e0) & ~7LL; }
template <int N>
__device__ __forceinline__ void si_words(const ScLayer& ly, long long base, int lo, int hi, SiBin& bn) {
  const int e0 = 2 * (threadIdx.x & 31);
  const unsigned int* g = reinterpret_cast<const unsigned int*>(ly.grouped + base) + (e0 >> 1);
  const bool pairs = base + hi + 1 <= ly.total;   // (the last element of all may have no partner)
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int e = 64 * i + e0;
    bn.w[i] = e + (pairs ? 0 : 1) < hi ? g[32 * i] : 0u;
  }
  if (!pairs && ((hi - 1) & 1) == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (64 * i + e0 == hi - 1) bn.w[i] = (unsigned int)ly.grouped[base + hi - 1];
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int e = 64 * i + e0;
    bn.w[i] &= (e >= lo && e < hi ? 0xffffu : 0u) | (e + 1 >= lo && e + 1 < hi ? 0xffff0000u : 0u);
  }
}
__device__ __forceinline__ void si_bin_load(const ScLayer& ly, int f, SiBin& bn) {
  bn.f = f;
  bn.e0 = ly.fstart[f];
  bn.e1 = ly.fstart[f + 1];
  const double2 r0 = reinterpret_cast<const double2*>(ly.frec + (size_t)f * 4)[0], r1 = reinterpret_cast<const double2*>(ly.frec + (size_t)f * 4)[1];
  const long long base = si_base(ly, bn);
  const int lo = (int)(ly.row0 + bn.e0 - base), n = lo + (int)(bn.e1 - bn.e0), hi = n < SI_HEAD ? n : SI_HEAD;
  // all loads first, then what is made of them
  if (hi > 256) si_words<SI_WORDS>(ly, base, lo, hi, bn);
  else if (hi > 64) si_words<4>(ly, base, lo, hi, bn);
  else si_words<1>(ly, base, lo, hi, bn);
  bn.m[0] = r0.x;
  bn.m[1] = r0.y;
  bn.m[2] = r1.x;
  bn.m[3] = r1.y;
}
// Sums over n places p (from 1; 0: none) that lie below pv, those at it counting half, without a comparison: with S(x) the sum
// of min(p, x), S(x) - S(x - 1) places are at x or beyond.  Two places per instruction.  Powers (`full`): of min(p, pv), those
// beyond taken off again in si_total.
struct SiSum {
  unsigned int a, b, c;   // S(pv), S(pv + 1), S(pv - 1)
  int q2, q3, q4;
};
struct SiCut {
  unsigned int a, b, c;   // pv, pv + 1, pv - 1 in both halves
  bool none;              // below the scale
};
__device__ __forceinline__ SiCut si_cut(int pv) {
  // beyond the ends of the scale: below everything the result is set to zero, above everything the three sums are equal
  const unsigned int a = (unsigned int)(pv < 1 ? 1 : (pv > 65535 ? 65535 : pv)), b = a < 65535u ? a + 1u : a, c = pv > 65535 ? a : a - 1u;
  SiCut t;
  t.a = a * 0x10001u;
  t.b = b * 0x10001u;
  t.c = c * 0x10001u;
  t.none = pv < 1;
  return t;
}
__device__ __forceinline__ void si_add(unsigned int x, const SiCut& t, bool full, SiSum& s) {
  const unsigned int y = __vminu2(x, t.a);
  s.a = __dp2a_lo(y, 0x0101u, s.a);
  s.b = __dp2a_lo(__vminu2(x, t.b), 0x0101u, s.b);
  s.c = __dp2a_lo(__vminu2(x, t.c), 0x0101u, s.c);
  if (full) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int u = (int)(i ? y >> 16 : y & 0xffffu), p = u > 0 ? u - 32768 : 0;
      int p2, p3, p4;
      sc_powers(p, p2, p3, p4);
      s.q2 += p2;
      s.q3 += p3;
      s.q4 += p4;
    }
  }
}
// Over the warp, n places in all (fewer than SC_CHUNK + 1024): twice the count and sums of powers.
__device__ __forceinline__ void si_total(const SiSum& s, int n, const SiCut& t, bool full, double (&b)[5]) {
  const unsigned int a = __reduce_add_sync(0xffffffffu, s.a), up = __reduce_add_sync(0xffffffffu, s.b - s.a), at = __reduce_add_sync(0xffffffffu, s.a - s.c);
  const int lt2 = 2 * n - (int)(up + at), over = (int)(at + up);   // up: beyond pv, at: at it or beyond
  // twice the sum of the places below (the sum of all, those beyond counted as pv), those at pv half
  const int pv = (int)(t.a & 0xffffu);
  const long long p2 = 2LL * a - (long long)pv * over;
  b[0] += t.none ? 0.0 : (double)lt2;
  b[1] += t.none ? 0.0 : (double)(p2 - 32768LL * lt2);
  if (full) {
    int v2, v3, v4;
    sc_powers(pv - 32768, v2, v3, v4);
    const int q2 = __reduce_add_sync(0xffffffffu, s.q2), q3 = __reduce_add_sync(0xffffffffu, s.q3), q4 = __reduce_add_sync(0xffffffffu, s.q4);
    b[2] += t.none ? 0.0 : (double)(2LL * q2 - (long long)v2 * over);
    b[3] += t.none ? 0.0 : (double)(2LL * q3 - (long long)v3 * over);
    b[4] += t.none ? 0.0 : (double)(2LL * q4 - (long long)v4 * over);
  }
}
// What lies below a centroid in its coarse bin.
struct SiBelow {
  int c;
  double n, m[4];
};
__device__ __forceinline__ void si_below(const ScShared& sh, const ScGrid& g, const ScLayer& ly, SiBin& bn, float v, SiBelow& o) {
  const int lane = threadIdx.x & 31;
  int place;
  const int f = sc_fine_place(g, fminf(fmaxf(v, g.lo), g.hi), place);
  // one beyond the ends of the scale where the centroid lies outside the weights' range
  const int pv = v > g.hi ? 72768 : (v < g.lo ? -7232 : place + 32768);
  if (bn.f != f) si_bin_load(ly, f, bn);
  const bool full = sc_full(g);
  const SiCut t = si_cut(pv);
  SiSum s = {0u, 0u, 0u, 0, 0, 0};
  const long long base = si_base(ly, bn), end = ly.row0 + bn.e1;
  const int hi = end - base < SI_HEAD ? (int)(end - base) : SI_HEAD;
#pragma unroll
  for (int i = 0; i < SI_WORDS; ++i) {
    if (i > 0 && 64 * i >= hi) break;
    si_add(bn.w[i], t, full, s);
  }
  double b[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  int n = hi - (int)(ly.row0 + bn.e0 - base);
  // the weights that are not in registers, in stretches whose 32-bit sums cannot overflow
  for (long long e = base + SI_HEAD; e < end;) {
    uint4 q[4];
    if (e + 1024 <= ly.total) {
#pragma unroll
      for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const uint4*>(ly.grouped + e + 256 * i + 8 * lane);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const long long x = e + 256 * i + 8 * lane;
        q[i] = x < end ? sc_load8(ly.grouped, x, ly.total) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (e + 1024 > end) {
      const int last = (int)(end - e) - 8 * lane;
      auto cut = [&](unsigned int w, int h) { return (h < last ? w & 0xffffu : 0u) | (h + 1 < last ? w & 0xffff0000u : 0u); };
#pragma unroll
      for (int i = 0; i < 4; ++i)
        q[i] = make_uint4(cut(q[i].x, 256 * i), cut(q[i].y, 256 * i + 2), cut(q[i].z, 256 * i + 4), cut(q[i].w, 256 * i + 6));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      si_add(q[i].x, t, full, s);
      si_add(q[i].y, t, full, s);
      si_add(q[i].z, t, full, s);
      si_add(q[i].w, t, full, s);
    }
    n += end - e < 1024 ? (int)(end - e) : 1024;
    e += 1024;
    if (n >= SC_CHUNK) {
      si_total(s, n, t, full, b);
      s = SiSum{0u, 0u, 0u, 0, 0, 0};
      n = 0;
    }
  }
  si_total(s, n, t, full, b);
#pragma unroll
  for (int i = 0; i < 5; ++i) b[i] *= 0.5;
  o.c = f >> g.fshift;
  sc_shift(g, sc_fine_x0(g, f), b[0], b[1], b[2], b[3], b[4], o.m);
  o.n = b[0] + ((double)bn.e0 - ly.rec.cn[o.c]);
#pragma unroll
  for (int i = 0; i < 4; ++i) o.m[i] += bn.m[i];
}
// Centroid j: the right end of interval j (even lanes) and the left end of interval j + 1 (odd lanes); where there is no such
// interval, all weights beyond.  `pairs` of lanes have a centroid each.
template <int SLOTS>
__device__ __forceinline__ void si_ends(ScShared& sh, const ScGrid& g, const ScLayer& ly, const SiBelow& o, int j, int pairs) {
  const int k = ly.k, lane = threadIdx.x & 31;
  const bool left = lane & 1;
  const int s = left ? j + 1 : j;
  const bool inner = s > 0 && s < k;
  const double v0 = (double)sh.v[0], ctr = sc_center(g, o.c), even = inner ? sh.even[s] : ctr;
  const bool whole = left && inner && (sh.fb[inner ? s : j] >> g.fshift) != o.c;
  const double nt = ly.rec.cn[g.nc], xt = ly.rec.cx[g.nc], xc = ly.rec.cx[o.c], nc = ly.rec.cn[o.c];
  float r[5];   // the whole bin
#pragma unroll
  for (int i = 0; i < 5; ++i) r[i] = ly.rec.r[i * ly.rec.stride + o.c];
  // everything below the centroid, or above it
  double nn = o.n + nc, xx = fma(ctr, o.n, fma(g.hc, o.m[0], xc));
  nn = left ? nt - nn : nn;
  xx = left ? xt - xx : xx;
  if (sh.n0 > 0) {   // weights that are exactly zero
    const float v = left ? -sh.v[k - 1] : sh.v[0];
    nn += (v > 0.f ? 1.0 : (v == 0.f ? 0.5 : 0.0)) * (double)sh.n0;
  }
  xx = fma(-v0, nn, xx);
  // the piece below the right end; above the left end the whole bin (unless the right end lies in it) minus what is below
  const ScCoef co = sc_coef((float)((ctr - even) * (double)ly.slope));
  double n = o.n, m[4];
  n = left ? (whole ? (double)r[0] : 0.0) - n : n;
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = left ? (whole ? (double)r[i + 1] : 0.0) - o.m[i] : o.m[i];
  double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  sc_bin_sums<false, double>(co, g.eta, n, m[0], m[1], m[2], m[3], ctr - v0, g.hc, acc);
  if (lane < 2 * pairs) {
    double2* d = reinterpret_cast<double2*>(sh.ev[s * SLOTS + (left ? SLOTS - 2 : SLOTS - 1)]);
    d[0] = inner ? make_double2(acc[0], acc[1]) : make_double2(left ? nn : 0.0, left ? xx : 0.0);
    d[1] = inner ? make_double2(acc[2], acc[3]) : make_double2(left ? 0.0 : nn, left ? 0.0 : xx);
  }
}
// Interval s: the whole bins between its ends, dealt to the lanes of tw warps of which this is number `sub`.
template <int SLOTS>
__device__ __forceinline__ void si_bins(ScShared& sh, const ScGrid& g, const ScLayer& ly, int s, int sub, int tw) {
  const int lane = threadIdx.x & 31;
  const int cl = sh.fb[s - 1] >> g.fshift, cr = sh.fb[s] >> g.fshift;
  const double even = sh.even[s], v0 = (double)sh.v[0];
  double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (cr - cl >= 2) {   // (uniform)
    // the zone where neither lambda nor mu vanishes: b0 .. b1 - 1
    const double at = (even - g.ctr0) * g.inv_hc, zb = ly.zone * g.inv_hc;
    int b0 = __double2int_rd(at - zb), b1 = __double2int_ru(at + zb) + 1;
    b0 = b0 < cl + 1 ? cl + 1 : (b0 < cr ? b0 : cr);
    b1 = b1 < cl + 1 ? cl + 1 : (b1 < cr ? b1 : cr);
    const double slope = (double)ly.slope, z1 = g.hc * slope, z0 = (g.ctr0 - even) * slope, x0 = g.ctr0 - v0;
    const float* r = ly.rec.r;
    const int st = ly.rec.stride, step = 32 * tw;
    auto add = [&](int b) {
      const double bd = (double)b;
      const ScCoef c = sc_coef((float)fma(bd, z1, z0));
      sc_bin_sums<false, float>(c, g.eta, r[b], r[st + b], r[2 * st + b], r[3 * st + b], r[4 * st + b], fma(bd, g.hc, x0), g.hc, acc);
    };
    int b = b0 + sub * 32 + lane;
    // where a lane has more than four (a cold softmax: the zone holds up to 390) two at a time, as one is a chain of some hundred
    // cycles: 21 layers of a ResNet-18, tau = 5e-4, k = 7, 30 iterations 515 us one by one, 494 so.  (9 to 16 centroids gain 3 %
    // there and lose 1 % where an interval has few bins.)
    if (SLOTS > 3 && b1 - b0 > 4 * step)
      for (; b + step < b1; b += 2 * step) {
        add(b);
        add(b + step);
      }
    for (; b < b1; b += step) add(b);
    if (sub == 0 && lane < 2) {
      // outside it: lambda = 1 left of it, mu = 1 right of it
      const int lo = lane ? b1 : cl + 1, hi = lane ? cr : b0;
      const double nn = ly.rec.cn[hi] - ly.rec.cn[lo], xx = fma(-v0, nn, ly.rec.cx[hi] - ly.rec.cx[lo]);
      acc[0] += lane ? 0.0 : nn;
      acc[1] += lane ? 0.0 : xx;
      acc[2] += lane ? nn : 0.0;
      acc[3] += lane ? xx : 0.0;
    }
  }
  if (sub == 0 && lane == 0 && sh.n0 > 0) {
    // the weights that are exactly zero (see sc_zeros)
    const float vl = sh.v[s - 1], vr = sh.v[s];
    const double n = (vl < 0.f && vr > 0.f ? 1.0 : ((vl == 0.f && vr > 0.f) || (vl < 0.f && vr == 0.f) ? 0.5 : 0.0)) * (double)sh.n0;
    float lam, mu;
    sc_lambda((float)(-even * (double)ly.slope), lam, mu);
    acc[0] += n * (double)lam;
    acc[1] -= v0 * (n * (double)lam);
    acc[2] += n * (double)mu;
    acc[3] -= v0 * (n * (double)mu);
  }
  __syncwarp();
  // four sums over the warp: the first two levels also deal the sums out, so that lanes 0, 8, 16, 24 end with one each
  const bool h4 = lane & 16, h3 = lane & 8;
  double p = h4 ? acc[2] : acc[0], q = h4 ? acc[3] : acc[1];
  p += __shfl_xor_sync(0xffffffffu, h4 ? acc[0] : acc[2], 16);
  q += __shfl_xor_sync(0xffffffffu, h4 ? acc[1] : acc[3], 16);
  double r = h3 ? q : p;
  r += __shfl_xor_sync(0xffffffffu, h3 ? p : q, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if ((lane & 7) == 0) sh.ev[s * SLOTS + sub][lane >> 3] = r;
}
// The last M-step, as the first warp's lanes hold it for the stop test.
struct SiLast {
  double cnew, cold, s;
};
// Algorithm 1's stop test (see sc_stop_test); result in all lanes: the loop is done.
template <int LOG>
__device__ __forceinline__ bool si_stop_test(ScShared& sh, const ScalarParams& sp, int layer, const SiLast& la, int test) {
  const int j = threadIdx.x;
  const bool own = j < sp.k;
  const double d = own ? la.cnew - la.cold : 0.0, c = own ? la.cnew : 0.0;
  double num = d * d, den = c * c;
  const bool bad = __any_sync(0xffffffffu, own && !(la.s <= 1e300 && fabs(la.cnew) <= 1e300));
  const int dead = __popc(__ballot_sync(0xffffffffu, own && !(la.s >= S_MIN)));
#pragma unroll
  for (int o = (1 << LOG) / 2; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
  }
  // (a reciprocal from an fp32 seed where that has the range)
  const float res = sqrtf((float)(den > 1e-30 && den < 1e30 ? num * sc_rcp(den) : num / fmax(den, 1e-300)));
  const bool stop = __shfl_sync(0xffffffffu, (int)(sp.tol > 0.f && res < sp.tol), 0);
  if (j == 0) {
    sh.iters = test;
    sh.res = res;
    sh.dead = dead;
    if (test <= HIST_CAP) sp.p.hist_fwd[(size_t)layer * HIST_CAP + test - 1] = res;
    if (bad) sh.status = ST_NONFINITE;
    else if (stop) sh.status = ST_OK;
    else if (sp.tol > 0.f && test >= sp.max_iter) sh.status = ST_MAXITER;
    if (bad || stop) sh.done = test;
  }
  return bad || stop;
}
// Returns the number of M-steps.
template <int LOG>
__device__ __forceinline__ int sc_iterate(ScShared& sh, const ScalarParams& sp, int layer) {
  constexpr int SLOTS = si_slots<LOG>();
  static_assert(((1 << LOG) + 1) * SLOTS <= SI_SLOTS, "slots of the intervals");
  const ScLayer& ly = sh.ly;
  const ScGrid& g = sh.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = sp.k, max_iter = sp.max_iter;
  for (int i = threadIdx.x; i < SI_SLOTS * 4; i += SC_T) (&sh.ev[0][0])[i] = 0.0;
  if (threadIdx.x == 0) sh.flag = 0;
  __syncthreads();
  int it = 0;
  if (warp == 0) {
    const int j = lane, jc = j < k ? j : k - 1;
    const bool own = j < k;
    ScScan<LOG> scn;
#pragma unroll
    for (int l = 0; l < LOG; ++l) scn.cb[l] = scn.cf[l] = 0.0;
    SiLast la = {0.0, 0.0, 1.0};
    float cn = sh.v[jc];
    for (;;) {
      if (it == max_iter) break;
      si_arrive(SI_B1);
      double rP, rQ;
      sc_tables_warp(sh, ly, cn, scn, rP, rQ);
      si_arrive(SI_B2);
      const bool done = it > 0 && si_stop_test<LOG>(sh, sp, layer, la, it);
      if (LOG == 4 && k == SC_WARPS && !done) {
        __syncwarp();
        si_bins<SLOTS>(sh, g, ly, 1, 0, 1);
      }
      si_meet(SI_A);
      if (done) {
        if (j == 0) sh.flag = 1;
        if (it + 1 < max_iter) {   // (the others wait at the next evaluation's meetings)
          si_arrive(SI_B1);
          si_arrive(SI_B2);
        }
        break;
      }
      // ---- M-step (Algorithm 1, step 5) ----
      const double v0 = (double)sh.v[0];
      double x[2] = {0.0, 0.0}, y[2] = {0.0, 0.0};
#pragma unroll
      for (int q = 0; q < SLOTS; ++q) {
        const double2 l = reinterpret_cast<const double2*>(sh.ev[(jc + 1) * SLOTS + q])[0], m = reinterpret_cast<const double2*>(sh.ev[jc * SLOTS + q])[1];
        x[0] += l.x;
        x[1] += l.y;
        y[0] += m.x;
        y[1] += m.y;
      }
      x[0] *= rP;   // (rP = rQ = 0 in lanes without a centroid)
      x[1] *= rP;
      y[0] *= rQ;
      y[1] *= rQ;
      sc_scan_both<2, LOG>(scn, x, y);
      la.cold = (double)cn;
      la.s = x[0] + y[0];
      la.cnew = la.s >= S_MIN ? fma(x[1] + y[1], sc_rcp(la.s), v0) : la.cold;
      cn = own ? (float)la.cnew : __int_as_float(0x7f800000);
      // (the map keeps the order of the centroids up to rounding)
      const float left = __shfl_up_sync(0xffffffffu, cn, 1);
      if (__any_sync(0xffffffffu, own && j > 0 && !(left <= cn))) {
        if (own) {
          sh.vn[j] = cn;
          sh.idn[j] = sh.id[j];
        }
        __syncwarp();
        sc_sort(sh, k);
      } else if (own) {
        sh.v[j] = cn;
      }
      __syncwarp();
      cn = sh.v[jc];
      ++it;
    }
    if (j == 0) sh.steps = it;
    if (own) {   // (for the stop test of the last M-step)
      sh.cnew[j] = la.cnew;
      sh.cold[j] = la.cold;
      sh.dead_j[j] = (la.s >= S_MIN ? 0 : 1) + (!(la.s <= 1e300 && fabs(la.cnew) <= 1e300) ? 0x10000 : 0);
    }
  } else {
    // centroid j by warp j + 1; intervals by the warps that are left, several each where there are enough, or by those of the
    // first centroids besides.  16 centroids: the second warp has the last one as well as the first and is what the others wait
    // for, so it takes the ends of both at once, and the first warp its interval while it waits itself (4096 weights, tau = 0.01,
    // 30 iterations: 159 us when it took them one after the other, 134 now, 130 with 15 centroids)
    constexpr int OTHERS = SC_WARPS - 1;
    int tw = 1, sub = 0, s = 0;   // this warp's interval, 0: none
    const int t = warp - 1 - k, free_warps = OTHERS - k;
    if (free_warps >= k - 1) {
      // (warps that do not go round: to the outer intervals, which hold the most bins)
      int first = 0;
      for (int i = 0; i < k - 1; ++i) {
        int n = free_warps / (k - 1) + (i < free_warps % (k - 1) ? 1 : 0);
        n = n > SLOTS - 2 ? SLOTS - 2 : n;
        if (t >= first && t < first + n) {
          s = (i & 1) ? k - 1 - (i >> 1) : 1 + (i >> 1);
          sub = t - first;
          tw = n;
        }
        first += n;
      }
    } else {
      const int u = t >= 0 ? t : (free_warps > 0 ? free_warps : 0) + warp - 1;
      if (u < k - 1 && !(LOG == 4 && k == SC_WARPS && u == 0)) s = u + 1;
    }
    const int j = warp - 1;
    SiBin bn;
    bn.f = -1;
    bn.e0 = bn.e1 = 0u;
#pragma unroll
    for (int i = 0; i < SI_WORDS; ++i) bn.w[i] = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) bn.m[i] = 0.0;
    SiBelow o;
    while (it < max_iter) {
      if (j < k) {
        si_meet(SI_B1);
        si_below(sh, g, ly, bn, sh.v[j], o);
      } else {
        si_arrive(SI_B1);
      }
      si_meet(SI_B2);
      if (sh.flag) break;
      if (LOG == 4 && j + OTHERS < k) {
        const SiBelow o1 = o;
        si_below(sh, g, ly, bn, sh.v[OTHERS], o);
        const bool second = lane & 2;
        o.c = second ? o.c : o1.c;
        o.n = second ? o.n : o1.n;
#pragma unroll
        for (int i = 0; i < 4; ++i) o.m[i] = second ? o.m[i] : o1.m[i];
        si_ends<SLOTS>(sh, g, ly, o, second ? OTHERS : 0, 2);
      } else if (j < k) {
        si_ends<SLOTS>(sh, g, ly, o, j, 1);
      }
      if (s > 0) si_bins<SLOTS>(sh, g, ly, s, sub, tw);
      si_arrive(SI_A);
      ++it;
    }
  }
  __syncthreads();
  return sh.steps;
}

constexpr int SC_INIT_T = 1024, SC_INIT_WARPS = SC_INIT_T / 32;
// ---- first launch: layer states, working centroids, counters to zero, value range of the weights ----
__global__ void __launch_bounds__(SC_INIT_T, 1) idkm_scalar_init(const __grid_constant__ ScalarParams sp) {
  __shared__ float red_lo[SC_INIT_WARPS], red_hi[SC_INIT_WARPS];
  __shared__ unsigned int red_z[SC_INIT_WARPS];
  grid_dependency_sync();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = sp.k;
  const int layer = sc_layer_of_block(sp, (int)blockIdx.x);
  const int b = (int)blockIdx.x - sp.blk_first[layer], NB = sp.blk_first[layer + 1] - sp.blk_first[layer];
  const long long m = sp.row_off[layer + 1] - sp.row_off[layer];
  const float* Wl = sp.p.W + sp.row_off[layer];
  if (b == 0) {
    if (tid < SC_SYNC_WORDS) sp.p.sync[(size_t)layer * SC_SYNC_WORDS + tid] = 0u;
    if (tid < k) sp.p.C[(size_t)layer * k + tid] = sp.p.C0[(size_t)layer * k + tid];
    if (tid == 0) {
      LayerState s;
      memset(&s, 0, sizeof(s));
      s.status = ST_OK;
      s.adj_prev = 3.0e38f;
      sp.p.st[layer] = s;
    }
  }
  for (int i = (int)blockIdx.x * SC_INIT_T + tid; i < sp.n_group_rows; i += (int)gridDim.x * SC_INIT_T) sp.p.gtick[i] = 0u;
  for (int h = 0; h < 2; ++h)
    for (int i = (int)blockIdx.x * SC_INIT_T + tid; i < sp.p.n_pair_ticks[h]; i += (int)gridDim.x * SC_INIT_T) sp.p.pair_ticks[h][i] = 0u;
  const int cap = sp.fine_off[layer + 1] - sp.fine_off[layer];
  if (NB > 1)
    for (int i = b * SC_INIT_T + tid; i < cap; i += NB * SC_INIT_T) sp.p.gcount[sp.fine_off[layer] + i] = 0u;
  const long long r0 = m * b / NB, r1 = m * (b + 1) / NB;
  float lo = __int_as_float(0x7f800000), hi = -lo;
  int bad = 0;
  unsigned int nz = 0;
  auto take = [&](float w) {
    bad |= !(fabsf(w) <= 3.4028235e38f);
    const bool z = (w == 0.f);
    nz += z ? 1u : 0u;
    lo = z ? lo : fminf(lo, w);
    hi = z ? hi : fmaxf(hi, w);
  };
  long long r = r0 + tid;
  for (; r + 7 * SC_INIT_T < r1; r += 8 * SC_INIT_T) {
    float w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __ldg(Wl + r + i * SC_INIT_T);
#pragma unroll
    for (int i = 0; i < 8; ++i) take(w[i]);
  }
  for (; r < r1; r += SC_INIT_T) take(__ldg(Wl + r));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  nz = __reduce_add_sync(0xffffffffu, nz);
  if (lane == 0) {
    red_lo[warp] = lo;
    red_hi[warp] = hi;
    red_z[warp] = nz;
  }
  bad = __syncthreads_or(bad);
  if (warp == 0) {
    lo = red_lo[lane];
    hi = red_hi[lane];
    nz = __reduce_add_sync(0xffffffffu, red_z[lane]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) sp.p.bstat[blockIdx.x] = make_float4(lo, hi, bad ? 1.f : 0.f, __uint_as_float(nz));
  }
}

// Nothing was computed: report, and leave tables that later passes can read without harm.
__device__ __noinline__ void sc_give_up(const ScalarParams& sp, int layer, int status) {
  const int tid = threadIdx.x, k = sp.k, K1 = k + 1;
  double* tab = sp.p.tab + (size_t)layer * SC_NTAB * K1;
  float* ft = sp.p.ftab + (size_t)layer * SC_NFTAB * K1;
  float* Cl = sp.p.C + (size_t)layer * k;
  LayerState* st = sp.p.st + layer;
  for (int i = tid; i < SC_NTAB * K1; i += SC_T) tab[i] = 0.0;
  for (int i = tid; i < SC_NFTAB * K1; i += SC_T) ft[i] = 0.f;
  const float nan = __int_as_float(0x7fc00000);
  for (int i = tid; i < k; i += SC_T) {
    sp.p.perm[(size_t)layer * k + i] = i;
    sp.p.S[(size_t)layer * k + i] = 0.f;
    sp.p.F[(size_t)layer * k + i] = status == ST_NONFINITE ? nan : Cl[i];
    if (status == ST_NONFINITE) Cl[i] = nan;
  }
  if (tid == 0) {
    st->status = status;
    st->fwd_iters = st->fwd_done = status == ST_NONFINITE ? 1 : 0;
    st->fwd_res = status == ST_NONFINITE ? nan : 0.f;
  }
}

// The iterations of a layer, by its first block, once the bins are there (DIRECT: without bins, by all its blocks alike).  LOG:
// codebooks of at most 2^LOG centroids, whose M-step one warp takes; 0: larger ones.
template <int LOG, bool DIRECT>
__device__ __forceinline__ void sc_rest(ScShared& sh, const ScalarParams& sp, int layer, bool in_smem, const unsigned int* fstart,
                                        const long long* frec, const unsigned short* grouped) {
  extern __shared__ __align__(16) unsigned char smem_all[];
  unsigned char* dyn = smem_all + SC_SH_BYTES;
  (void)dyn;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = sp.k, K1 = k + 1;
  const int kw = LOG > 0 ? 1 : (k + 31) >> 5;
  const int cap = sp.fine_off[layer + 1] - sp.fine_off[layer];
  double* tab = sp.p.tab + (size_t)layer * SC_NTAB * K1;
  float* ft = sp.p.ftab + (size_t)layer * SC_NFTAB * K1;
  LayerState* st = sp.p.st + layer;
  float* Cl = sp.p.C + (size_t)layer * k;
  const bool leader = !DIRECT || (int)blockIdx.x == sp.blk_first[layer];   // (all blocks of the layer come to the same results)
  const ScGrid& g = sh.g;
  ScLayer ly;
  ly.grouped = sp.p.grouped;
  ly.row0 = sp.row_off[layer];
  ly.total = sp.row_off[sp.n_layers];
  ly.fstart = fstart;
  ly.frec = reinterpret_cast<const double*>(frec);
  ly.k = k;
  ly.tau = 1.0 / sp.inv_tau_d;
  ly.inv_tau = sp.inv_tau_d;
  ly.slope = (float)(2.0 * 1.4426950408889634 * sp.inv_tau_d);
  ly.zone = SC_ZONE / (double)ly.slope;
  ly.twl = 0;
  ly.wl = 0;
  ly.lpi = k - 1 <= SC_WARPS ? 32 : (k - 1 <= 2 * SC_WARPS ? 16 : 8);
  while (ly.wl < 1 && (k << (ly.wl + 1)) <= SC_WARPS) ++ly.wl;
  while (!DIRECT && ly.twl < 2 && k > 1 && ((k - 1) << (ly.twl + 1)) <= SC_WARPS) ++ly.twl;
  if constexpr (!DIRECT) {
    // ---- coarse records: into shared memory where they fit; running counts and x sums ----
    const ScRec gr = sc_global_rec(sp, layer, cap);
    ly.rec = gr;
    if (g.nc <= SC_REC_SMEM) {
      const int stride = g.nc <= SC_SMALL_NC ? SC_SMALL_NC : SC_REC_SMEM;
      ly.rec.cn = reinterpret_cast<double*>(dyn);
      ly.rec.cx = ly.rec.cn + stride + 1;
      ly.rec.r = reinterpret_cast<float*>(ly.rec.cx + stride + 1);
      ly.rec.stride = stride;
    }
    __syncthreads();   // (the counters, which lie in the same place, are no longer read)
    double carry = 0.0;
    for (int t = 0; t < g.nc; t += SC_T) {
      const int c = t + tid;
      double x = c < g.nc ? __ldcg(gr.cx + c + 1) : 0.0;
      if (c < g.nc && g.nc <= SC_REC_SMEM) {
#pragma unroll
        for (int q = 0; q < 5; ++q) ly.rec.r[q * ly.rec.stride + c] = __ldcg(gr.r + (size_t)q * cap + c);
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) sh.scan_x[warp] = x;
      __syncthreads();
      double before = 0.0, total = 0.0;
      for (int w = 0; w < SC_WARPS; ++w) {
        const double y = sh.scan_x[w];
        before += w < warp ? y : 0.0;
        total += y;
      }
      if (c < g.nc) {
        ly.rec.cx[c + 1] = carry + before + x;
        ly.rec.cn[c + 1] = (double)fstart[(c + 1) << g.fshift];
      }
      carry += total;
      __syncthreads();
    }
    if (tid == 0) ly.rec.cx[0] = ly.rec.cn[0] = 0.0;
    if (in_smem) {
      ly.row0 = 0;
      ly.grouped = grouped;
      ly.total = sp.row_off[layer + 1] - sp.row_off[layer];
    }
  }
  constexpr bool one_warp = LOG > 0;
  double a = 0.0, ap = 0.0, rP = 0.0, rQ = 0.0;   // (more than 32 centroids)
  ScScan<LOG> scn;
#pragma unroll
  for (int l = 0; l < (LOG > 0 ? LOG : 1); ++l) scn.cb[l] = scn.cf[l] = 0.0;
  for (int i = tid; i < SC_PARTS * 2; i += SC_T) (&sh.Ls[0][0])[i] = (&sh.Ms[0][0])[i] = (&sh.Xs[0][0])[i] = 0.0;
  if (tid == 0) {
    sh.done = 0;
    sh.iters = 0;
    sh.dead = 0;
    sh.status = ST_OK;
    sh.res = 0.f;
  }
  if (tid == 0) sh.ly = ly;
  auto tables = [&]() {
    if constexpr (one_warp) {
      if (warp == 0) sc_tables_warp(sh, ly, lane < k ? sh.v[lane] : sh.v[k - 1], scn, rP, rQ);
    } else if (tid < kw * 32) {
      sc_tables_block(sh, ly, a, ap, rP, rQ);
    }
  };
  // sums of the two sides -> what every centroid receives from all intervals
  auto spread2 = [&](double (&x)[2], double (&y)[2]) {
    if constexpr (one_warp) {
      sc_scan_both<2, LOG>(scn, x, y);
    } else {
      lin_scan<2, false>(a, x, k, sh.tmp);
      lin_scan<2, true>(ap, y, k, sh.tmp);
    }
  };
  constexpr bool quick = !DIRECT && LOG > 0 && (1 << LOG) <= SI_K;   // the iterations are sc_iterate's
  if constexpr (!quick) tables();
  __syncthreads();

  int it = 0;
  if constexpr (quick) {
    it = sc_iterate<LOG>(sh, sp, layer);
    tables();
    __syncthreads();
  }
  while (!quick && it < sp.max_iter) {
    if constexpr (DIRECT) {
      if (!sd_sums(sh, sp, layer, false, it)) {
        if (leader) sc_give_up(sp, layer, ST_TIMEOUT);
        return;
      }
    } else {
      sc_evaluate<false, quick>(sh, ly, sp, layer, it);
      __syncthreads();
    }
    if (sh.done) break;
    if (tid < kw * 32) {
      // ---- M-step (Algorithm 1, step 5) ----
      const int j = tid;
      const bool own = j < k;
      const int jc = own ? j : k - 1;
      double L0, L1, M0, M1;
      sc_gather(sh.Ls, jc, ly.twl, L0, L1);
      sc_gather(sh.Ms, jc, ly.twl, M0, M1);
      double x[2] = {L0 * rP, L1 * rP}, y[2] = {M0 * rQ, M1 * rQ};   // (rP = rQ = 0 in threads without a centroid)
      spread2(x, y);
      const double v0 = (double)sh.v[0], cold = (double)sh.v[jc];
      const double s = x[0] + y[0];
      const bool alive = (s >= S_MIN);
      const double cnew = alive ? fma(x[1] + y[1], sc_rcp(s), v0) : cold;
      float cn = (float)cnew;
      if (own) {
        sh.cnew[j] = cnew;
        sh.cold[j] = cold;
        sh.dead_j[j] = (alive ? 0 : 1) + ((!(s == s) || s > 1e300 || !(cnew == cnew) || fabs(cnew) > 1e300) ? 0x10000 : 0);
      } else {
        cn = __int_as_float(0x7f800000);
      }
      // (the map keeps the order of the centroids up to rounding)
      float left = __shfl_up_sync(0xffffffffu, cn, 1);
      bool out_of_order;
      if constexpr (one_warp) {
        out_of_order = __any_sync(0xffffffffu, own && j > 0 && !(left <= cn));
      } else {
        sc_bar(kw);   // (everybody has read the old centroids)
        if (own) sh.vn[j] = cn;
        if (j == 0) sh.flag = 0;
        sc_bar(kw);
        if ((j & 31) == 0 && j > 0) left = sh.vn[j - 1];
        if (own && j > 0 && !(left <= cn)) sh.flag = 1;
        sc_bar(kw);
        out_of_order = sh.flag != 0;
      }
      if (out_of_order) {
        if (own) {
          sh.vn[j] = cn;
          sh.idn[j] = sh.id[j];
        }
        sc_sync(kw);
        sc_sort(sh, k);
      } else {
        if (one_warp) __syncwarp();
        if (own) sh.v[j] = cn;
        sc_sync(kw);
      }
    }
    tables();
    ++it;
    __syncthreads();
  }

  // ---- sums at the returned centroids: S, F and the tables of the passes that follow ----
  if constexpr (DIRECT) {
    if (!sd_sums(sh, sp, layer, true, (it == sp.max_iter && !sh.done) ? it : 0)) {
      if (leader) sc_give_up(sp, layer, ST_TIMEOUT);
      return;
    }
    if (!leader) return;
  } else {
    sc_evaluate<true, quick>(sh, ly, sp, layer, (it == sp.max_iter && !sh.done) ? it : 0);
  }
  __syncthreads();
  if (tid < kw * 32) {
    const bool own = tid < k;
    const int jc = own ? tid : k - 1;
    double L0, L1, M0, M1, X0, X1;
    sc_gather(sh.Ls, jc, ly.twl, L0, L1);
    sc_gather(sh.Ms, jc, ly.twl, M0, M1);
    sc_gather(sh.Xs, jc, ly.twl, X0, X1);
    double x[2] = {L0 * rP, L1 * rP}, y[2] = {M0 * rQ, M1 * rQ};
    spread2(x, y);
    // averages of the centroids from every centroid on resp. up to it, relative to v_0
    const double v0 = (double)sh.v[0], dv = own ? (double)sh.v[tid] - v0 : 0.0;
    double qp[2] = {dv, 0.0}, pp[2] = {dv, 0.0};
    spread2(qp, pp);
    double bad[1] = {0.0};
    sc_sync(kw);
    if (own) {
      const double s = x[0] + y[0];
      const bool alive = (s >= S_MIN);
      const double f = alive ? (x[1] + y[1]) / s : dv;
      if (!(s == s) || s > 1e300 || !(f == f)) bad[0] = 1.0;
      const int id = sh.id[tid];
      const size_t lk = (size_t)layer * k;
      sp.p.perm[lk + tid] = id;
      Cl[id] = sh.v[tid];
      sp.p.S[lk + id] = alive ? (float)s : 0.f;
      sp.p.F[lk + id] = (float)(v0 + f);
      double* t = tab + tid;
      t[TB_V * K1] = dv;
      t[TB_A * K1] = one_warp ? scn.cb[0] : a;
      t[TB_RP * K1] = rP;
      t[TB_RQ * K1] = rQ;
      t[TB_L0 * K1] = L0;
      t[TB_L1 * K1] = L1;
      t[TB_M0 * K1] = M0;
      t[TB_M1 * K1] = M1;
      t[TB_X0 * K1] = X0;
      t[TB_X1 * K1] = X1;
      t[TB_S * K1] = alive ? s : 0.0;
      t[TB_F * K1] = f;
      if (tid == 0) tab[TB_V * K1 + k] = v0;
      sh.qs[tid] = qp[0] * rQ;
    }
    sc_sync(kw);
    if (own) {
      // interval tid + 1 (and interval 0): the outer ones have their even point far outside
      const double cl = pp[0] * rP, cr = tid + 1 < k ? sh.qs[tid + 1] : cl;
      float* o = ft + tid + 1;
      float e = 3.0e38f, off = 0.f;
      if (tid + 1 < k) {
        const double even = sh.even[tid + 1];
        e = (float)even;
        off = (float)(((double)e - even) * (double)ly.slope);
      }
      ft[FT_V * K1 + tid] = sh.v[tid];
      o[FT_E * K1] = e;
      o[FT_O * K1] = off;
      o[FT_R * K1] = (float)(v0 + cr);
      o[FT_D * K1] = (float)(cl - cr);
      if (tid == 0) {
        ft[FT_E * K1] = -3.0e38f;
        ft[FT_O * K1] = 0.f;
        ft[FT_R * K1] = (float)(v0 + sh.qs[0]);
        ft[FT_D * K1] = 0.f;
      }
    }
    sc_reduce<1>(bad, k, sh.tmp);
    if (tid == 0) {
      st->fwd_iters = sh.iters;
      st->fwd_res = sh.res;
      st->dead = sh.dead;
      st->fwd_done = sh.done;
      st->status = bad[0] > 0.0 ? ST_NONFINITE : sh.status;
    }
  }
}
template <int LOG>
__device__ __noinline__ void sd_rest(ScShared& sh, const ScalarParams& sp, int layer) {
  sc_rest<LOG, true>(sh, sp, layer, false, nullptr, nullptr, nullptr);
}

// LOG: as above.
template <int LOG>
__global__ void __launch_bounds__(SC_T, 1) idkm_scalar_loop(const __grid_constant__ ScalarParams sp) {
  extern __shared__ __align__(16) unsigned char smem_all[];
  ScShared& sh = *reinterpret_cast<ScShared*>(smem_all);
  unsigned char* dyn = smem_all + SC_SH_BYTES;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = sp.k;
  const int layer = sc_layer_of_block(sp, (int)blockIdx.x);
  const int b = (int)blockIdx.x - sp.blk_first[layer], NB = sp.blk_first[layer + 1] - sp.blk_first[layer];
  const long long m = sp.row_off[layer + 1] - sp.row_off[layer];
  const float* Wl = sp.p.W + sp.row_off[layer];
  unsigned short* grouped = sp.p.grouped + sp.row_off[layer];
  const int fo = sp.fine_off[layer], cap = sp.fine_off[layer + 1] - fo;
  unsigned int* fstart = sp.p.fstart + fo + layer;
  unsigned int* gcount = sp.p.gcount + fo;
  long long* frec = sp.p.frec + (size_t)fo * 4;
  unsigned int* sync = sp.p.sync + (size_t)layer * SC_SYNC_WORDS;
  LayerState* st = sp.p.st + layer;
  float* Cl = sp.p.C + (size_t)layer * k;
  const bool alone = (NB == 1) && (sp.missing_arrivals == 0);
  unsigned int meet = 0;
  auto barrier = [&](bool stay) {
    if (alone) {
      __syncthreads();
      return true;
    }
    ++meet;
    return sc_team_barrier(sync, meet * (unsigned int)(NB + sp.missing_arrivals), sp.spin_limit, &sh.ok, stay);
  };
  const long long r0 = m * b / NB, r1 = m * (b + 1) / NB;
  unsigned int* cnt = reinterpret_cast<unsigned int*>(dyn);
  auto in_smem = [&](const ScGrid& g) {
    return alone && g.nc <= SC_SMALL_NC &&
           36 * (size_t)g.nf + 64 + 2 * ((size_t)m + 16) + 4 * (size_t)g.nf <= (size_t)(SC_BIN_BYTES - SC_SMALL_OFF);
  };
  grid_dependency_sync();
  if (warp == 0) {
    float lo = __int_as_float(0x7f800000), hi = -lo, bad = 0.f;
    long long nz = 0;
    for (int i = lane; i < NB; i += 32) {
      const float4 s = __ldcg(sp.p.bstat + sp.blk_first[layer] + i);
      lo = fminf(lo, s.x);
      hi = fmaxf(hi, s.y);
      bad = fmaxf(bad, s.z);
      nz += (long long)__float_as_uint(s.w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      bad = fmaxf(bad, __shfl_xor_sync(0xffffffffu, bad, o));
      nz += __shfl_xor_sync(0xffffffffu, nz, o);
    }
    if (lane == 0) {
      sh.bad = bad > 0.f;
      sh.g = sc_make_grid(lo, hi, 1.0 / sp.inv_tau_d, m, cap);
      sh.n0 = nz;
    }
  }
  __syncthreads();
  int status = ST_OK;
  bool direct = sh.g.eta > SC_ETA_MAX;   // (uniform over the layer's blocks, as all that is read here and below)
  if (sh.bad) {
    status = ST_NONFINITE;   // NaN or Inf among the weights
    if (b != 0) return;
  } else if (!direct) {
    const ScGrid g = sh.g;
    const int nf = g.nf;
    bool ok = true;
    if (in_smem(g)) {
      // a small layer of one block: everything stays in shared memory (the counters at its end)
      frec = reinterpret_cast<long long*>(dyn + SC_SMALL_OFF);
      fstart = reinterpret_cast<unsigned int*>(frec + 4 * (size_t)nf);
      grouped = reinterpret_cast<unsigned short*>(fstart + ((nf + 4) & ~3));
      cnt = reinterpret_cast<unsigned int*>(dyn + SC_BIN_BYTES) - ((nf + 3) & ~3);
    }
    // ---- count the block's weights per fine bin ----
    for (int i = tid; i < nf; i += SC_T) cnt[i] = 0u;
    __syncthreads();
    {
      long long r = r0 + tid;
      for (; r + 15 * SC_T < r1; r += 16 * SC_T) {
        float w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = __ldg(Wl + r + i * SC_T);
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (w[i] != 0.f) atomicAdd(&cnt[sc_fine(g, w[i])], 1u);
      }
      for (; r < r1; r += SC_T) {
        const float w = __ldg(Wl + r);
        if (w != 0.f) atomicAdd(&cnt[sc_fine(g, w)], 1u);
      }
    }
    __syncthreads();
    if (NB > 1) {
      // where this block's share of every bin begins inside the bin (which block comes first does not matter)
      for (int i = tid; i < nf; i += SC_T) {
        const unsigned int c = cnt[i];
        cnt[i] = c ? atomicAdd(&gcount[i], c) : 0u;
      }
    }
    ok = barrier(true);
    constexpr unsigned int BIG = 4 * SC_CHUNK;
    if (ok) {
      // ---- first element of every bin: exclusive prefix over the bins, four per thread and round ----
      unsigned int carry = 0, most = 0;
      auto fetch = [&](int i) {
        uint4 c = make_uint4(0u, 0u, 0u, 0u);
        if (i < nf) {
          // (capacities and shared memory are multiples of four bins; what lies past the last bin is masked)
          c = NB > 1 ? __ldcg(reinterpret_cast<const uint4*>(gcount + i)) : *reinterpret_cast<const uint4*>(cnt + i);
          if (i + 1 >= nf) c.y = 0u;
          if (i + 2 >= nf) c.z = 0u;
          if (i + 3 >= nf) c.w = 0u;
        }
        return c;
      };
      uint4 next = fetch(4 * tid);
      for (int t = 0; t < nf; t += 4 * SC_T) {
        const int i = t + 4 * tid;
        const uint4 c = next;
        if (NB > 1) next = fetch(i + 4 * SC_T);
        const unsigned int sum = c.x + c.y + c.z + c.w;
        most = max(max(most, max(c.x, c.y)), max(c.z, c.w));
        unsigned int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        if (lane == 31) sh.scan[warp] = x;
        __syncthreads();
        const unsigned int y = lane < SC_WARPS ? sh.scan[lane] : 0u;   // (every warp adds up the warp totals itself)
        const unsigned int before = __reduce_add_sync(0xffffffffu, lane < warp ? y : 0u);
        const unsigned int total = __reduce_add_sync(0xffffffffu, y);
        if (i < nf) {
          const unsigned int f0 = carry + before + x - sum;
          const uint4 f = make_uint4(f0, f0 + c.x, f0 + c.x + c.y, f0 + c.x + c.y + c.z);
          uint4* o = reinterpret_cast<uint4*>(cnt + i);
          if (NB > 1) {
            uint4 q = *o;
            q.x += f.x;
            q.y += f.y;
            q.z += f.z;
            q.w += f.w;
            *o = q;
          } else {
            *o = f;
          }
          if (b == 0) {
            const unsigned int fs[4] = {f.x, f.y, f.z, f.w}, cs[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (i + q < nf) {
                fstart[i + q] = fs[q];
                if (cs[q] > BIG) {   // (its moments are added up by all warps of the layer)
                  long long* z = frec + (size_t)(i + q) * 4;
                  z[0] = z[1] = z[2] = z[3] = 0;
                }
              }
          }
        }
        carry += total;
        __syncthreads();
        if (NB == 1) next = fetch(i + 4 * SC_T);
      }
      if (b == 0 && tid == 0) fstart[nf] = carry;
      direct = __syncthreads_or((long long)most > SC_CROWD + m / 256) != 0;
    }
    if (ok && !direct) {
      // ---- group the weights' places by fine bin ----
      auto put = [&](float w) {
        if (w == 0.f) return;
        int p;
        const int i = sc_fine_place(g, w, p);
        grouped[atomicAdd(&cnt[i], 1u)] = (unsigned short)(p + 32768);
      };
      long long r = r0 + tid;
      for (; r + 7 * SC_T < r1; r += 8 * SC_T) {
        float w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = __ldg(Wl + r + i * SC_T);
#pragma unroll
        for (int i = 0; i < 8; ++i) put(w[i]);
      }
      for (; r < r1; r += SC_T) put(__ldg(Wl + r));
      ok = barrier(true);
    }
    if (ok && !direct) {
      // ---- integer sums of powers of the places, per fine bin; groups of 32 bins are dealt to the layer's warps ----
      if (NB > 1) {
        for (int i = tid; i < nf; i += SC_T) cnt[i] = __ldcg(fstart + i + 1);
        __syncthreads();
      }   // (otherwise the counters have moved on to the end of every bin)
      int have_big = 0;
      if (m <= 24LL * nf) {
        // few weights per bin: one thread each
        for (int i = b * SC_T + tid; i < nf; i += NB * SC_T) {
          const unsigned int e0 = i > 0 ? cnt[i - 1] : 0u, e1 = cnt[i];
          if (e1 - e0 > BIG) continue;
          long long t1 = 0, t2 = 0, t3 = 0, t4 = 0;
#pragma unroll 4
          for (unsigned int e = e0; e < e1; ++e) {
            const int p = (int)grouped[e] - 32768;
            int p2, p3, p4;
            sc_powers(p, p2, p3, p4);
            t1 += p;
            t2 += p2;
            t3 += p3;
            t4 += p4;
          }
          longlong2* o = reinterpret_cast<longlong2*>(frec + (size_t)i * 4);
          o[0] = make_longlong2(t1, t2);
          o[1] = make_longlong2(t3, t4);
        }
      } else {
        // a quarter of a warp each, eight places per lane and load, the next bin's first two loads issued ahead
        const bool own = in_smem(g);
        const unsigned short* all = own ? grouped : sp.p.grouped;
        const long long row0 = own ? 0 : sp.row_off[layer], total = own ? m : sp.row_off[sp.n_layers];
        const int step = NB * SC_T / 8, ql = lane & 7;
        const bool full = sc_full(g);
        const unsigned int qmask = 0xffu << (lane & 24);
        int i = (b * SC_T + tid) >> 3;
        long long A0 = 0, A1 = 0;
        uint4 x0 = make_uint4(0u, 0u, 0u, 0u), x1 = x0;
        auto first = [&](int bi, long long& a0, long long& a1, uint4& y0, uint4& y1) {
          a0 = a1 = 0;
          y0 = y1 = make_uint4(0u, 0u, 0u, 0u);
          if (bi < nf) {
            a0 = row0 + (bi > 0 ? cnt[bi - 1] : 0u);
            a1 = row0 + cnt[bi];
            const long long e = (a0 & ~7LL) + 8 * ql;
            if (e < a1) y0 = sc_load8(all, e, total);
            if (e + 64 < a1) y1 = sc_load8(all, e + 64, total);
          }
        };
        first(i, A0, A1, x0, x1);
        for (; i < nf; i += step) {
          long long B0, B1;
          uint4 n0, n1;
          first(i + step, B0, B1, n0, n1);
          if (A1 - A0 <= (long long)BIG) {   // (32-bit sums per lane: at most BIG / 8 = 4096 places of at most 2^16)
            int s1 = 0, s2 = 0, s3 = 0, s4 = 0;
            long long e = (A0 & ~7LL) + 8 * ql;
            while (e < A1) {
              const unsigned int xs[4] = {x0.x, x0.y, x0.z, x0.w};
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const bool in = q >= (int)(A0 - e) && q < (int)(A1 - e);
                const int p = in ? (int)((q & 1) ? xs[q >> 1] >> 16 : xs[q >> 1] & 0xffffu) - 32768 : 0;
                s1 += p;
                s2 += (p * p + 8192) >> 14;
                if (full) {
                  int p2, p3, p4;
                  sc_powers(p, p2, p3, p4);
                  s3 += p3;
                  s4 += p4;
                }
              }
              e += 64;
              x0 = x1;
              if (e + 64 < A1) x1 = sc_load8(all, e + 64, total);
            }
            long long t[4] = {s1, s2, s3, s4};
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int o = 4; o > 0; o >>= 1) t[q] += __shfl_xor_sync(qmask, t[q], o);
            if (ql < 4) frec[(size_t)i * 4 + ql] = ql == 0 ? t[0] : (ql == 1 ? t[1] : (ql == 2 ? t[2] : t[3]));
          }
          A0 = B0;
          A1 = B1;
          x0 = n0;
          x1 = n1;
        }
      }
      // bins with very many nearly equal weights: all warps of the layer share them
      if (m > (long long)BIG)
        for (int i = tid; i < nf; i += SC_T) have_big |= (cnt[i] - (i > 0 ? cnt[i - 1] : 0u) > BIG);
      have_big = __syncthreads_or(have_big);
      if (have_big) {   // (uniform over the layer's blocks: all read the same counts)
        for (int i0 = 0; i0 < nf; i0 += SC_T) {
          const int i = i0 + tid;
          const unsigned int mask_w = __ballot_sync(0xffffffffu, i < nf && cnt[i] - (i > 0 ? cnt[i - 1] : 0u) > BIG);
          if (lane == 0) sh.scan[warp] = mask_w;
          __syncthreads();
          for (int w = 0; w < SC_WARPS; ++w) {
            unsigned int mask = sh.scan[w];
            while (mask) {
              const int bi = i0 + w * 32 + __ffs(mask) - 1;
              mask &= mask - 1;
              const unsigned int e0 = bi > 0 ? cnt[bi - 1] : 0u, e1 = cnt[bi];
              for (unsigned long long eb = (unsigned long long)e0 + 1024ull * (b * SC_WARPS + warp); eb < e1; eb += 1024ull * NB * SC_WARPS) {
                int t[4] = {0, 0, 0, 0};
                for (int q = 0; q < 32; ++q) {
                  const unsigned long long e = eb + 32ull * q + lane;
                  if (e < e1) {
                    const int p = (int)grouped[e] - 32768;
                    int p2, p3, p4;
                    sc_powers(p, p2, p3, p4);
                    t[0] += p;
                    t[1] += p2;
                    t[2] += p3;
                    t[3] += p4;
                  }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const int s = __reduce_add_sync(0xffffffffu, t[q]);
                  if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(frec + (size_t)bi * 4 + q), (unsigned long long)(long long)s);
                }
              }
            }
          }
          __syncthreads();
        }
      }
      ok = barrier(true);
    }
    if (ok && !direct) {
      // ---- moments about the coarse bins' centres, prefixed over the fine bins of every coarse bin; coarse records ----
      const ScRec gr = sc_global_rec(sp, layer, cap);
      const int wd = g.F < 32 ? g.F : 32;      // lanes per coarse bin
      const int per = g.F < 32 ? 32 / g.F : 1; // coarse bins per step of a warp
      for (int c0 = (b * SC_WARPS + warp) * per; c0 < g.nc; c0 += NB * SC_WARPS * per) {
        const int c = c0 + lane / wd;
        const bool in = c < g.nc;
        double run[4] = {0.0, 0.0, 0.0, 0.0};
        for (int f0 = 0; f0 < g.F; f0 += wd) {
          const int f = (c << g.fshift) + f0 + (lane % wd);
          double x[4] = {0.0, 0.0, 0.0, 0.0}, y[4];
          if (in) {
            // (written by other blocks a barrier ago and not read before: plain loads see it; the place may be shared memory)
            const longlong2 u0 = reinterpret_cast<const longlong2*>(frec + (size_t)f * 4)[0];
            const longlong2 u1 = reinterpret_cast<const longlong2*>(frec + (size_t)f * 4)[1];
            const double n = (double)(cnt[f] - (f > 0 ? cnt[f - 1] : 0u));
            sc_shift(g, sc_fine_x0(g, f), n, (double)u0.x, (double)u0.y, (double)u1.x, (double)u1.y, x);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) y[q] = x[q];
          for (int o = 1; o < wd; o <<= 1)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const double t = __shfl_up_sync(0xffffffffu, y[q], o, wd);
              if ((lane % wd) >= o) y[q] += t;
            }
          if (in) {
            double2* o = reinterpret_cast<double2*>(frec + (size_t)f * 4);
            o[0] = make_double2(run[0] + (y[0] - x[0]), run[1] + (y[1] - x[1]));
            o[1] = make_double2(run[2] + (y[2] - x[2]), run[3] + (y[3] - x[3]));
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) run[q] += __shfl_sync(0xffffffffu, y[q], wd - 1, wd);
        }
        if (in && lane % wd == 0) {
          const unsigned int e0 = c > 0 ? cnt[(c << g.fshift) - 1] : 0u, e1 = cnt[((c + 1) << g.fshift) - 1];
          gr.r[c] = (float)(e1 - e0);
#pragma unroll
          for (int q = 0; q < 4; ++q) gr.r[(size_t)(q + 1) * cap + c] = (float)run[q];
          gr.cx[c + 1] = fma(sc_center(g, c), (double)(e1 - e0), g.hc * run[0]);
        }
      }
      ok = barrier(b == 0);
    }
    if (!ok) status = ST_TIMEOUT;
  }
  if (tid == 0) {
    sh.meet = meet;
    sh.W = Wl;
    sh.r0 = r0;
    sh.r1 = r1;
  }
  if (b != 0 && !(direct && status == ST_OK)) return;

  // ================= from here on one block per layer (or all, without bins) =================
  const int kw = LOG > 0 ? 1 : (k + 31) >> 5;
  if (tid < kw * 32) {
    if (tid < k) {
      sh.vn[tid] = Cl[tid];
      sh.idn[tid] = tid;
    }
    sc_sync(kw);
    sc_sort(sh, k);
  }
  if (status != ST_OK) {
    sc_give_up(sp, layer, status);
    return;
  }
  if (direct) {
    sd_rest<LOG>(sh, sp, layer);
    return;
  }
  sc_rest<LOG, false>(sh, sp, layer, in_smem(sh.g), fstart, frec, grouped);
}

cudaError_t launch_scalar_init(const ScalarParams& sp, int grid, cudaStream_t stream) {
  idkm_scalar_init<<<grid, SC_INIT_T, 0, stream>>>(sp);
  return cudaGetLastError();
}

template <int LOG>
static cudaError_t launch_loop(const ScalarParams& sp, int grid, cudaStream_t stream) {
  static PerDevice limit;
  const cudaError_t allowed = allow_smem(limit, idkm_scalar_loop<LOG>, SC_DYN);
  if (allowed != cudaSuccess) return allowed;
  // blocks of one layer wait for each other: a cooperative launch is refused if they cannot all be resident.  (A grid of
  // one block per layer has no barriers and is launched plainly.)
  void* args[1] = {const_cast<ScalarParams*>(&sp)};
  if (grid == sp.n_layers && sp.missing_arrivals == 0) {
    idkm_scalar_loop<LOG><<<grid, SC_T, SC_DYN, stream>>>(sp);
    return cudaGetLastError();
  }
  return cudaLaunchCooperativeKernel((const void*)&idkm_scalar_loop<LOG>, dim3((unsigned)grid, 1, 1), dim3(SC_T, 1, 1), args, (size_t)SC_DYN, stream);
}
cudaError_t launch_scalar_loop(const ScalarParams& sp, int grid, cudaStream_t stream) {
  if (sp.k <= 2) return launch_loop<1>(sp, grid, stream);
  if (sp.k <= 4) return launch_loop<2>(sp, grid, stream);
  if (sp.k <= 8) return launch_loop<3>(sp, grid, stream);
  if (sp.k <= 16) return launch_loop<4>(sp, grid, stream);
  if (sp.k <= 32) return launch_loop<5>(sp, grid, stream);
  return launch_loop<0>(sp, grid, stream);
}

}  // namespace idkm
