// One Lanczos step after the operator has been applied, as one cooperative kernel: the
// three-term recurrence, the re-orthogonalisation, the next basis vector and the lowest
// eigenpair of the tridiagonal, all in FP64 on the device.
//
// A step on a small problem is bound by launches, by host waits and by chains of FP64
// instructions (64 cycles each on this part, whatever the number of active lanes), a step on
// a large one by the FP64 pipe (two multiply-adds per entry and basis vector).  As
// separate kernels a step took 13 launches, three host waits and 170 us in a one-warp
// bisection at Krylov size 40.  Here:
//   * every worker block keeps its slice of w in shared memory through the step; the blocks
//     meet at three grid barriers (alpha; the projections; the norm);
//   * a warp takes every eighth basis vector over the block's slice and reduces its up to
//     eight sums together (nine adds instead of forty);
//   * after the recurrence one projection pass is made, and a second one only if the first
//     took more than half of the squared norm (the criterion of Daniel, Gragg, Kaufman and
//     Stewart, Math. Comp. 30, 1976): w is then orthogonal to working precision;
//   * one more block solves the tridiagonal while the workers re-orthogonalise.
// Mean of the steps j = 0 .. 20, device time: N = 4096 23 us (208 us as separate kernels),
// N = 2^20 126 us (380 us; the vectors' traffic alone is ~40 us at this part's copy rate).
#include <algorithm>

#include "kernels.cuh"

namespace a2 {
namespace {

constexpr int kLzThreads = 256;
constexpr unsigned kLzWaitLimit = 1u << 22;

struct LzArgs {
  double* V;            // basis vectors, v_q at V + q * N
  double* w;            // H v_j on entry
  long long N;
  int j;                // v_0 .. v_j are set
  int workers;          // blocks 0 .. workers - 1; block `workers` solves the tridiagonal
  int chunk;            // entries per worker
  int in_smem;          // the slice of w lives in shared memory (else in place)
  int write_next;       // store v_{j+1}
  double beta_prev;     // beta_{j-1} (0 for j = 0)
  double* tri;          // a[64], b[64], eigenvector[64]
  double* partial;      // partial sums: (2 + 64) x workers
  unsigned* bar;        // {arrivals, abort} of this step, zero on entry
  unsigned* bar_next;   // those of the next step, zeroed here
  double* out;          // pinned host: alpha, |w|^2, theta, |last component|, gave-up flag
  unsigned wait_limit;  // polls of a bounded wait
  unsigned extra;       // self-test only: arrivals waited for beyond those that come
};

__device__ __forceinline__ double shfl_xor_d(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += shfl_xor_d(v, o);
  return v;
}
// Sums of eight values over the warp: lane l returns that of value (l >> 2) & 7.
__device__ __forceinline__ double warp_sum8(double (&v)[8], int lane) {
  double u[4], t[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double give = h16 ? v[i] : v[i + 4], keep = h16 ? v[i + 4] : v[i];
    u[i] = keep + shfl_xor_d(give, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double give = h8 ? u[i] : u[i + 2], keep = h8 ? u[i + 2] : u[i];
    t[i] = keep + shfl_xor_d(give, 8);
  }
  const double give = h4 ? t[0] : t[1], keep = h4 ? t[1] : t[0];
  double r = keep + shfl_xor_d(give, 4);
  r += shfl_xor_d(r, 2);
  r += shfl_xor_d(r, 1);
  return r;
}
__device__ __forceinline__ int warp_sum8_index(int lane) { return (lane >> 2) & 7; }

// Arrival of the whole block at the grid barrier; every write before it is visible to the
// blocks that pass wait_all for the same count.
__device__ void lz_arrive(unsigned* bar) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
  }
}
// Bounded wait for `target` arrivals; false if it (or another block) gave up.
__device__ bool lz_wait(unsigned* bar, unsigned target, unsigned limit) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    for (unsigned it = 0;; ++it) {
      if (*(volatile unsigned*)bar >= target) break;
      if (*(volatile unsigned*)(bar + 1)) { ok = 0; break; }
      if (it >= limit) {
        atomicExch(bar + 1, 1u);
        ok = 0;
        break;
      }
      if (it > 64) __nanosleep(20);
    }
    __threadfence();
  }
  __syncthreads();
  const bool r = ok != 0;
  __syncthreads();
  return r;
}

// This warp's share of lz_dots: M values, U entries of each per lane at a time (the loads
// of a batch are issued together; the loop is bound by their latency otherwise).
template <int M, int U>
__device__ __forceinline__ void lz_dot_loop(const double* V, long long ld, const double* x, int n,
                                            int k, int vg, int g, int mine, int beg, int step,
                                            double (&acc)[8]) {
  for (int e = beg; e < n; e += step * U) {
    double xe[U], ve[M][U];
#pragma unroll
    for (int i = 0; i < U; ++i) xe[i] = e + i * step < n ? x[e + i * step] : 0.0;
#pragma unroll
    for (int u = 0; u < M; ++u) {
      const int q = vg + u * g;
      const double* v = V + (long long)q * ld + e;
#pragma unroll
      for (int i = 0; i < U; ++i)
        ve[u][i] = u < mine && e + i * step < n ? (q < k ? __ldg(v + i * step) : xe[i]) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < M; ++u)
      if (u < mine)
#pragma unroll
        for (int i = 0; i < U; ++i) acc[u] = fma(ve[u][i], xe[i], acc[u]);
  }
}

// Partial sums of <V_q, x> for q < k (and of <x, x> as value k when `norm`), over the
// block's n entries: warps split the values g ways and the entries 8 / g ways.
__device__ void lz_dots(const double* V, long long ld, const double* x, int n, int k, bool norm,
                        double* part, int stride, double (*red)[64]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kk = k + (norm ? 1 : 0);
  const int g = kk > 4 ? 8 : kk > 2 ? 4 : kk > 1 ? 2 : 1, slices = 8 / g;
  const int vg = warp % g, sl = warp / g;
  const int mine = (kk - vg + g - 1) / g;          // values vg, vg + g, ... (<= 8)
  double acc[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) acc[u] = 0.0;
  const int beg = sl * 32 + lane, step = 32 * slices;
  if (mine > 4) lz_dot_loop<8, 2>(V, ld, x, n, k, vg, g, mine, beg, step, acc);
  else if (mine > 2) lz_dot_loop<4, 4>(V, ld, x, n, k, vg, g, mine, beg, step, acc);
  else if (mine > 1) lz_dot_loop<2, 6>(V, ld, x, n, k, vg, g, mine, beg, step, acc);
  else if (mine > 0) lz_dot_loop<1, 8>(V, ld, x, n, k, vg, g, mine, beg, step, acc);
  const double s = mine > 1 ? warp_sum8(acc, lane) : warp_sum_d(acc[0]);
  const int u = mine > 1 ? warp_sum8_index(lane) : 0;
  if ((lane & 3) == 0 && u < mine && (mine > 1 || lane == 0)) red[sl][vg + u * g] = s;
  __syncthreads();
  if (threadIdx.x < kk) {
    double t = red[0][threadIdx.x];
    for (int i = 1; i < slices; ++i) t += red[i][threadIdx.x];
    part[(long long)threadIdx.x * stride] = t;
  }
}

// One warp's share of lz_totals: M values (warp, warp + 8, ...), U rounds of 32 workers of each
// loaded at a time.
template <int M, int U>
__device__ __forceinline__ void lz_total_loop(const double* part, int workers, int stride, int warp,
                                              int lane, int mine, double (&acc)[8]) {
  for (int i = 0; i < workers; i += 32 * U) {
    double v[M][U];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
      for (int u = 0; u < U; ++u)
        v[m][u] = m < mine && i + 32 * u + lane < workers
                      ? __ldcg(part + (long long)(warp + 8 * m) * stride + i + 32 * u + lane)
                      : 0.0;
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (m < mine)
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + 32 * u < workers) acc[m] += v[m][u];   // (uniform: no add that does nothing)
  }
}

// tot[q] = sum over the workers of part[q * stride + i], q < kk, in a fixed order.  WIDE (above 64
// workers): a warp takes every eighth value and its lanes the workers; four threads per value,
// each adding a quarter of the partial sums one after the other, wait for 38 loads and adds at
// 150 workers (chemistry L = 8, D = 64, mean of a sweep's steps: 30.1 -> 28.0 us).  With fewer the
// four threads are the faster form, as they need no sums over a warp (Heisenberg, D = 32, 32
// workers: 26.8 us, by warps 27.6).
template <bool WIDE>
__device__ void lz_totals(const double* part, int workers, int stride, int kk, double* tot,
                          double (*red)[64]) {
  if constexpr (!WIDE) {
    const int q = threadIdx.x & 63, sl = threadIdx.x >> 6;
    double t = 0.0;
    if (q < kk)
      for (int i = sl; i < workers; i += 4) t += __ldcg(part + (long long)q * stride + i);
    red[sl][q] = t;
    __syncthreads();
    if (threadIdx.x < kk)
      tot[threadIdx.x] = (red[0][threadIdx.x] + red[1][threadIdx.x]) +
                         (red[2][threadIdx.x] + red[3][threadIdx.x]);
    __syncthreads();
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mine = (kk - warp + 7) / 8;
  double acc[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) acc[u] = 0.0;
  if (mine > 4) lz_total_loop<8, 2>(part, workers, stride, warp, lane, mine, acc);
  else if (mine > 2) lz_total_loop<4, 5>(part, workers, stride, warp, lane, mine, acc);
  else if (mine > 1) lz_total_loop<2, 5>(part, workers, stride, warp, lane, mine, acc);
  else if (mine > 0) lz_total_loop<1, 5>(part, workers, stride, warp, lane, mine, acc);
  if (mine > 1) {
    const double s = warp_sum8(acc, lane);
    const int m = warp_sum8_index(lane);
    if ((lane & 3) == 0 && m < mine) tot[warp + 8 * m] = s;
  } else if (mine > 0) {
    const double s = warp_sum_d(acc[0]);
    if (lane == 0) tot[warp] = s;
  }
  __syncthreads();
}

// ------------------------------------------------------------------ tridiagonal eigenpair
struct TriShared {
  double a[64], b[64], b2[64];
  float af[64], bf[64];
  double pv[128];          // leading minor at the sample points, with its exponent
  int pe[128];
  double Dp[64], Rp[64], Dm[64], Rm[64], z[64];
  double x, theta, resid;
  int state, low, high;    // state: 1 = accepted
  double y[64], v[64], dl[64], d[64], du[64], du2[64], rhs[64];   // fallback
};

// Lowest eigenpair by 32-way multisection of the Sturm count and inverse iteration with a
// partially pivoted elimination, one warp: the general method, for spectra that the fast
// one below does not settle (two eigenvalues closer than its sample points).
__device__ int sturm_below(const double* a, const double* b, int k, double x) {
  int cnt = 0;
  double d = a[0] - x;
  if (d < 0) ++cnt;
  for (int i = 1; i < k; ++i) {
    const double dd = (d == 0.0) ? 1e-300 : d;
    d = a[i] - x - b[i - 1] * b[i - 1] / dd;
    if (d < 0) ++cnt;
  }
  return cnt;
}
__device__ void tri_lowest_general(TriShared& S, int k) {
  const int lane = threadIdx.x & 31;
  const double* a = S.a;
  const double* b = S.b;
  double lo = 1e300, hi = -1e300, scale = 0.0;
  for (int i = 0; i < k; ++i) {
    const double r = (i > 0 ? fabs(b[i - 1]) : 0.0) + (i + 1 < k ? fabs(b[i]) : 0.0);
    lo = fmin(lo, a[i] - r);
    hi = fmax(hi, a[i] + r);
    scale = fmax(scale, fabs(a[i]) + r);
  }
  for (int it = 0; it < 40 && hi - lo > 4e-16 * fmax(scale, 1e-300); ++it) {
    const double x = lo + (hi - lo) * (double)(lane + 1) / 33.0;
    const bool above = sturm_below(a, b, k, x) >= 1;     // lowest eigenvalue <= x
    const unsigned m = __ballot_sync(0xffffffffu, above);
    const int j = m ? __ffs(m) - 1 : 32;                 // first point above the eigenvalue
    const double nlo = j == 0 ? lo : lo + (hi - lo) * (double)j / 33.0;
    const double nhi = j == 32 ? hi : lo + (hi - lo) * (double)(j + 1) / 33.0;
    if (!(nlo >= lo && nhi <= hi && nlo < nhi)) break;   // no further progress in FP64
    lo = nlo;
    hi = nhi;
  }
  const double theta = 0.5 * (lo + hi);
  if (lane != 0) return;
  // inverse iteration: (T - theta I) y = v, partially pivoted tridiagonal elimination
  double *y = S.y, *v = S.v, *dl = S.dl, *d = S.d, *du = S.du, *du2 = S.du2, *rhs = S.rhs;
  for (int i = 0; i < k; ++i) v[i] = 1.0 / sqrt((double)k) * (1.0 + 0.01 * i);
  const double eps = 1e-14 * fmax(scale, 1e-300);
  for (int rep = 0; rep < 3; ++rep) {
    for (int i = 0; i < k; ++i) {
      d[i] = a[i] - theta;
      du[i] = (i + 1 < k) ? b[i] : 0.0;
      dl[i] = (i + 1 < k) ? b[i] : 0.0;
      du2[i] = 0.0;
      rhs[i] = v[i];
    }
    for (int i = 0; i + 1 < k; ++i) {
      if (fabs(d[i]) >= fabs(dl[i])) {
        const double piv = (d[i] == 0.0) ? eps : d[i];
        d[i] = piv;
        const double f = dl[i] / piv;
        d[i + 1] -= f * du[i];
        rhs[i + 1] -= f * rhs[i];
        dl[i] = 0.0;
      } else {
        const double f = d[i] / dl[i];
        d[i] = dl[i];
        double t = d[i + 1];
        d[i + 1] = du[i] - f * t;
        if (i + 2 < k) {
          du2[i] = du[i + 1];
          du[i + 1] = -f * du2[i];
        }
        du[i] = t;
        t = rhs[i];
        rhs[i] = rhs[i + 1];
        rhs[i + 1] = t - f * rhs[i + 1];
      }
    }
    if (d[k - 1] == 0.0) d[k - 1] = eps;
    y[k - 1] = rhs[k - 1] / d[k - 1];
    if (k > 1) y[k - 2] = (rhs[k - 2] - du[k - 2] * y[k - 1]) / d[k - 2];
    for (int i = k - 3; i >= 0; --i) y[i] = (rhs[i] - du[i] * y[i + 1] - du2[i] * y[i + 2]) / d[i];
    double nrm = 0.0;
    for (int i = 0; i < k; ++i) nrm += y[i] * y[i];
    const double inv = 1.0 / sqrt(nrm);
    for (int i = 0; i < k; ++i) v[i] = y[i] * inv;
  }
  S.theta = theta;
  for (int i = 0; i < k; ++i) S.z[i] = v[i];
}

// Number of non-positive pivots of T - x I (eigenvalues below x), one thread.
__device__ int tri_count(const TriShared& S, int k, double x) {
  int c = 0;
  double q = S.a[0] - x;
  c += !(q > 0.0);
  for (int i = 1; i < k; ++i) {
    if (q == 0.0) q = 1e-300;
    q = fma(-S.b2[i - 1], 1.0 / q, S.a[i] - x);
    c += !(q > 0.0);
  }
  return c;
}

// Lowest eigenvalue S.theta and unit eigenvector S.z of the k x k tridiagonal in S.a, S.b
// (whole block, k <= 64):
//   1. FP32 sign tests of the pivots at 256 points at a time, three rounds: a bracket of
//      2^-18 of the matrix scale (the margin covers the rounding of the FP32 pivots);
//   2. the FP64 leading minors at 128 points of that bracket: the sign change brackets the
//      eigenvalue to 2^-25, and inverse quadratic interpolation of the last minor through
//      three points gives it to ~1e-15;
//   3. the twisted factorisation at that shift (Fernando, SIAM J. Matrix Anal. Appl. 18,
//      1997): pivots from the top (one warp) and from the bottom (another), the vector from
//      the smallest twist element gamma outwards, theta = x + gamma / |z|^2, residual
//      |gamma| / |z|; repeated once from theta when the residual is above rounding.
// It is accepted if the residual is small, no eigenvalue lies below it and at most one below
// it + 1e-8 scale (so theta is off by less than residual^2 / gap); otherwise the general
// method runs.
__device__ void tri_lowest(TriShared& S, int k) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (k == 1) {
    if (tid == 0) {
      S.theta = S.a[0];
      S.z[0] = 1.0;
    }
    __syncthreads();
    return;
  }
  if (tid < k) {
    S.af[tid] = (float)S.a[tid];
    if (tid + 1 < k) {
      const double t = S.b[tid] * S.b[tid];
      S.b2[tid] = t;
      S.bf[tid] = (float)t;
    }
  }
  if (tid == 0) S.state = 0;
  __syncthreads();
  float lo = 3e38f, hi = 3e38f, scale = 0.f;
  for (int i = lane; i < k; i += 32) {
    const float r = (i > 0 ? sqrtf(S.bf[i - 1]) : 0.f) + (i + 1 < k ? sqrtf(S.bf[i]) : 0.f);
    lo = fminf(lo, S.af[i] - r);
    hi = fminf(hi, S.af[i]);
    scale = fmaxf(scale, fabsf(S.af[i]) + r);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fminf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    scale = fmaxf(scale, __shfl_xor_sync(0xffffffffu, scale, o));
  }
  // outside this range the FP32 phase under- or overflows: the general method
  const bool ranged = scale > 1e-15f && scale < 1e15f;
  const float m = scale * 0x1p-19f;
  lo -= m;
  hi += m;
  for (int pass = 0; pass < 3; ++pass) {
    const float wd = hi - lo, x = fmaf(wd, (float)(tid + 1) * (1.f / 257.f), lo);
    float q = S.af[0] - x;
    bool above = !(q > 0.f);
    for (int i = 1; i < k; ++i) {
      if (above) q = 1.f;
      q = (S.af[i] - x) - __fdividef(S.bf[i - 1], q);
      above |= !(q > 0.f);
    }
    const int below = __syncthreads_count(!above);       // points under the eigenvalue
    const float nlo = below == 0 ? lo : fmaf(wd, (float)below * (1.f / 257.f), lo);
    const float nhi = below == 256 ? hi : fmaf(wd, (float)(below + 1) * (1.f / 257.f), lo);
    lo = nlo;
    hi = nhi;
  }
  const double L = (double)lo - (double)m, W = (double)hi + (double)m - L;
  bool above = true;
  if (warp < 4) {
    const double x = fma(W, (double)(tid + 1) * (1.0 / 129.0), L);
    double pm = 1.0, p = S.a[0] - x;
    int ex = 0;
    above = !(p > 0.0);
    for (int i = 1; i < k; ++i) {
      double pn = fma(S.a[i] - x, p, -(S.b2[i - 1] * pm));
      above |= !(pn > 0.0);
      // rescale by a power of two through the exponent fields (the larger of the pair)
      const int en = (__double2hiint(pn) >> 20) & 0x7ff, ep = (__double2hiint(p) >> 20) & 0x7ff;
      const int big = max(en, ep);
      if (big > 1023 + 200 || (big > 0 && big < 1023 - 200)) {
        const int sh = 1023 - big;
        ex -= sh;
        p = ep + sh > 0 && ep > 0 ? __hiloint2double(__double2hiint(p) + sh * (1 << 20),
                                                     __double2loint(p)) : 0.0;
        pn = en + sh > 0 && en > 0 ? __hiloint2double(__double2hiint(pn) + sh * (1 << 20),
                                                      __double2loint(pn)) : 0.0;
      }
      pm = p;
      p = pn;
    }
    S.pv[tid] = p;
    S.pe[tid] = ex;
  }
  const int below = __syncthreads_count(!above);
  const bool bracketed = ranged && below > 0 && below < 128;
  if (tid == 0 && bracketed) {
    const int i0 = below - 1, i1 = below, i2 = below + 1 < 128 ? below + 1 : below - 2;
    const double step = W * (1.0 / 129.0);
    auto val = [&](int i) {
      const int de = S.pe[i] - S.pe[i0];
      return de > 900 ? S.pv[i] * 0x1p900 : de < -900 ? 0.0 : ldexp(S.pv[i], de);
    };
    const double f0 = S.pv[i0], f1 = val(i1), f2 = val(i2);
    if (f0 > 0.0 && f1 <= 0.0) {
      const double d2 = i2 > i1 ? 2.0 : -1.0;            // abscissae 0, 1, d2 (in steps)
      double t = f0 * f2 / ((f1 - f0) * (f1 - f2)) + d2 * f0 * f1 / ((f2 - f0) * (f2 - f1));
      if (!(t >= 0.0 && t <= 1.0)) t = f0 / (f0 - f1);
      S.x = fma(W, (double)(i0 + 1) * (1.0 / 129.0), L) + t * step;
      S.state = 2;
    }
  }
  __syncthreads();
  const double sc = (double)scale;
  for (int rep = 0; rep < 2 && S.state == 2; ++rep) {
    const double x = S.x;
    if (warp == 0) {
      if (lane == 0) {
        double q = S.a[0] - x;
        for (int i = 0;; ++i) {
          if (q == 0.0) q = 1e-300;
          S.Dp[i] = q;
          if (i == k - 1) break;
          const double r = 1.0 / q;
          S.Rp[i] = r;
          q = fma(-S.b2[i], r, S.a[i + 1] - x);
        }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        double q = S.a[k - 1] - x;
        for (int i = k - 1;; --i) {
          if (q == 0.0) q = 1e-300;
          S.Dm[i] = q;
          if (i == 0) break;
          const double r = 1.0 / q;
          S.Rm[i] = r;
          q = fma(-S.b2[i - 1], r, S.a[i - 1] - x);
        }
      }
    } else if (warp == 2) {
      if (lane == 0) S.low = tri_count(S, k, x - 1e-12 * sc);
    } else if (warp == 3) {
      if (lane == 0) S.high = tri_count(S, k, x + 1e-8 * sc);
    }
    __syncthreads();
    if (warp == 0) {
      // twist element of smallest magnitude; multipliers of the two halves of z
      double g = 0.0;
      float best = 3e38f;
      int at = 0;
      for (int i = lane; i < k; i += 32) {
        const double t = S.Dp[i] + (S.Dm[i] - (S.a[i] - x));
        const float ft = fabsf((float)t);
        if (ft < best) {
          best = ft;
          at = i;
          g = t;
        }
        if (i + 1 < k) S.y[i] = -S.b[i] * S.Rp[i];       // z_i = y_i z_{i+1} above the twist
        if (i > 0) S.v[i] = -S.b[i - 1] * S.Rm[i];       // z_i = v_i z_{i-1} below it
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oa = __shfl_xor_sync(0xffffffffu, at, o);
        const double og = shfl_xor_d(g, o);
        if (ob < best || (ob == best && oa < at)) {
          best = ob;
          at = oa;
          g = og;
        }
      }
      __syncwarp();
      if (lane == 0) {
        S.z[at] = 1.0;
        double z = 1.0;
        for (int i = at - 1; i >= 0; --i) {
          z *= S.y[i];
          S.z[i] = z;
        }
      } else if (lane == 1) {
        double z = 1.0;
        for (int i = at + 1; i < k; ++i) {
          z *= S.v[i];
          S.z[i] = z;
        }
      }
      __syncwarp();
      double n2 = 0.0;
      for (int i = lane; i < k; i += 32) n2 = fma(S.z[i], S.z[i], n2);
      n2 = warp_sum_d(n2);
      const double inv = rsqrt(n2);
      for (int i = lane; i < k; i += 32) S.z[i] *= inv;
      const double rs = fabs(g) * inv, th = fma(g, inv * inv, x);
      if (lane == 0) {
        S.theta = th;
        const bool good = rs <= 1e-12 * sc && S.low == 0 && S.high <= 1;
        const bool fine = rs <= 1e-15 * sc;
        S.state = !good ? 0 : (fine || rep == 1) ? 1 : 2;
        S.x = th;
      }
    }
    __syncthreads();
  }
  if (S.state != 1) {
    __syncthreads();
    if (warp == 0) tri_lowest_general(S, k);
    __syncthreads();
  }
}

template <bool WIDE>
__global__ void __launch_bounds__(kLzThreads) lanczos_step_kernel(LzArgs p) {
  extern __shared__ __align__(16) double lz_smem[];
  const int tid = threadIdx.x, b = blockIdx.x, G = p.workers;
  const int k = p.j + 1;
  double* part_a = p.partial;            // alpha, [G]
  double* part_h = p.partial + G;        // projections and norm, [k + 1][G]
  double* part_n = part_h + 64LL * G;    // norm, [G]
  if (b == G) {
    // ---- the tridiagonal: a_0 .. a_{j-1}, b_0 .. b_{j-1} are stored, a_j is the alpha of
    // this step
    TriShared& S = *reinterpret_cast<TriShared*>(lz_smem);
    __shared__ double tot[64];
    __shared__ double red[4][64];
    if (tid < k - 1) {
      S.a[tid] = p.tri[tid];
      S.b[tid] = tid < k - 2 ? p.tri[64 + tid] : p.beta_prev;
    }
    if (!lz_wait(p.bar, (unsigned)G + p.extra, p.wait_limit)) {
      if (tid == 0) p.out[4] = 1.0;
      return;
    }
    lz_totals<WIDE>(part_a, G, G, 1, tot, red);
    if (tid == 0) {
      S.a[k - 1] = tot[0];
      p.tri[k - 1] = tot[0];
      if (k > 1) p.tri[64 + k - 2] = p.beta_prev;
    }
    __syncthreads();
    tri_lowest(S, k);
    if (tid < k) p.tri[128 + tid] = S.z[tid];
    if (tid == 0) {
      p.out[2] = S.theta;
      p.out[3] = fabs(S.z[k - 1]);
    }
    return;
  }
  __shared__ double red[8][64];
  __shared__ double tot[64];
  __shared__ double h[64];
  if (b == 0 && tid < 2) p.bar_next[tid] = 0;
  const long long e0 = (long long)b * p.chunk;
  const int n = (int)min((long long)p.chunk, p.N - e0);
  double* x = p.w + e0;
  const double* V = p.V + e0;
  if (p.in_smem) {
    for (int e = tid; e < n; e += kLzThreads) lz_smem[e] = x[e];
    x = lz_smem;
    __syncthreads();
  }
  unsigned epoch = 0;
  // ---- alpha = <v_j, w>
  lz_dots(V + (long long)p.j * p.N, p.N, x, n, 1, false, part_a + b, G, red);
  lz_arrive(p.bar);
  if (!lz_wait(p.bar, ++epoch * G + p.extra, p.wait_limit)) {
    if (tid == 0) p.out[4] = 1.0;
    return;
  }
  lz_totals<WIDE>(part_a, G, G, 1, tot, red);
  const double alpha = tot[0];
  // ---- w -= alpha v_j + beta v_{j-1}
  {
    const double* vj = V + (long long)p.j * p.N;
    const double* vp = vj - p.N;
    for (int e = tid; e < n; e += kLzThreads) {
      double t = fma(-alpha, vj[e], x[e]);
      if (p.j > 0) t = fma(-p.beta_prev, vp[e], t);
      x[e] = t;
    }
    __syncthreads();
  }
  // ---- projections on all basis vectors, removed; a second time if they mattered
  double n2 = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    lz_dots(V, p.N, x, n, k, true, part_h + b, G, red);
    lz_arrive(p.bar);
    if (!lz_wait(p.bar, ++epoch * G + p.extra, p.wait_limit)) {
      if (tid == 0) p.out[4] = 1.0;
      return;
    }
    lz_totals<WIDE>(part_h, G, G, k + 1, tot, red);
    if (tid < k) h[tid] = tot[tid];
    const double n1 = tot[k];
    __syncthreads();
    int e = tid;
    for (; e + kLzThreads < n; e += 2 * kLzThreads) {   // two entries, eight vectors at a time
      double t0 = x[e], t1 = x[e + kLzThreads];
      int q = 0;
      for (; q + 8 <= k; q += 8) {
        double v[8], u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = __ldg(V + (long long)(q + i) * p.N + e);
          u[i] = __ldg(V + (long long)(q + i) * p.N + e + kLzThreads);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          t0 = fma(-h[q + i], v[i], t0);
          t1 = fma(-h[q + i], u[i], t1);
        }
      }
#pragma unroll 4
      for (; q < k; ++q) {
        t0 = fma(-h[q], __ldg(V + (long long)q * p.N + e), t0);
        t1 = fma(-h[q], __ldg(V + (long long)q * p.N + e + kLzThreads), t1);
      }
      x[e] = t0;
      x[e + kLzThreads] = t1;
    }
    if (e < n) {
      double t0 = x[e];
#pragma unroll 8
      for (int q = 0; q < k; ++q) t0 = fma(-h[q], __ldg(V + (long long)q * p.N + e), t0);
      x[e] = t0;
    }
    __syncthreads();
    lz_dots(x, 0, x, n, 0, true, part_n + b, G, red);
    lz_arrive(p.bar);
    if (!lz_wait(p.bar, ++epoch * G + p.extra, p.wait_limit)) {
      if (tid == 0) p.out[4] = 1.0;
      return;
    }
    lz_totals<WIDE>(part_n, G, G, 1, tot, red);
    n2 = tot[0];
    __syncthreads();
    if (!(n2 < 0.5 * n1)) break;
  }
  if (b == 0 && tid == 0) {
    p.out[0] = alpha;
    p.out[1] = n2;
  }
  if (p.write_next) {
    if (tid == 0) tot[1] = rsqrt(n2);
    __syncthreads();
    const double inv = tot[1];
    double* vn = p.V + (long long)k * p.N + e0;
    for (int e = tid; e < n; e += kLzThreads) vn[e] = x[e] * inv;
  }
}

__global__ void __launch_bounds__(kLzThreads)
dot_multi_partial(const double* __restrict__ V, long long ldv, int k,
                  const double* __restrict__ w, long long n, long long chunk,
                  double* __restrict__ partial) {
  __shared__ double red[8][64];
  const long long e0 = (long long)blockIdx.x * chunk;
  lz_dots(V + e0, ldv, w + e0, (int)min(chunk, n - e0), k, false, partial + blockIdx.x,
          gridDim.x, red);
}

__global__ void __launch_bounds__(32) reduce_partials(const double* __restrict__ partial, int nb,
                                                      double* __restrict__ out) {
  const int j = blockIdx.x;
  double acc = 0.0;
  for (int b = threadIdx.x; b < nb; b += 32) acc += partial[(long long)j * nb + b];
  acc = warp_sum_d(acc);
  if (threadIdx.x == 0) out[j] = acc;
}

}  // namespace

// Deterministic: fixed slices of at least 512 entries, sums in a fixed order.
void dot_multi(const double* V, long long ldv, int k, const double* w, long long n,
               double* partial, double* out, cudaStream_t s) {
  if (k <= 0) return;
  A2_REQUIRE(k <= 64, "at most 64 vectors");
  const long long chunk = std::max<long long>(512, (n + kReduceBlocks - 1) / kReduceBlocks);
  const int nb = (int)std::max<long long>(1, (n + chunk - 1) / chunk);
  A2_REQUIRE(chunk < (1LL << 30), "vector too long");
  dot_multi_partial<<<nb, kLzThreads, 0, s>>>(V, ldv, k, w, n, chunk, partial);
  A2_CHECK_LAUNCH();
  reduce_partials<<<k, 32, 0, s>>>(partial, nb, out);
  A2_CHECK_LAUNCH();
}

namespace {

__global__ void __launch_bounds__(kLzThreads)
tridiag_kernel(const double* a, const double* b, int k, double* out) {
  extern __shared__ __align__(16) double lz_smem[];
  TriShared& S = *reinterpret_cast<TriShared*>(lz_smem);
  const int tid = threadIdx.x;
  if (tid < k) S.a[tid] = a[tid];
  if (tid + 1 < k) S.b[tid] = b[tid];
  __syncthreads();
  tri_lowest(S, k);
  if (tid < k) out[2 + tid] = S.z[tid];
  if (tid == 0) {
    out[0] = S.theta;
    out[1] = k > 1 && S.state != 1 ? 1.0 : 0.0;
  }
}

// The slice of a worker: at least 128 entries (four warps' worth), at most what spreads N
// over all SMs but the one of the tridiagonal block.
void launch_step(double* V, double* w, long long N, int j, double beta_prev, bool write_next,
                 double* tri, double* partial, unsigned* bar, unsigned* bar_next, double* out,
                 unsigned wait_limit, unsigned extra, cudaStream_t s) {
  A2_REQUIRE(j >= 0 && j < 63, "Lanczos step: at most 63 basis vectors");
  constexpr size_t kSliceMax = 160 * 1024;
  static PerDevice<bool> set;
  set.at(current_device(), [] {
    for (const void* f : {(const void*)lanczos_step_kernel<false>,
                          (const void*)lanczos_step_kernel<true>})
      A2_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSliceMax));
    return true;
  });
  const int sms = device_sms();
  const int most = std::max(1, std::min(sms - 1, kReduceBlocks / 2));
  LzArgs p;
  p.V = V;
  p.w = w;
  p.N = N;
  p.j = j;
  long long chunk = std::max<long long>(128, (N + most - 1) / most);
  chunk = (chunk + 31) / 32 * 32;
  A2_REQUIRE(chunk < (1LL << 30), "Lanczos step: vector too long");
  p.chunk = (int)chunk;
  p.workers = (int)((N + chunk - 1) / chunk);
  p.in_smem = sizeof(double) * (size_t)chunk <= kSliceMax ? 1 : 0;
  p.write_next = write_next ? 1 : 0;
  p.beta_prev = beta_prev;
  p.tri = tri;
  p.partial = partial;
  p.bar = bar;
  p.bar_next = bar_next;
  p.out = out;
  p.wait_limit = wait_limit;
  p.extra = extra;
  const size_t smem = std::max(sizeof(TriShared),
                               p.in_smem ? sizeof(double) * (size_t)chunk : (size_t)0);
  void* args[] = {&p};
  const void* kernel = p.workers > 64 ? (const void*)lanczos_step_kernel<true>
                                      : (const void*)lanczos_step_kernel<false>;
  A2_CUDA(cudaLaunchCooperativeKernel(kernel, dim3(p.workers + 1), dim3(kLzThreads), args, smem, s));
  A2_CHECK_LAUNCH();
}

}  // namespace

void lanczos_step(double* V, double* w, long long N, int j, double beta_prev, bool write_next,
                  double* tri, double* partial, unsigned* bar, unsigned* bar_next,
                  double* out, cudaStream_t s) {
  launch_step(V, w, N, j, beta_prev, write_next, tri, partial, bar, bar_next, out, kLzWaitLimit, 0,
              s);
}

bool lanczos_selftest_timeout(double* partial, double* out, cudaStream_t s) {
  constexpr long long N = 4096;
  DevBuf v, tri, bar;
  v.ensure(sizeof(double) * 3 * N, s);
  tri.ensure(sizeof(double) * 192, s);
  bar.ensure(sizeof(unsigned) * 4, s);
  fill_zero(v.p, sizeof(double) * 3 * N, s);
  fill_zero(bar.p, sizeof(unsigned) * 4, s);
  double* V = v.as<double>();
  out[4] = 0.0;
  launch_step(V, V + 2 * N, N, 0, 0.0, false, tri.as<double>(), partial, bar.as<unsigned>(),
              bar.as<unsigned>() + 2, out, 1u << 14, 1, s);
  A2_CUDA(cudaStreamSynchronize(s));
  return out[4] != 0.0;
}

void tridiag_lowest(const double* a, const double* b, int k, double* out, cudaStream_t s) {
  A2_REQUIRE(k >= 1 && k <= 63, "tridiagonal size 1..63");
  tridiag_kernel<<<1, kLzThreads, sizeof(TriShared), s>>>(a, b, k, out);
  A2_CHECK_LAUNCH();
}

}  // namespace a2
