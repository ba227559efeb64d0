// The Schur-complement solve of constant-coefficient systems: spectrum of S p(D)^2, the weights
// of the Chebyshev iteration, the outer residual r = b - (a + kt G_h^2) eta on 2D grids, and the
// device-side choice of each amplitude's number of passes (cheb2d.cuh runs them).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "apfc_internal.cuh"
#include "dfloat.cuh"
#include "host_common.h"
#include "resid_point.cuh"

namespace apfc {

// ---------------------------------------------------------------------------
// Host: spectrum and weights
// ---------------------------------------------------------------------------
namespace {

// Symbol of S p(D)^2 at wave numbers q (radians per grid point) for amplitude j.
struct Symbol {
  const OpCoef& c;
  const double* h;
  int m;
  double theta[kMaxJ], delta[kMaxJ], tsig[kMaxJ];
  static double cheb(int n, double x) {
    double t0 = 1.0, t1 = x;
    if (n == 0) return t0;
    for (int k = 1; k < n; ++k) {
      const double t2 = 2.0 * x * t1 - t0;
      t0 = t1;
      t1 = t2;
    }
    return t1;
  }
  Symbol(const OpCoef& c_, const double* h_, int m_) : c(c_), h(h_), m(m_) {
    double lapmax = 0.0;
    for (int d = 0; d < c.dim; ++d) lapmax += 4.0 / (h[d] * h[d]);
    for (int j = 0; j < c.J; ++j) {
      const double lo = c.sD[j], hi = c.sD[j] + c.mu[j] * lapmax;
      theta[j] = 0.5 * (hi + lo);
      delta[j] = 0.5 * (hi - lo);
      tsig[j] = cheb(m + 1, theta[j] / delta[j]);
    }
  }
  // from K = -L_h's symbol and g = G_h's
  double of(int j, double K, double g) const {
    const double d = c.sD[j] + c.mu[j] * K;
    const double p = (1.0 - cheb(m + 1, (theta[j] - d) / delta[j]) / tsig[j]) / d;
    return (c.a[j] + c.kt[j] * g * g) * p * p;
  }
  // Of all wave numbers with the same K = 2 sum_d (1 - cos q_d) / h_d^2 (d takes no other part in
  // S p(D)^2), those where A = 2 sum_d (k_d / h_d) sin q_d is largest: sin is concave in 1 - cos, so
  // there is one such point for every K, tan q_d = k_d h_d / lambda, and lambda from infinity to
  // minus infinity makes the curve of them.  At lambda = 0 a dimension with k_d = 0 runs from 0 to
  // pi.  s in [0, 3]: lambda > 0, that stretch, lambda < 0.
  void curve(int j, double s, double* K, double* A) const {
    const double th = 1.57079632679489661923 * (s < 1.0 ? s : s < 2.0 ? 1.0 : s - 1.0);
    const double sn = std::sin(th), cs = s < 1.0 || s > 2.0 ? std::cos(th) : 0.0;
    *K = *A = 0.0;
    for (int d = 0; d < c.dim; ++d) {
      const double ih2 = 1.0 / (h[d] * h[d]), kh = std::fabs(c.kh[j][d]) / ih2 * sn;  // |k_d| h_d sin(theta)
      double sq = 0.0, cq = s < 1.0 ? 1.0 : s < 2.0 ? std::cos(3.14159265358979323846 * (s - 1.0)) : -1.0;
      if (kh > 1e-12) {
        const double ir = 1.0 / std::sqrt(kh * kh + cs * cs);
        sq = kh * ir;
        cq = cs * ir;
      }
      *K += 2.0 * ih2 * (1.0 - cq);
      *A += 2.0 * std::fabs(c.kh[j][d]) * sq;
    }
  }
};

}  // namespace

// Bounds of the spectrum of S_j p(D)^2 over all wave numbers.  G_h's symbol is -K - A, and -A occurs
// with every A: for each K the symbol lies between its values at |G| = max(0, K - A) and K + A with A
// at its largest, so the extremes over the curve of these points bound it.  The curve is sampled, and
// every extremum of the samples narrowed down (golden section); 1% to spare on both sides.  Against
// dense samples of the symbol (1024^2 wave numbers, h 0.2 to 1.5, dt 0.1 to 100, degrees 1 to 4) both
// ends are within 0.4%.  A 32 x 32 sample improved by a pattern search left the least eigenvalue up to
// 1.5 times too high: the symbol has a narrow valley along G = 0.
void schur_spectrum(const OpCoef& c, const apfc_grid& grid, int m, double* lmin, double* lmax) {
  const Symbol sym(c, grid.h, m);
  constexpr int n = 128;  // samples of each stretch
  constexpr double kGolden = 0.61803398874989484820;
  std::vector<double> at, v[2];
  for (int j = 0; j < c.J; ++j) {
    bool free = false;
    for (int d = 0; d < c.dim; ++d) free = free || std::fabs(c.kh[j][d]) * grid.h[d] * grid.h[d] <= 1e-12;
    at.clear();  // where every k_d is nonzero, lambda = 0 is the one point s = 1, and s = 2 + follows on it
    for (int i = 0; i <= 3 * n; ++i)
      if (free || i <= n || i > 2 * n) at.push_back((double)i / n);
    auto value = [&](int w, double s) {
      double K, A;
      sym.curve(j, s, &K, &A);
      const double g = w == 0 ? std::max(0.0, K - A) : K + A;
      return w == 0 ? sym.of(j, K, g) : -sym.of(j, K, g);
    };
    const int ns = (int)at.size();
    double ext[2] = {1e300, 1e300};
    for (int w = 0; w < 2; ++w) {
      v[w].resize(ns);
      for (int i = 0; i < ns; ++i) v[w][i] = value(w, at[i]);
      for (int i = 0; i < ns; ++i) {
        if ((i > 0 && v[w][i - 1] < v[w][i]) || (i + 1 < ns && v[w][i + 1] < v[w][i])) continue;
        ext[w] = std::min(ext[w], v[w][i]);
        const int i0 = std::max(i - 1, 0), i1 = std::min(i + 1, ns - 1);
        double lo = at[i0], hi = at[i1];
        const bool jump = !free && lo <= 1.0 && hi > 2.0;
        if (jump) hi -= 1.0;
        for (int it = 0; it < 30; ++it) {
          const double x = hi - kGolden * (hi - lo), y = lo + kGolden * (hi - lo);
          const double fx = value(w, jump && x > 1.0 ? x + 1.0 : x), fy = value(w, jump && y > 1.0 ? y + 1.0 : y);
          ext[w] = std::min(ext[w], std::min(fx, fy));
          (fx < fy ? hi : lo) = fx < fy ? y : x;
        }
      }
    }
    lmin[j] = 0.99 * ext[0];
    lmax[j] = -1.01 * ext[1];
  }
}

// S's own bounds are those of its symbol a + kt g^2, g = c0 + 2 sum_d w_d cos(q_d + phi_d) (which
// takes the value 0).  A term of the plain iteration costs about half of one with p(D)^2 (measured
// at 4096^2: 123 against 245 us in FP32), so the latter is taken where it halves their number;
// below a condition number of 40 it cannot.  No limit on its number of terms: a step
// took 1 / 2.4 of BiCGStab's time or less at each of the 170 points it serves among 256^2 and 1024^2,
// h 0.2 to 0.7, dt 0.5 to 20, degrees 1 to 4 and both precisions (up to 1500 terms a step).
bool schur_build(const OpCoef& c, const apfc_grid& grid, int m, SchurCoef& s) {
  SchurCoef q{};
  auto finish = [&](SchurCoef& r) {
    for (int j = 0; j < c.J; ++j) {
      if (!(r.lmin[j] > 0.0) || !(r.lmax[j] > r.lmin[j]) || !std::isfinite(r.lmax[j])) return false;
      r.lnrate[j] = std::acosh((r.lmax[j] + r.lmin[j]) / (r.lmax[j] - r.lmin[j]));
    }
    return true;
  };
  double slow = 1e300, kappa = 0.0;
  s = SchurCoef{};
  s.plain = true;
  for (int j = 0; j < c.J; ++j) {
    double g = -c.c0;
    for (int d = 0; d < c.dim; ++d) g += 2.0 * gauge_w(c, j, d);
    s.lmin[j] = c.a[j];
    s.lmax[j] = c.a[j] + c.kt[j] * g * g;
    kappa = std::max(kappa, s.lmax[j] / s.lmin[j]);
  }
  s.kappa = kappa;
  if (!finish(s)) return false;
  if (c.dim == 3) {
    // no preconditioned variant: on fine grids, where a solve would need about 100 terms, an
    // iteration of BiCGStab with its preconditioner costs 7 (FP64) to 11 (FP32) of them
    for (int j = 0; j < c.J; ++j)
      if (s.lnrate[j] < 0.1) return false;
    return true;
  }
  if (!(kappa > 40.0)) return true;
  schur_spectrum(c, grid, m, q.lmin, q.lmax);
  if (!finish(q)) return true;
  double slow_q = 1e300;
  for (int j = 0; j < c.J; ++j) {
    slow = std::min(slow, s.lnrate[j]);
    slow_q = std::min(slow_q, q.lnrate[j]);
  }
  q.kappa = kappa;
  if (slow_q > 2.0 * slow) s = q;
  return true;
}

// S + d(x), d real within [dmin, dmax]: both ends of the spectrum move by no more than d's.  False
// (NaN included) where it may not be positive, or where a solve would need about 100 terms; an
// iteration of BiCGStab with its preconditioner costs about 12 of them (512^2: 100 of its
// iterations 10 ms, three terms 12 us).
bool schur_widen(const SchurCoef& s, const double* dmin, const double* dmax, int J, SchurCoef& out) {
  if (!s.plain) return false;
  out = s;
  out.kappa = 0.0;
  for (int j = 0; j < J; ++j) {
    out.lmin[j] += dmin[j];
    out.lmax[j] += dmax[j];
    if (!(out.lmin[j] > 0.0) || !(out.lmax[j] > out.lmin[j]) || !std::isfinite(out.lmax[j])) return false;
    out.lnrate[j] = std::acosh((out.lmax[j] + out.lmin[j]) / (out.lmax[j] - out.lmin[j]));
    if (!(out.lnrate[j] >= 0.1)) return false;
    out.kappa = std::max(out.kappa, out.lmax[j] / out.lmin[j]);
  }
  return true;
}

// Saad, Alg. 12.1: rho_0 = 1/sigma, d_0 = z/theta; rho_k = 1/(2 sigma - rho_(k-1)),
// d_k = rho_k rho_(k-1) d_(k-1) + (2 rho_k / delta) z_k: weights of d_first .. d_(first+count-1).
namespace {
template <typename F>
void chebyshev_weights(const SchurCoef& s, int j, int first, int count, F&& put) {
  const double theta = 0.5 * (s.lmax[j] + s.lmin[j]), delta = 0.5 * (s.lmax[j] - s.lmin[j]), sigma = theta / delta;
  double rho = 1.0 / sigma;
  for (int k = 1; k < first + count; ++k) {
    const double rn = 1.0 / (2.0 * sigma - rho);
    if (k >= first) put(k - first, rn * rho, 2.0 * rn / delta);
    rho = rn;
  }
}
}  // namespace
// Pass 0 makes d_0 and d_1, pass k >= 1 the next ni terms.
ChebPass schur_pass(const SchurCoef& s, int J, int pass, int ni) {
  ChebPass cp;
  std::memset(&cp, 0, sizeof(cp));
  for (int j = 0; j < J; ++j) {
    cp.inv_theta[j] = 2.0 / (s.lmax[j] + s.lmin[j]);
    chebyshev_weights(s, j, pass == 0 ? 1 : 2 + (pass - 1) * ni, pass == 0 ? 1 : ni, [&](int i, double c1, double c2) {
      cp.c1[i][j] = c1;
      cp.c2[i][j] = c2;
    });
  }
  return cp;
}
// Pass 0 makes d_0 = r / theta and ni terms, later ones ni.
GaugeWeights gauge_weights(const SchurCoef& s, int J, int pass, int ni) {
  GaugeWeights w;
  std::memset(&w, 0, sizeof(w));
  for (int j = 0; j < J; ++j) {
    w.inv_theta[j] = 2.0 / (s.lmax[j] + s.lmin[j]);
    chebyshev_weights(s, j, 1 + pass * ni, ni, [&](int i, double c1, double c2) {
      w.c1[i][j] = c1;
      w.c2[i][j] = c2;
    });
  }
  return w;
}

int schur_terms(double tin, double lnrate) {
  const double x = 1.0 / tin;
  const double need = x > 1.0 ? std::log(x + std::sqrt(x * x - 1.0)) / lnrate : 0.0;
  return need < 1e9 ? std::max(2, (int)std::ceil(need)) : 1000000000;
}

// ---------------------------------------------------------------------------
// Device: norms and passes
// ---------------------------------------------------------------------------
namespace {

constexpr float kSchurLast64 = 0.4f, kSchurLast32 = 1.f / 16.f, kSchurLeast = 0.03f, kSchurOnce = 0.2f;

// Sums the partials of ||r||^2 and ||b||^2 (have bits 1, 2) of amplitude blockIdx.x of the run
// and sets the number of passes of its next solve.
__global__ void __launch_bounds__(256) k_schur_plan(const __grid_constant__ SchurPlan p, KScal* ks, const RunGeom* rg) {
  const int run = rg != nullptr ? blockIdx.x / p.J : 0, j = blockIdx.x - run * p.J;
  dependent_wait();
  const double* part = p.part;
  int npart = p.npart;
  long long ss = p.slot_stride, sj = p.amp_stride;
  if (rg != nullptr) {
    if (p.by_run) {  // the residual kernel's layout [run][J][2][npart of the run]
      npart = rg[run].npart_r;
      part += rg[run].part_off_r;
      ss = npart;
      sj = 2ll * npart;
    } else {
      part += (long long)run * p.J * sj;
    }
  }
  __shared__ double sh[2][8];
  for (int q = 0; q < 2; ++q) {
    double v = 0.0;
    if (p.have & (1 << q))
      for (int i = threadIdx.x; i < npart; i += 256) v += part[j * sj + q * ss + (long long)i * p.elem];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  KScal& k = ks[blockIdx.x];
  double s[2] = {0.0, 0.0};
  for (int q = 0; q < 2; ++q)
    for (int w = 0; w < 8; ++w) s[q] += sh[q][w];
  if (p.have & 1) k.rnorm2 = s[0];
  if (p.have & 2) k.bnorm2 = s[1];
  const double r2 = k.rnorm2, b2 = k.bnorm2;
  k.iters = 0;
  const bool more = isfinite(r2) && isfinite(b2) && r2 > p.tol * p.tol * b2;
  if (p.follow) {
    // A stencil residual may exceed the tolerance where the first check's, formed pointwise, met it:
    // the refinement ended there, and what was queued behind it must leave the state alone.
    bool any = false;
    for (int i = 0; i < p.J; ++i) any = any || ks[i].active != 0;
    if (!any) return;
  } else {
    k.active = more;
  }
  if (!more) return;
  // The residual that a Chebyshev solve leaves sits in the low end of the spectrum, where it
  // weighs most in the error: the solve that is to meet the outer tolerance goes further below
  // it than a Krylov solve has to for the same error.  A solve need not stop at tol_inner where that
  // would leave the tolerance within a factor of five: passes end past their aim, and such solves met
  // the tolerance by chance with 0.3 to 0.8 of it left (error of two steps at 1024^2 1.0e-11, now
  // 8.6e-13; of the gradient of 12 steps at 256^2 2.6e-10, now 3.9e-11).
  // (FP32 is plenty for a number of terms; the FP64 pipe's square roots and logarithms took 3 us.)
  const float tol = (float)p.tol, tol_inner = (float)p.tol_inner;
  const float want = b2 > 0.0 ? tol * sqrtf((float)(b2 / r2)) : tol_inner;
  float tin;
  if (p.fp64) {
    tin = kSchurLast64 * (b2 > 0.0 ? want : tol);
  } else {
    tin = fminf(0.5f, fmaxf(tol_inner, 0.25f * want));
    if (want >= kSchurOnce * tol_inner) tin = fminf(tin, fmaxf(kSchurLeast * tol_inner, kSchurLast32 * want));
  }
  const float x = 1.f / tin;
  const float need = x > 1.f ? logf(x + sqrtf(x * x - 1.f)) / (float)p.lnrate[j] : 0.f;
  const float n = fminf(fmaxf(2.f, ceilf(need)), 1e9f);
  k.iters = min(max(1, (int)ceilf((n - p.t0) / p.ni)), p.max_pass);
}

// e^{i phi_d i}: blockIdx.y = amplitude
template <typename T>
__global__ void k_gauge_table(cplx<T>* tab, const __grid_constant__ OpCoef c, int tx, int ty, int tz) {
  const int j = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x, n = tx + ty + tz;
  if (i >= n) return;
  const int d = i < tx ? 0 : (i < tx + ty ? 1 : 2), k = i - (d > 0 ? tx : 0) - (d > 1 ? ty : 0);
  double sn, cs;
  sincos(atan2(c.kh[j][d], c.ih2[d]) * k, &sn, &cs);
  tab[(long long)j * n + i] = mkc<T>((T)cs, (T)sn);
}

// ---------------------------------------------------------------------------
// Outer residual r = b - a eta - kt G_h (G_h eta) on 2D grids, streamed down the rows: a block
// owns 64 columns (60 of them valid) and a segment of rows; at step t a thread forms zeta =
// G_h eta at row t - 1 and r at row t - 2 of its column, the y-neighbours in registers (the row
// below is the one just formed), the x-neighbours from two-row shared-memory rings.  Every
// double is split once.  Writes zeta into the state (the solve never reads it, so it always
// belongs to the latest eta), r as RT, optionally r in FP64, and per block the sums ||r||^2 and,
// on request, ||b||^2.  JAC: a + d(x) in place of a (Picard with the Jacobian).  Where
// SchurCoef::kappa asks for FP64 arithmetic resid_f64.cu's kernels run instead.
// ---------------------------------------------------------------------------
// Two warps a block, twelve blocks per SM (80 registers): bound by the packed FP32 instructions (about
// 190 a point, that pipe busy 59 per cent of the time) and the conversions' integer ones (44).  us, three amplitudes, at
// 128^2 / 256^2 / 512^2 / 1024^2 / 1531 x 997 / 4096^2: 8.7 / 15 / 30 / 88 / 115 / 1023; four warps in
// six blocks 10.6 / 15 / 33 / 88 / 116 / 1017, in four (126 registers) 12.5 / 15 / 33 / 91 / 120 / 1052;
// eight in two 15 / 23 / 42 / 109 / 142 / 1147; one in 24 8.7 / 15 / 29 / 87 / 119 / 1078; tiles of
// 28 x 28 held by a block 8.8 / 13 / 31 / 95 / 125 / 1220.
constexpr int kRsNT = 64, kRsPF = 2, kRsV = kRsNT - 4;

__device__ __forceinline__ void rs_copy16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src));
}

template <bool JAC>
__global__ void __launch_bounds__(kRsNT, 12)
    k_resid_schur2d(const double2* b, double2* x, float2* __restrict__ r_out, double2* __restrict__ r64,
                    double* __restrict__ part, const __grid_constant__ OpCoef c, int Ly, int nstrips, int nsegs,
                    int want_b, const RunGeom* rg) {
  __shared__ float4 ring[2][2][kRsNT + 2];             // eta, zeta
  __shared__ double2 stg[kRsPF + 1][2][kRsNT];     // eta, b rows in flight
  __shared__ double shn[2][kRsNT / 32];
  const int j = blockIdx.y, t = threadIdx.x;
  dependent_wait();
  int nx = c.nx, ny = c.ny;
  long long pts = c.pts, fo = 0;
  if (rg != nullptr) {
    const RunGeom& q = rg[blockIdx.z];
    nx = q.nx;
    ny = q.ny;
    pts = q.pts;
    b += q.elem_off;
    x += q.elem_off;
    fo = q.field_off;
    part += q.part_off_r;
    Ly = q.rows_r;
    nstrips = (nx + kRsV - 1) / kRsV;
    nsegs = (ny + Ly - 1) / Ly;
  }
  const int npart = nstrips * nsegs;
  if ((int)blockIdx.x >= npart) return;
  const int sy = blockIdx.x / nstrips, sx = blockIdx.x - sy * nstrips;
  if (c.prof != nullptr && blockIdx.x == 0 && t == 0)
    atomicAdd(c.prof + KID_RESID_REFINE,
              (unsigned long long)pts * (3 * sizeof(double2) + sizeof(float2) +
                                         (r64 != nullptr ? sizeof(double2) : 0)));
  double2* zt = x + 2LL * j * pts;
  const double2* et = zt + pts;
  const double2* bt = b + (2LL * j + 1) * pts;
  fo += (long long)j * pts;
  r_out += fo;
  if (r64 != nullptr) r64 += fo;

  const ResidCoef<2> q = resid_coef<2>(c, j);
  LaneC ma = lane_c(c.a[j], -1.f, -1.f);
  const PDF zero{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};

  const int x_first = sx * kRsV - 2;
  int gxx = (x_first + t) % nx;
  if (gxx < 0) gxx += nx;
  const int xo = x_first + t;
  const bool col_own = t >= 2 && t < kRsNT - 2 && xo < nx;
  const int y0 = sy * Ly, rows = min(ny, y0 + Ly) - y0, steps = rows + 4;
  int fy = (y0 - 2) % ny;
  if (fy < 0) fy += ny;
  auto issue = [&](int tf, int slot) {
    if (tf < steps) {
      rs_copy16(&stg[slot][0][t], et + (long long)fy * nx + gxx);
      fy = fy + 1 == ny ? 0 : fy + 1;
      const int lr = tf - 2;  // row of r: local rows 2 .. rows + 1
      if (col_own && lr >= 2) rs_copy16(&stg[slot][1][t], bt + (long long)(y0 + lr - 2) * nx + xo);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  if (t == 0) {
    for (int k = 0; k < 2; ++k)
      for (int p = 0; p < 2; ++p) ring[k][p][0] = ring[k][p][kRsNT + 1] = pdf_pack(zero);
  }
  for (int k = 0; k < 2; ++k)
    for (int p = 0; p < 2; ++p) ring[k][p][t + 1] = pdf_pack(zero);
  for (int tf = 0; tf < kRsPF; ++tf) issue(tf, tf);
  __syncthreads();
  PDF e1 = zero, e2 = zero, z1 = zero, z2 = zero;  // rows formed 1 and 2 steps ago
  float rr = 0.f, bb = 0.f;
  int slot = 0, islot = kRsPF, par = 0;
  for (int tt = 0; tt < steps; ++tt) {
    issue(tt + kRsPF, islot);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kRsPF));
    const int lr = tt - 2;
    [[maybe_unused]] double jd = 0.0;  // JAC: on its way while zeta is formed
    if constexpr (JAC) {
      if (col_own && lr >= 2) jd = c.jd[(long long)j * pts + (long long)(y0 + lr - 2) * nx + xo];
    }
    const PDF e0 = pdf_split(stg[slot][0][t]);
    ring[0][par][t + 1] = pdf_pack(e0);
    // zeta at row tt - 1
    const PDF el = pdf_unpack(ring[0][par ^ 1][t]), er = pdf_unpack(ring[0][par ^ 1][t + 2]);
    PDF z0;
    double2 zd;
    {
      PAcc a;
      a.init(zero, c.zero);
      a.fma(q.g0.h, q.g0.l, e1);
      a.fma(q.gl[0].h, q.gl[0].l, pdf_add(er, el));
      a.fma(q.gl[1].h, q.gl[1].l, pdf_add(e0, e2));
      a.fma(q.ga[0].h, q.ga[0].l, pdf_swap(pdf_sub(er, el)));
      a.fma(q.ga[1].h, q.ga[1].l, pdf_swap(pdf_sub(e0, e2)));
      a.result(z0.h, z0.l);
      zd = make_double2(df_to_d(DF{z0.h.x, z0.l.x}), df_to_d(DF{z0.h.y, z0.l.y}));
    }
    ring[1][par][t + 1] = pdf_pack(z0);
    const int lz = tt - 1;
    if (col_own && lz >= 2 && lz < rows + 2) zt[(long long)(y0 + lz - 2) * nx + xo] = zd;
    // r at row tt - 2
    if (lr >= 2) {
      const PDF zl = pdf_unpack(ring[1][par ^ 1][t]), zr = pdf_unpack(ring[1][par ^ 1][t + 2]);
      if (col_own) {
        const double2 bv = stg[slot][1][t];
        const long long p = (long long)(y0 + lr - 2) * nx + xo;
        {
          const PDF bp = pdf_split(bv);
          PAcc a;
          a.init(bp, c.zero);
          a.fma(q.k0.h, q.k0.l, z1);
          a.fma(q.kl[0].h, q.kl[0].l, pdf_add(zr, zl));
          a.fma(q.kl[1].h, q.kl[1].l, pdf_add(z0, z2));
          a.fma(q.ka[0].h, q.ka[0].l, pdf_swap(pdf_sub(zr, zl)));
          a.fma(q.ka[1].h, q.ka[1].l, pdf_swap(pdf_sub(z0, z2)));
          if constexpr (JAC) ma = lane_c(c.a[j] + jd, -1.f, -1.f);
          a.fma(ma.h, ma.l, e2);
          float2 f, l;
          a.result(f, l);
          r_out[p] = f;
          if (r64 != nullptr) r64[p] = make_double2(df_to_d(DF{f.x, l.x}), df_to_d(DF{f.y, l.y}));
          rr = fmaf(f.x, f.x, fmaf(f.y, f.y, rr));
          if (want_b) bb = fmaf(bp.h.x, bp.h.x, fmaf(bp.h.y, bp.h.y, bb));
        }
      }
    }
    e2 = e1;
    e1 = e0;
    z2 = z1;
    z1 = z0;
    slot = slot == kRsPF ? 0 : slot + 1;
    islot = islot == kRsPF ? 0 : islot + 1;
    par ^= 1;
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  double rrd = (double)rr, bbd = (double)bb;
  for (int o = 16; o > 0; o >>= 1) {
    rrd += __shfl_xor_sync(0xffffffffu, rrd, o);
    bbd += __shfl_xor_sync(0xffffffffu, bbd, o);
  }
  if ((t & 31) == 0) shn[0][t >> 5] = rrd, shn[1][t >> 5] = bbd;
  __syncthreads();
  if (t < 2) {
    double v = 0.0;
    for (int w = 0; w < kRsNT / 32; ++w) v += shn[t][w];
    part[(2LL * j + t) * npart + blockIdx.x] = v;
  }
}

}  // namespace

// Rows per segment of the passes: each step of a block costs about the same, so the heights ceil(ny / s)
// are compared by (what the busiest multiprocessor has to run) x (rows + 2S).  One or two of its blocks
// together cost 1, a full round of them 1.56 (wide strips 1.5), and blocks drift apart (0.2).  Two
// steps, ms by height: 4096^2 512 23.5, 342 25.7, 296 24.4, 256 23.3, 205 24.4, 171 23.1, 164 22.8, 147
// 24.0, 128 23.3, 64 23.8; 3000^2 334 14.2, 160 13.7, 100 13.4, 64 13.7; 2048^2 187 7.2, 128 6.6, 100
// 7.6, 64 6.8; 1024^2 64 2.65, 47 2.37, 32 2.23.
int schur_auto_rows(const SchurCoef& sc, const int* nx, const int* ny, int n, int J, int m, int elem_bytes, int tile,
                    int sms) {
  const bool f32 = elem_bytes == 8, wide = f32 && sc.plain && (tile == 2 || tile == 4 || tile == 5);
  const int S = sc.plain ? 2 * (f32 ? kGaugeNI32 : kGaugeNI64) : (f32 && m == 1 ? 8 : 2 + 2 * m);
  const int NC = wide ? 256 : 128;
  const int res = wide ? 3 : 6;       // resident blocks per SM
  const double thr = wide ? 0.5 : 0.26;  // a step of one block of a full round, a lone block's being 1
  int most = 1;
  for (int i = 0; i < n; ++i) most = std::max(most, ny[i]);
  double best = 1e300;
  int best_rows = std::min(most, 128);
  for (int seg = (most + 511) / 512; seg <= most; ++seg) {
    const int rows = (most + seg - 1) / seg;
    if (rows < 4 && seg > 1) break;
    long long blocks = 0;
    for (int i = 0; i < n; ++i)
      blocks += (long long)((nx[i] + NC - 2 * S - 1) / (NC - 2 * S)) * ((ny[i] + rows - 1) / rows) * J;
    const long long per = (blocks + sms - 1) / sms;  // blocks of the busiest SM
    const long long full = per / res, rest = per - full * res;
    const double round = res * thr;
    double t = full * round + 0.2;
    if (rest > 0) t += std::max(1.0, 1.0 + (rest - 2) * (round - 1.0) / (res - 2));
    t *= std::min(rows, most) + 2 * S + 4;
    if (t < best) best = t, best_rows = rows;
  }
  return best_rows;
}

// Rows per segment: two rounds of the resident blocks (3648 = 2 x 12 x 152 multiprocessors), at least
// eight rows (and four of halo), or four where eight give fewer than two blocks to a multiprocessor
// (304; 128^2: 12.3 against 8.7 us).  Constants, not the device's count: a batch and its runs alone
// split alike.
int schur_resid_rows(int nx, int ny, int J) {
  const long long strips = (nx + kRsV - 1) / kRsV;
  const long long rows = (long long)ny * strips * J / 3648;
  const long long least = (ny + 7) / 8 * strips * J < 304 ? 4 : 8;
  return (int)std::min<long long>(128, std::max(least, rows));
}
int schur_resid_parts(int nx, int ny, int J) {
  const int Ly = schur_resid_rows(nx, ny, J);
  return ((nx + kRsV - 1) / kRsV) * ((ny + Ly - 1) / Ly);
}

template <typename T>
void launch_resid_schur2d(const double2* b, double2* x, cplx<T>* r, double2* r64, double* part, const OpCoef& c,
                          bool want_b, bool f64, cudaStream_t s, const BatchLaunch* bl) {
  const int Ly = schur_resid_rows(c.nx, c.ny, c.J);
  const int ns = (c.nx + kRsV - 1) / kRsV, ng = (c.ny + Ly - 1) / Ly;
  dim3 grid(ns * ng, c.J);
  if (bl != nullptr) {
    int most = 0;
    for (int i = 0; i < bl->R; ++i) most = std::max(most, bl->host[i].npart_r);
    grid = dim3(most, c.J, bl->R);
  }
  if constexpr (sizeof(T) == 4) {
    if (!f64) {
      ProfScope ps_(KID_RESID_REFINE, s);
      const auto k = c.jd != nullptr ? k_resid_schur2d<true> : k_resid_schur2d<false>;
      launch_dependent(k, grid, kRsNT, 0, s, b, x, r, r64, part, c, Ly, ns, ng, want_b, bl != nullptr ? bl->dev : nullptr);
      return;
    }
  }
  launch_resid64<T>(b, x, r, r64, part, c, want_b, grid.x, s, bl);
}
template void launch_resid_schur2d<float>(const double2*, double2*, float2*, double2*, double*, const OpCoef&, bool,
                                          bool, cudaStream_t, const BatchLaunch*);
template void launch_resid_schur2d<double>(const double2*, double2*, double2*, double2*, double*, const OpCoef&, bool,
                                           bool, cudaStream_t, const BatchLaunch*);

template <typename T>
void launch_gauge_table(cplx<T>* tab, const OpCoef& c, int tx, int ty, int tz, cudaStream_t s) {
  k_gauge_table<T><<<dim3((tx + ty + tz + 127) / 128, c.J), 128, 0, s>>>(tab, c, tx, ty, tz);
}
template void launch_gauge_table<float>(float2*, const OpCoef&, int, int, int, cudaStream_t);
template void launch_gauge_table<double>(double2*, const OpCoef&, int, int, int, cudaStream_t);

// Passes that no FP32 solve of plan p exceeds (one to spare for the rounding of the device's logarithm).
int schur_most_passes(const SchurPlan& p) {
  long long n = 1;
  for (int j = 0; j < p.J; ++j) {
    const long long terms = schur_terms(kSchurLeast * p.tol_inner, p.lnrate[j]);
    n = std::max(n, (terms - p.t0 + p.ni - 1) / p.ni + 1);
  }
  return (int)std::min<long long>(n, p.max_pass);
}

void launch_schur_plan(const SchurPlan& p, KScal* ks, cudaStream_t s, const BatchLaunch* bl) {
  ProfScope ps_(kid_of<double>(KID_FINALIZE), s);
  launch_dependent(k_schur_plan, (bl ? bl->R : 1) * p.J, 256, 0, s, p, ks, bl ? bl->dev : nullptr);
}

}  // namespace apfc
