// FP64 passes of the Chebyshev iteration on the Schur complement (the gauge and the recurrence
// of gauge2d.cuh), 2D and 3D: one kernel for g' = N v, one for the update, a thread per point.
//
// These passes are bound by the FP64 pipe (1/64 of the FP32 rate): 26 (2D) and 34 (3D)
// operations a point and term.  Fused passes with halos, as in FP32, compute 1.3 to 2.8 times as
// many points; here none is computed twice, and the 7 field transfers of 16 bytes stay far under
// the pipe's time.  Measured per term: 512^2 x 3 54 us (fused 131, the pipe alone 34), 64^3 x 6 146 us
// (fused 316, the pipe alone 88).
#include "gauge2d.cuh"

namespace apfc {

namespace {

constexpr int kGX = 32, kGY = 8;

struct G64Amp {
  double n0, w[3];               // N
  double m0, mp, mb, u0, u[3];   // v_(n+1) = m0 v + mp v_(n-1) + mb (-b) + mc2 N g', N scaled
  double mith;
};
struct G64Param {
  G64Amp amp[kMaxJ];
  unsigned long long* prof;
  const double2* tab;
  const double* jd;  // Picard with the Jacobian: d(x), else null
  int J, nx, ny, nz, tx, ty, tz;
};

template <int DIM>
struct G64Point {
  int j, x, y, z;
  long long p;  // within the amplitude's field
  bool in;
};
// blockIdx.y = amplitude; blockIdx.x counts the tiles of all planes (a grid's other dimensions end at
// 65535, which long boxes have more of)
template <int DIM>
__device__ __forceinline__ G64Point<DIM> g64_point(const G64Param& c) {
  const unsigned ntx = (c.nx + kGX - 1) / kGX, row = blockIdx.x / ntx;
  G64Point<DIM> q;
  q.j = blockIdx.y;
  unsigned ty = row;
  q.z = 0;
  if constexpr (DIM == 3) {
    const unsigned nty = (c.ny + kGY - 1) / kGY;
    q.z = row / nty;
    ty = row - q.z * nty;
  }
  q.x = (blockIdx.x - row * ntx) * kGX + (threadIdx.x & 31);
  q.y = ty * kGY + (threadIdx.x >> 5);
  q.in = q.x < c.nx && q.y < c.ny;
  q.p = ((long long)q.z * c.ny + q.y) * c.nx + q.x;
  return q;
}

// The value of a neighbour across the periodic boundary: times the wrap's phase (sg -1: its
// conjugate).  A call, not an inlined product: inlined, the compiler predicates it in every warp,
// and predicated-off instructions still occupy the FP64 pipe (g' at 512^2 x 3: 43 us).
__noinline__ __device__ double2 g64_edge(const double2* wrap, double2 v, double sg) {
  double2 e = *wrap;
  e.y *= sg;
  return g_cmul(e, v);
}

// add + n0 c + sum_d w_d (minus + plus)
template <int DIM>
__device__ __forceinline__ double2 g64_stencil(const double2* f, const G64Point<DIM>& q, const G64Param& c,
                                               const double2* tab, double2 add, double n0,
                                               const double* w) {
  const long long plane = (long long)c.nx * c.ny;
  double2 m[DIM], p[DIM];
  double2 s = add;
  if (q.in) {
    s = q_fma(n0, f[q.p], s);
    m[0] = f[q.x == 0 ? q.p + c.nx - 1 : q.p - 1];
    p[0] = f[q.x + 1 == c.nx ? q.p - q.x : q.p + 1];
    m[1] = f[q.y == 0 ? q.p + (long long)(c.ny - 1) * c.nx : q.p - c.nx];
    p[1] = f[q.y + 1 == c.ny ? q.p - (long long)q.y * c.nx : q.p + c.nx];
    if constexpr (DIM == 3) {
      m[2] = f[q.z == 0 ? q.p + (c.nz - 1) * plane : q.p - plane];
      p[2] = f[q.z + 1 == c.nz ? q.p - q.z * plane : q.p + plane];
    }
  }
  const int at[3] = {q.x, q.y, q.z}, n[3] = {c.nx, c.ny, c.nz}, t0[3] = {0, c.tx, c.tx + c.ty};
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    if (q.in && at[d] == 0) m[d] = g64_edge(tab + t0[d] + n[d], m[d], -1.0);
    if (q.in && at[d] + 1 == n[d]) p[d] = g64_edge(tab + t0[d] + n[d], p[d], 1.0);
  }
#pragma unroll
  for (int d = 0; d < DIM; ++d) s = q_fma(w[d], q_add(m[d], p[d]), s);
  return s;
}

__device__ __forceinline__ double2 g64_phase(const G64Param& c, const double2* tab, int x, int y, int z, bool three) {
  double2 ph = g_cmul(tab[x], tab[c.tx + y]);
  return three ? g_cmul(ph, tab[c.tx + c.ty + z]) : ph;
}

// b = -e^{i phi.x} r, v_1 = b / theta
template <int DIM>
__global__ void __launch_bounds__(256) k_g64_start(const __grid_constant__ G64Param c, const double2* r,
                                                   double2* b, double2* v1, const KScal* ks) {
  const G64Point<DIM> q = g64_point<DIM>(c);
  dependent_wait();
  if (ks[q.j].iters == 0 || !q.in) return;
  const long long pts = (long long)c.nx * c.ny * c.nz, i = q.j * pts + q.p;
  const double2* tab = c.tab + (long long)q.j * (c.tx + c.ty + c.tz);
  const double2 w = g_cmul(g64_phase(c, tab, q.x, q.y, q.z, DIM == 3), r[i]);
  const double2 bn = make_double2(-w.x, -w.y);
  b[i] = bn;
  v1[i] = q_mul(c.amp[q.j].mith, bn);
}

template <int DIM>
__global__ void __launch_bounds__(256) k_g64_n(const __grid_constant__ G64Param c, const double2* v,
                                               double2* g, const KScal* ks, int pass) {
  const G64Point<DIM> q = g64_point<DIM>(c);
  dependent_wait();
  if (pass >= ks[q.j].iters) return;
  const long long o = (long long)q.j * c.nx * c.ny * c.nz;
  const double2* tab = c.tab + (long long)q.j * (c.tx + c.ty + c.tz);
  const G64Amp& a = c.amp[q.j];
  const double2 s = g64_stencil<DIM>(v + o, q, c, tab, make_double2(0.0, 0.0), a.n0, a.w);
  if (q.in) g[o + q.p] = s;
}

// vp: v_(n-1) in (first: zero), v_(n+1) out; an amplitude's last pass adds it to the state instead
template <int DIM>
__global__ void __launch_bounds__(256)
    k_g64_update(const __grid_constant__ G64Param c, const double2* g, const double2* v,
                 const double2* b, double2* vp, double2* x64, const KScal* ks,
                 int pass, int kid) {
  const G64Point<DIM> q = g64_point<DIM>(c);
  dependent_wait();
  const int npass = ks[q.j].iters;
  if (pass >= npass) return;
  const long long pts = (long long)c.nx * c.ny * c.nz, o = q.j * pts;
  if (c.prof != nullptr && q.p == 0 && q.in)
    atomicAdd(c.prof + kid, (unsigned long long)pts * 7ull * sizeof(double2));
  const double2* tab = c.tab + (long long)q.j * (c.tx + c.ty + c.tz);
  const G64Amp& a = c.amp[q.j];
  double2 s = make_double2(0.0, 0.0);
  if (q.in) {
    const double m0 = c.jd != nullptr ? fma(a.mb, c.jd[o + q.p], a.m0) : a.m0;  // a + d(x): Picard with the Jacobian
    s = q_fma(a.mb, b[o + q.p], q_mul(m0, v[o + q.p]));
    if (pass > 0) s = q_fma(a.mp, vp[o + q.p], s);
  }
  s = g64_stencil<DIM>(g + o, q, c, tab, s, a.u0, a.u);
  if (!q.in) return;
  if (pass + 1 < npass) {
    vp[o + q.p] = s;
    return;
  }
  const double2 un = g_cmul(g_conj(g64_phase(c, tab, q.x, q.y, q.z, DIM == 3)), s);
  double2* xp = x64 + 2 * o + pts + q.p;
  double2 xv = *xp;
  xv.x += un.x;
  xv.y += un.y;
  *xp = xv;
}

template <int DIM>
void pass64(const G64Param& in, const ChebBufs<double>& b, int pass, cudaStream_t s) {
  const int kid = kid_of<double>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  const dim3 grid((unsigned)((in.nx + kGX - 1) / kGX) * ((in.ny + kGY - 1) / kGY) * in.nz, in.J);
  double2* two[2] = {b.r[1], b.d[0]};  // v of even and odd passes; g' in d[1], b in u
  if (pass == 0) launch_dependent(k_g64_start<DIM>, grid, kGX * kGY, 0, s, in, b.r0, b.u, two[0], b.ks);
  launch_dependent(k_g64_n<DIM>, grid, kGX * kGY, 0, s, in, two[pass & 1], b.d[1], b.ks, pass);
  launch_dependent(k_g64_update<DIM>, grid, kGX * kGY, 0, s, in, b.d[1], two[pass & 1], b.u, two[1 - (pass & 1)], b.x64, b.ks, pass,
                                             kid);
}

}  // namespace

bool launch_gauge64(const OpCoef& c, const GaugeTab<double>& gt, const GaugeWeights& w, const ChebBufs<double>& b,
                    int pass, cudaStream_t s) {
  G64Param in;
  std::memset(&in, 0, sizeof(in));
  in.prof = c.prof;
  in.jd = c.jd;
  in.tab = gt.tab;
  in.tx = gt.tx;
  in.ty = gt.ty;
  in.tz = gt.tz;
  in.J = c.J;
  in.nx = c.nx;
  in.ny = c.ny;
  in.nz = c.nz;
  for (int j = 0; j < c.J; ++j) {
    G64Amp& a = in.amp[j];
    const double sk = -std::sqrt(c.kt[j]), c1 = w.c1[0][j], c2 = w.c2[0][j];
    a.n0 = sk * c.c0;
    a.u0 = -c2 * a.n0;
    for (int d = 0; d < c.dim; ++d) {
      a.w[d] = sk * gauge_w(c, j, d);
      a.u[d] = -c2 * a.w[d];
    }
    a.m0 = 1.0 + c1 - c2 * c.a[j];
    a.mp = -c1;
    a.mb = -c2;
    a.mith = -w.inv_theta[j];
  }
  if (c.dim == 3)
    pass64<3>(in, b, pass, s);
  else
    pass64<2>(in, b, pass, s);
  return true;
}

}  // namespace apfc
