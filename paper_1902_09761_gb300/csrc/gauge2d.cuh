// Chebyshev iteration on the Schur complement S = a + kt G_h^2 itself, 2D grids.
//
// G_h's symbol in dimension d, -(2/h^2)(1 - cos q) - (2k/h) sin q, is a shifted cosine:
//   G_h = c0 + sum_d w_d (e^{i phi_d} T_+d + e^{-i phi_d} T_-d),  w_d = sqrt(1 + (k_d h_d)^2) / h_d^2,
//   phi_d = atan(k_d h_d),
// T the shifts.  So v(x) = e^{i phi.x} u(x) (x the grid index) turns G_h into a real symmetric
// stencil, c0 + sum_d w_d (T_+ + T_-): 5 instead of 11 packed instructions a point.  The solve
// works on v; only values fetched across the periodic boundary need a factor, e^{+-i phi_d n_d}.
// Its first pass multiplies the residual by e^{i phi.x}, its last one the correction by the
// conjugate.
//
// Without the preconditioner p(D)^2 an application of S costs two stencil stages instead of 2 + 2M.
// At the spacings amplitudes need (about h <= pi/2: few points per atom) S is hardly worse
// conditioned than S p(D)^2 (16.5 against 15.4 at h = pi/2, dt = 1, degree 1), so the plain
// iteration needs fewer stages; schur_build (schur.cu) compares the two and takes cheb2d.cuh's on
// finer grids.
//
// k_gauge2d makes NI terms of the iteration (Saad, Alg. 12.1, in the two-vector form
// v_(n+1) = v_n + c1 (v_n - v_(n-1)) + c2 (b - S v_n)) in one pass: stages
//   g' = N v_n | v_(n+1) = v_n + c1 (v_n - v_(n-1)) - c2 (a v_n - b + N g'),   N = -sqrt(kt) G_h,
// streamed down the rows of strips as in cheb2d.cuh: at step t stage s forms its row t - s from the
// row the previous stage has just formed, two rows in registers and x-neighbours from a two-row
// shared-memory ring; one barrier a row.  Reads v_n, v_(n-1), b; writes v_(n+NI), v_(n+NI-1): 40
// bytes a point in FP32 for NI terms.  START (v_1 = b / theta, v_0 = 0) reads the residual and
// writes b too; an amplitude's last pass adds the correction to the FP64 state.
#pragma once
#include "cheb2d.cuh"

namespace apfc {

namespace {

template <typename T, int NI_, int V_, int NT_, int PF_, bool START_>
struct GaugeShape {
  static constexpr int NI = NI_, V = V_, NT = NT_, PF = PF_;
  static constexpr bool START = START_;
  static constexpr int S = 2 * NI;                  // stages = halo radius
  static constexpr int NC = NT * V;                 // columns of a strip
  static constexpr int RW = NT + 2;                 // row of one ring part
  static constexpr int SLOTS = PF + 1;
  // own-column ring of b: START writes row t at step t, otherwise row t - 2 lands there for step
  // t; stage 2(i + 1) reads row t - 2(i + 1)
  static constexpr int DB = START ? 2 * NI + 1 : PF + 2 * NI - 1;
  static constexpr int NU = START ? 1 : 2;          // staged rows besides b: the residual, or v_n and v_(n-1)
  static constexpr size_t ring_elems = (size_t)S * 2 * V * RW;
  static constexpr size_t b_elems = (size_t)DB * NC;
  static constexpr size_t stage_elems = (size_t)NU * SLOTS * NC;
  static constexpr size_t smem = sizeof(cplx<T>) * (ring_elems + b_elems + stage_elems);
};

// Coefficients of one amplitude in the field precision: N = n0 + nx (l + r) + ny (u + d); a; the
// terms' weights c1 and -c2; START's -1/theta (b is kept negated).
template <typename T>
struct GaugeAmp {
  T n0, nx, ny, a;
  T c1[kGaugeMaxNI], mc2[kGaugeMaxNI];
  T mith;
};
template <typename T>
struct GaugeParam {
  GaugeAmp<T> amp[kMaxJ];
  unsigned long long* prof;
  const cplx<T>* tab;   // [J][tx + ty]: e^{i phi_x i}, i < tx, then e^{i phi_y i}
  int J, tx, ty;
};

// explicitly rounded: every instantiation of the kernel gives the same bits
__device__ __forceinline__ float2 g_cmul(float2 z, float2 a) {
  return make_float2(__fmaf_rn(z.x, a.x, -__fmul_rn(z.y, a.y)), __fmaf_rn(z.x, a.y, __fmul_rn(z.y, a.x)));
}
__device__ __forceinline__ double2 g_cmul(double2 z, double2 a) {
  return make_double2(fma(z.x, a.x, -(z.y * a.y)), fma(z.x, a.y, z.y * a.x));
}
template <typename C>
__device__ __forceinline__ C g_conj(C z) {
  z.y = -z.y;
  return z;
}
// e^m for a unit complex e and a small integer m
template <typename C>
__device__ __forceinline__ C g_pow(C e, int m, C one) {
  if (m < 0) e = g_conj(e), m = -m;
  C r = one;
  for (; m > 0; --m) r = g_cmul(r, e);
  return r;
}

template <typename T, int NI, int V, int NT, int PF, int MINB, bool START, class TAB>
__global__ void __launch_bounds__(NT, MINB)
    k_gauge2d(const __grid_constant__ GaugeParam<T> c, ChebGeom g, const cplx<T>* v_in, const cplx<T>* vp_in,
              cplx<T>* v_out, cplx<T>* vp_out, cplx<T>* b_io, double2* x64, const KScal* ks, int pass, int kid,
              const __grid_constant__ TAB tab) {
  using SH = GaugeShape<T, NI, V, NT, PF, START>;
  using C = cplx<T>;
  constexpr int S = SH::S, NC = SH::NC, RW = SH::RW, DB = SH::DB, U = 4;
  extern __shared__ __align__(16) unsigned char gauge_smem[];
  C* ring = reinterpret_cast<C*>(gauge_smem);  // [S][2][V][RW]: inputs of stages 1 .. S
  C* bring = ring + SH::ring_elems;            // [DB][NC]
  C* stg = bring + SH::b_elems;                // [SLOTS][NU][NC]

  int sx, sy, j;
  if constexpr (std::is_same<TAB, ChebTab>::value) {
    const ChebRun& q = tab.run[blockIdx.y];
    const int b = blockIdx.x;
    if (b >= q.nblk) return;
    g.nx = q.nx;
    g.ny = q.ny;
    g.Ly = q.Ly;
    g.nstrips = q.nstrips;
    g.nsegs = q.nsegs;
    g.pts = q.pts;
    sx = b % q.nstrips;
    sy = (b / q.nstrips) % q.nsegs;
    j = b / (q.nstrips * q.nsegs);
    v_in += q.foff;
    if constexpr (!START) vp_in += q.foff;
    v_out += q.foff;
    vp_out += q.foff;
    b_io += q.foff;
    x64 += q.xoff;
    ks += (long long)q.run * c.J;
  } else {
    sx = blockIdx.x;
    sy = blockIdx.y;
    j = blockIdx.z;
  }
  const int npass = ks[j].iters;
  if (pass >= npass) return;
  const bool last = pass + 1 == npass;
  const int t = threadIdx.x;
  if (c.prof != nullptr && sx == 0 && sy == 0 && t == 0) {
    const unsigned long long f = sizeof(C), rd = START ? f : 3 * f, wr = START ? 3 * f : 2 * f;
    atomicAdd(c.prof + kid, (unsigned long long)g.pts * (rd + (last ? 2 * sizeof(double2) : wr)));
  }
  {
    const long long o = (long long)j * g.pts;
    v_in += o;
    if constexpr (!START) vp_in += o;
    v_out += o;
    vp_out += o;
    b_io += o;
    x64 += 2 * o + g.pts;  // the eta-part of amplitude j
  }
  const GaugeAmp<T>& q_ = c.amp[j];
  const T n0 = q_.n0, nwx = q_.nx, nwy = q_.ny, aa = q_.a;
  const C* tabx = c.tab + (long long)j * (c.tx + c.ty);
  const C* taby = tabx + c.tx;

  const C zero = mkc<T>((T)0, (T)0), one = mkc<T>((T)1, (T)0);
  for (int i = t; i < (int)(SH::ring_elems + SH::b_elems); i += NT) ring[i] = zero;
  __syncthreads();  // the first fetches land in b's ring, over zeros that other threads have stored

  // columns of this thread: V t .. V t + V - 1 of the strip; a column beyond the grid is the
  // periodic image times e^{i phi_x nx m}
  const int x_first = sx * g.wv - S;
  int gxc[V], mx[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int X = x_first + V * t + v;
    int x = X % g.nx;
    if (x < 0) x += g.nx;
    gxc[v] = x;
    mx[v] = (X - x) / g.nx;
  }
  bool colw = false;
  C colf[V];
  {
    const C ex = tabx[g.nx];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      colf[v] = g_pow(ex, mx[v], one);
      colw = colw || mx[v] != 0;
    }
  }
  const bool vec = V == 1 || (g.nx & 1) == 0;
  const int xo = sx * g.wv + (V * t - S);  // first owned column
  const bool col_own = V * t >= S && V * t < NC - S && xo < g.nx;
  [[maybe_unused]] const bool own1 = col_own && xo + 1 < g.nx;
  C pcol[V];  // e^{i phi_x x} of the columns (START: of their unwrapped positions)
#pragma unroll
  for (int v = 0; v < V; ++v) {
    pcol[v] = one;
    if (START || last) pcol[v] = START ? g_cmul(tabx[gxc[v]], colf[v]) : tabx[gxc[v]];
  }
  const int y0 = sy * g.Ly;
  const int y_end = min(g.ny, y0 + g.Ly);
  const int steps = (y_end - y0) + 2 * S;
  const long long nx = g.nx, wrap = (long long)(g.ny - 1) * nx;
  // row of the next fetch and of the current step, and the row factors of rows t and t - 2
  int fy = (y0 - S) % g.ny;
  if (fy < 0) fy += g.ny;
  const C ey = taby[g.ny];
  int my = (y0 - S - fy) / g.ny;  // wraps of row t
  int cy = fy;                    // row t
  C rf = g_pow(ey, my, one);
  [[maybe_unused]] int fy2 = (y0 - S - 2) % g.ny, cy2, my2;
  if (fy2 < 0) fy2 += g.ny;
  cy2 = fy2;
  my2 = (y0 - S - 2 - fy2) / g.ny;
  [[maybe_unused]] C rf2 = g_pow(ey, my2, one);
  const C* f_v = v_in + fy * nx;
  [[maybe_unused]] const C* f_p = vp_in + fy2 * nx;
  [[maybe_unused]] const C* f_b = b_io + fy2 * nx;
  auto fetch = [&](C* dst, const C* p) {
    if constexpr (V == 1) {
      cheb_cp_async(dst, p + gxc[0]);
    } else {
      if (vec) {
        cheb_cp_async16(dst, p + gxc[0]);
      } else {
        cheb_cp_async(dst, p + gxc[0]);
        cheb_cp_async(dst + 1, p + gxc[V - 1]);
      }
    }
  };
  auto issue = [&](int tf, int slot, int bslot) {
    C* st = stg + (size_t)slot * SH::NU * NC + V * t;
    if (tf < steps) {
      fetch(st, f_v);
      f_v += fy + 1 == g.ny ? -wrap : nx;
      fy = cheb_wrap(fy, g.ny);
      if constexpr (!START) {
        fetch(st + NC, f_p);
        fetch(bring + (size_t)bslot * NC + V * t, f_b);
        f_p += fy2 + 1 == g.ny ? -wrap : nx;
        f_b += fy2 + 1 == g.ny ? -wrap : nx;
        fy2 = cheb_wrap(fy2, g.ny);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  auto store = [&](C* p, const C (&v)[V]) {
    if constexpr (V == 1) {
      p[0] = v[0];
    } else {
      if (vec) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
      } else {
        p[0] = v[0];
        if (own1) p[1] = v[1];
      }
    }
  };
  // addresses of the last stage's row (START's b: of row t)
  C* o_v = v_out + (long long)(y0 - 2 * S) * nx + xo;
  C* o_p = vp_out + (long long)(y0 - 2 * S) * nx + xo;
  [[maybe_unused]] C* o_b = b_io + (long long)(y0 - S) * nx + xo;
  double2* o_x = x64 + (long long)(y0 - 2 * S) * nx + xo;

  // own-column history of the stage inputs: HV[i] v_(n+i) (four rows, v_(n+i-1) is read two
  // stages later), HG[i] g'
  C HV[NI][4][V], HG[NI][2][V];
#pragma unroll
  for (int i = 0; i < NI; ++i)
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
      for (int k = 0; k < 4; ++k) HV[i][k][v] = zero;
      HG[i][0][v] = HG[i][1][v] = zero;
    }
#pragma unroll
  for (int tf = 0; tf < PF; ++tf) issue(tf, tf, tf);
  __syncthreads();

  int slot = 0, islot = PF;
  int b0 = 0;                       // START: ring slot of row t; else of the row (t - 2) landed for step t
  int bis = START ? 0 : PF % DB;    // b's slot of the next fetch
  for (int t0 = 0; t0 < steps; t0 += U) {
#pragma unroll
    for (int ph = 0; ph < U; ++ph) {
      const int tt = t0 + ph;
      if (tt >= steps) break;
      if constexpr (U % SH::SLOTS == 0) slot = ph % SH::SLOTS, islot = (ph + PF) % SH::SLOTS;
      issue(tt + PF, islot, bis);
      asm volatile("cp.async.wait_group %0;\n" ::"n"(PF));
      C* st = stg + (size_t)slot * SH::NU * NC + V * t;
      C F[V];  // row of the value formed last
      C FV[NI][V];
      [[maybe_unused]] C vp[V];
      if constexpr (START) {
        const C prow = g_cmul(taby[cy], rf);
        C bt[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const C r = g_cmul(g_cmul(prow, pcol[v]), st[v]);
          bt[v] = mkc<T>(-r.x, -r.y);
          F[v] = q_mul(q_.mith, bt[v]);  // v_1 = b / theta
          bring[(size_t)b0 * NC + V * t + v] = bt[v];
        }
        if (!last && col_own && tt >= S && tt < steps - S) store(o_b, bt);
      } else {
#pragma unroll
        for (int v = 0; v < V; ++v) F[v] = st[v], vp[v] = st[NC + v];
        if (colw || my != 0 || my2 != 0) {  // beyond the grid: the image's phase
          C* bb = bring + (size_t)b0 * NC + V * t;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            F[v] = g_cmul(g_cmul(rf, colf[v]), F[v]);
            const C f2 = g_cmul(rf2, colf[v]);
            vp[v] = g_cmul(f2, vp[v]);
            bb[v] = g_cmul(f2, bb[v]);
          }
        }
      }
      auto put = [&](int q, const C (&f)[V]) {
        C* w = ring + ((size_t)q * 2 + (ph & 1)) * V * RW + t + 1;
#pragma unroll
        for (int v = 0; v < V; ++v) w[v * RW] = f[v];
      };
      put(0, F);
      C vl[V];  // v_(n+NI-1) at the last stage's row
      for_stages<0, NI - 1>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        C G[V];
        // g' = N v_(n+i) at row tt - 2i - 1
        {
          const C* rq = ring + ((size_t)(2 * i) * 2 + ((ph + 1) & 1)) * V * RW + t + 1;
          const C L = rq[(V - 1) * RW - 1], R = rq[1];
          const C(&cc)[V] = HV[i][(ph + 3) & 3];
          const C(&uu)[V] = HV[i][(ph + 2) & 3];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const C l = v == 0 ? L : cc[v > 0 ? v - 1 : 0], r = v == V - 1 ? R : cc[v < V - 1 ? v + 1 : 0];
            G[v] = q_fma(nwy, q_add(uu[v], F[v]), q_fma(nwx, q_add(l, r), q_mul(n0, cc[v])));
          }
          put(2 * i + 1, G);
        }
        // v_(n+i+1) at row tt - 2i - 2
        {
          const C* rq = ring + ((size_t)(2 * i + 1) * 2 + ((ph + 1) & 1)) * V * RW + t + 1;
          const C L = rq[(V - 1) * RW - 1], R = rq[1];
          const C(&cc)[V] = HG[i][(ph + 1) & 1];
          const C(&uu)[V] = HG[i][ph & 1];
          int bs = b0 - (START ? 2 * (i + 1) : 2 * i);
          if (bs < 0) bs += DB;
          const C* bp = bring + (size_t)bs * NC + V * t;
          C W[V];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const C l = v == 0 ? L : cc[v > 0 ? v - 1 : 0], r = v == V - 1 ? R : cc[v < V - 1 ? v + 1 : 0];
            const C vc = HV[i][(ph + 2) & 3][v];
            // r^ = a v - b + N g'  (b is kept negated)
            const C rh = q_fma(nwy, q_add(uu[v], G[v]),
                               q_fma(nwx, q_add(l, r), q_fma(n0, cc[v], q_fma(aa, vc, bp[v]))));
            C old;
            if constexpr (i == 0)
              old = START ? zero : vp[v];
            else
              old = HV[i - 1][ph & 3][v];
            W[v] = q_fma(q_.mc2[i], rh, q_fma(q_.c1[i], q_sub(vc, old), vc));
            if constexpr (i == NI - 1) vl[v] = vc;
          }
#pragma unroll
          for (int v = 0; v < V; ++v) HG[i][ph & 1][v] = G[v];
          if constexpr (i + 1 < NI) put(2 * i + 2, W);
          // v_(n+i)'s new row enters its history at the end of the step: the next term still
          // reads the row it replaces
#pragma unroll
          for (int v = 0; v < V; ++v) {
            FV[i][v] = F[v];
            F[v] = W[v];
          }
        }
      });
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int v = 0; v < V; ++v) HV[i][ph & 3][v] = FV[i][v];
      // the last stage's row
      if (col_own && tt >= 2 * S) {
        if (!last) {
          store(o_v, F);
          store(o_p, vl);
        } else {
          const C prow = taby[y0 + tt - 2 * S];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            if (v > 0 && !own1) break;
            const C un = g_cmul(g_conj(g_cmul(prow, pcol[v])), F[v]);
            double2 xv = o_x[v];
            if constexpr (sizeof(T) == 4) {  // exact widening by integer operations
              xv.x += f2d(un.x);
              xv.y += f2d(un.y);
            } else {
              xv.x += un.x;
              xv.y += un.y;
            }
            o_x[v] = xv;
          }
        }
      }
      o_v += nx;
      o_p += nx;
      if constexpr (START) o_b += nx;
      o_x += nx;
      if (cy + 1 == g.ny) {
        cy = 0;
        ++my;
        rf = g_cmul(rf, ey);
      } else {
        ++cy;
      }
      if constexpr (!START) {
        if (cy2 + 1 == g.ny) {
          cy2 = 0;
          ++my2;
          rf2 = g_cmul(rf2, ey);
        } else {
          ++cy2;
        }
        bis = bis + 1 == DB ? 0 : bis + 1;
      }
      b0 = b0 + 1 == DB ? 0 : b0 + 1;
      if constexpr (U % SH::SLOTS != 0) {
        slot = slot + 1 == SH::SLOTS ? 0 : slot + 1;
        islot = islot + 1 == SH::SLOTS ? 0 : islot + 1;
      }
      __syncthreads();
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
}

template <typename T>
GaugeParam<T> gauge_param(const OpCoef& c, const GaugeTab<T>& gt, const GaugeWeights& w, int terms) {
  GaugeParam<T> in;
  std::memset(&in, 0, sizeof(in));
  in.prof = c.prof;
  in.tab = gt.tab;
  in.tx = gt.tx;
  in.ty = gt.ty;
  in.J = c.J;
  for (int j = 0; j < c.J; ++j) {
    GaugeAmp<T>& a = in.amp[j];
    const double sk = -std::sqrt(c.kt[j]);
    a.n0 = (T)(sk * c.c0);
    a.nx = (T)(sk * gauge_w(c, j, 0));
    a.ny = (T)(sk * gauge_w(c, j, 1));
    a.a = (T)c.a[j];
    for (int i = 0; i < terms; ++i) {
      a.c1[i] = (T)w.c1[i][j];
      a.mc2[i] = (T)(-w.c2[i][j]);
    }
    a.mith = (T)(-w.inv_theta[j]);
  }
  return in;
}

// One pass over one grid or, with bl, over every run of a batch.
template <typename T, int NI, int V, int NT, int PF, int MINB, bool START>
bool launch_gauge_pass(const OpCoef& c, const GaugeTab<T>& gt, const GaugeWeights& w, int Ly, const ChebBufs<T>& b,
                       int pass, cudaStream_t s, const BatchLaunch* bl, int take = 0) {
  using SH = GaugeShape<T, NI, V, NT, PF, START>;
  static_assert(NI <= kGaugeMaxNI && SH::S % V == 0 && (SH::NC - 2 * SH::S) % V == 0, "strips start on a pair");
  const int kid = kid_of<T>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  const GaugeParam<T> in = gauge_param<T>(c, gt, w, NI);
  // fields: v in r / d by pass parity (r0 the residual), b in u
  const int cur = pass & 1;
  const cplx<T>* vin = START ? b.r0 : b.r[cur];
  if (bl == nullptr) {
    auto kern = k_gauge2d<T, NI, V, NT, PF, MINB, START, ChebNoTab>;
    static const cudaError_t attr =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (attr != cudaSuccess) return false;
    const ChebGeom g = cheb_geom(c.nx, c.ny, SH::S, SH::NC, Ly);
    kern<<<dim3(g.nstrips, g.nsegs, c.J), NT, SH::smem, s>>>(in, g, vin, b.d[cur], b.r[1 - cur], b.d[1 - cur], b.u,
                                                            b.x64, b.ks, pass, kid, ChebNoTab{});
    return true;
  }
  if constexpr (sizeof(T) == 8) {
    return false;  // batched runs are FP32
  } else {
    auto kern = k_gauge2d<T, NI, V, NT, PF, MINB, START, ChebTab>;
    static const cudaError_t attr =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (attr != cudaSuccess) return false;
    for (int r0 = 0; r0 < bl->R; r0 += kChebRuns) {
      ChebTab tab;
      int maxblk = 0;
      const int nr = cheb_table(*bl, r0, SH::S, SH::NC, Ly, c.J, tab, maxblk, take);
      if (maxblk == 0) continue;
      kern<<<dim3(maxblk, nr), NT, SH::smem, s>>>(in, ChebGeom{0, 0, 0, SH::NC - 2 * SH::S, 0, 0, 0}, vin, b.d[cur],
                                                  b.r[1 - cur], b.d[1 - cur], b.u, b.x64, b.ks, pass, kid, tab);
    }
    return true;
  }
}

}  // namespace

}  // namespace apfc
