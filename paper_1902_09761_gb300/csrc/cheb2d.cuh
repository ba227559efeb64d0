// Preconditioned Chebyshev iteration on the Schur complement, 2D grids, constant coefficients.
//
// The first block row of Eq. linear_system2 with M = I, zeta = G_h eta, holds exactly on the
// solver's iterates, so the block system A_j (zeta, eta) = (0, b) is
//   S_j eta = b,   S_j = a_j + kt_j G_h^2                  (its Schur complement),
// and the preconditioner of Eq. preconditioner acts on it as p(D)^2, p(D) the Chebyshev
// approximant of D^{-1} (f = beta2 - kt G_h beta1 obeys f(A P^{-1} beta) = S p(D)^2 f(beta)).
// All operators are constant-coefficient periodic stencils: they commute, S p(D)^2 is Hermitian
// positive definite, and its spectrum is known from the stencils' symbols (schur_spectrum in
// schur.cu).  So the solve needs no inner products: the Chebyshev semi-iteration (Saad, Alg. 12.1)
//   d_0 = p^2 r_0 / theta,  u = d_0;   r -= S d,  d = c1 d + c2 p^2 r,  u += d
// reaches a given reduction in a number of applications known beforehand.
//
// k_cheb2d runs NI of these iterations in one pass over the grid (START: d_0 and the first one):
// a chain of radius-1 stencil stages per iteration,
//   g = G d | r' = r - a d - kt G g | M stages w = p r' | M stages z = p w, d' = c1 d + c2 z.
// A block owns a strip of NC columns (S = the number of stages of them halo on each side) and a
// segment of rows and streams down the rows.  At step t stage s works on row t - s: its input's
// row below (t - s + 1) is the value the previous stage has just formed in the same thread, the
// row itself and the one above are in registers, and the x-neighbours come from a two-row
// shared-memory ring written one step earlier, so one barrier per row serves every stage.
// A value needed again LM = 2 + 2M rows later (d for c1 d, r for the next iteration) stays in
// registers when LM = 4 (the loop is unrolled by four, so that the history never moves) and in
// an own-column shared-memory ring otherwise.  Global rows are fetched PF rows ahead (cp.async).
//
// Bytes per point of a pass, FP32: reads r, d, u, writes r', d', u' (48) for NI iterations
// (NI = 2 at M = 1); START reads r and writes r', d', u (32); an amplitude's last pass adds the
// sum u to the FP64 state instead (24 + 32).
#pragma once
#include "acc.cuh"
#include "apfc_internal.cuh"
#include "dfloat.cuh"

#include <algorithm>
#include <cstring>
#include <type_traits>

namespace apfc {

namespace {

__device__ __forceinline__ float2 q_add(float2 a, float2 b) { return p_add(a, b); }
__device__ __forceinline__ float2 q_sub(float2 a, float2 b) { return p_sub(a, b); }
__device__ __forceinline__ float2 q_mul(float s, float2 a) { return p_mul(make_float2(s, s), a); }
__device__ __forceinline__ float2 q_fma(float s, float2 a, float2 b) { return p_fma(make_float2(s, s), a, b); }
__device__ __forceinline__ double2 q_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 q_sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 q_mul(double s, double2 a) { return make_double2(s * a.x, s * a.y); }
__device__ __forceinline__ double2 q_fma(double s, double2 a, double2 b) {
  return make_double2(fma(s, a.x, b.x), fma(s, a.y, b.y));
}
// a + i b
__device__ __forceinline__ float2 q_addi(float2 a, float2 b) {
  return make_float2(__fsub_rn(a.x, b.y), __fadd_rn(a.y, b.x));
}
__device__ __forceinline__ double2 q_addi(double2 a, double2 b) { return make_double2(a.x - b.y, a.y + b.x); }

template <typename C>
__device__ __forceinline__ void cheb_cp_async(C* dst, const C* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(C) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src));
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void cheb_cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src));
}

template <int I, int N, typename F>
__device__ __forceinline__ void for_stages(F&& f) {
  if constexpr (I <= N) {
    f(std::integral_constant<int, I>{});
    for_stages<I + 1, N>(f);
  }
}

template <typename T, int M_, int NI_, int V_, int NT_, int PF_, bool START_>
struct ChebShape {
  static constexpr int M = M_, V = V_, NT = NT_, PF = PF_;
  static constexpr bool START = START_;
  static constexpr int SI = 2 + 2 * M;             // stages of one iteration
  static constexpr int PRE = START ? 2 * M : 0;    // START: stages of d_0 = p^2 r / theta
  static constexpr int NIT = START ? 1 : NI_;      // iterations of the pass
  static constexpr int S = PRE + NIT * SI;         // stages = halo radius
  static constexpr int LM = SI;                    // rows until a delayed value's second use
  static constexpr bool REG = LM == 4;             // delayed values in registers
  static constexpr int U = 4;                      // unrolling of the row loop
  static constexpr int NC = NT * V;                // columns of a strip
  static constexpr int HD = REG ? 4 : 2;           // rows of own-column history in registers
  static constexpr int NF = START ? 1 : 3;         // fetched rows: the input, r, u
  static constexpr int SLOTS = PF + 1;
  static constexpr int RW = NT + 2;                // row of one ring part (padding left and right)
  static constexpr int NDEL = START ? 2 : 2 * NIT - 1;  // delayed quantities (see del_index)
  static constexpr size_t ring_elems = (size_t)S * 2 * V * RW;
  static constexpr size_t keep_elems = REG ? 0 : (size_t)NDEL * LM * NC;
  static constexpr size_t stage_elems = (size_t)NF * SLOTS * NC;
  static constexpr size_t smem = sizeof(cplx<T>) * (ring_elems + keep_elems + stage_elems);
  // stage q's output (q = 0: the input) needed again LM rows later: the index of its delay
  // line, or -1
  __host__ __device__ static constexpr int del_index(int q) {
    if (START) return q == 0 ? 0 : (q == PRE ? 1 : -1);
    const int it = q / SI, pos = q % SI;
    if (it >= NIT) return -1;
    if (pos == 0) return 2 * it;                          // d_it
    if (pos == 2 && it + 1 < NIT) return 2 * it + 1;      // r_(it+1)
    return -1;
  }
};

struct ChebGeom {
  int nx, ny, Ly, wv, nstrips, nsegs;
  long long pts;
};

// Coefficients of one amplitude in the field precision, formed on the host (a conversion from
// FP64 at the start of every block costs more than a row of a short segment):
//   G = g0 + gx (l + r) + gy (u + d) + i (ax (r - l) + ay (d - u)); k*, b*: -kt G; ma = -a;
//   M = 1: p = p0 + px (l + r) + py (u + d) (the Chebyshev approximant pa + pb D collapsed);
//   M > 1: D itself in p*, and the weights of Saad's recurrence;
//   c1, c2: this pass's iterations d = c1 d + c2 p^2 r; ith_out: START's d_0 = p^2 r / theta.
template <typename T, int M>
struct ChebAmp {
  T g0, gx, gy, ax, ay, k0, kx, ky, bx, by, ma, p0, px, py;
  T ith, w1[M], w2[M];
  T c1[2], c2[2], ith_out;
};
template <typename T, int M>
struct ChebParam {
  ChebAmp<T, M> amp[kMaxJ];
  unsigned long long* prof;
  int J;
};
template <typename T, int M>
ChebParam<T, M> cheb_param(const OpCoef& c, const ChebStep* w, const ChebPass& cp) {
  ChebParam<T, M> q;
  std::memset(&q, 0, sizeof(q));
  q.prof = c.prof;
  q.J = c.J;
  for (int j = 0; j < c.J; ++j) {
    ChebAmp<T, M>& a = q.amp[j];
    const double kt = c.kt[j];
    a.g0 = (T)c.c0, a.gx = (T)c.ih2[0], a.gy = (T)c.ih2[1], a.ax = (T)c.kh[j][0], a.ay = (T)c.kh[j][1];
    a.k0 = (T)(-kt * c.c0), a.kx = (T)(-kt * c.ih2[0]), a.ky = (T)(-kt * c.ih2[1]);
    a.bx = (T)(-kt * c.kh[j][0]), a.by = (T)(-kt * c.kh[j][1]), a.ma = (T)(-c.a[j]);
    const double D0 = c.sD[j] - c.mu[j] * c.c0, Dx = -c.mu[j] * c.ih2[0], Dy = -c.mu[j] * c.ih2[1];
    double pa = 0.0, pb = 1.0;
    if (M == 1) pa = c.inv_theta[j] * (1.0 + w[0].c1[j]) + w[0].c2[j], pb = -w[0].c2[j] * c.inv_theta[j];
    a.p0 = (T)(pa + pb * D0), a.px = (T)(pb * Dx), a.py = (T)(pb * Dy);
    a.ith = (T)c.inv_theta[j];
    for (int k = 0; k < M; ++k) a.w1[k] = (T)w[k].c1[j], a.w2[k] = (T)w[k].c2[j];
    for (int i = 0; i < 2; ++i) a.c1[i] = (T)cp.c1[i][j], a.c2[i] = (T)cp.c2[i][j];
    a.ith_out = (T)cp.inv_theta[j];
  }
  return q;
}

// Batched runs: geometry of up to kChebRuns runs of one launch in the kernel parameters.
constexpr int kChebRuns = 64;
struct ChebRun {
  long long pts, foff, xoff;  // points; first element in a field array, in the state block
  int nx, ny, Ly, nstrips, nsegs, nblk, run, pad;
};
struct ChebTab {
  ChebRun run[kChebRuns];
};
struct ChebNoTab {};

__device__ __forceinline__ int cheb_wrap(int y, int n) { return y + 1 == n ? 0 : y + 1; }

// Grid: (nstrips, nsegs, J), or for batched runs (blocks of the largest run, runs).
// ks[j].iters: passes of amplitude j in this solve; pass `pass` (0 = START) of it runs while
// pass < iters, and the last one adds u to the state x64.
template <typename T, int M, int NI, int V, int NT, int PF, bool START, class TAB>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 && M == 1) ? 256 / NT : 1)
    k_cheb2d(const __grid_constant__ ChebParam<T, M> c, ChebGeom g, const cplx<T>* r_in, const cplx<T>* d_in,
             cplx<T>* r_out, cplx<T>* d_out, cplx<T>* u_io, double2* x64, const KScal* ks, int pass, int kid,
             const __grid_constant__ TAB tab) {
  using SH = ChebShape<T, M, NI, V, NT, PF, START>;
  using C = cplx<T>;
  constexpr int S = SH::S, NC = SH::NC, U = SH::U, LM = SH::LM, RW = SH::RW, PRE = SH::PRE, SI = SH::SI;
  extern __shared__ __align__(16) unsigned char cheb_smem[];
  C* ring = reinterpret_cast<C*>(cheb_smem);       // [S][2][V][RW]
  C* keep = ring + SH::ring_elems;                 // [NDEL][LM][NC]
  C* stg = keep + SH::keep_elems;                  // [SLOTS][NF][NC]

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
    r_in += q.foff;
    if constexpr (!START) d_in += q.foff;
    r_out += q.foff;
    d_out += q.foff;
    u_io += q.foff;
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
    const unsigned long long rd = START ? 1 : 3, f = sizeof(C);
    atomicAdd(c.prof + kid, (unsigned long long)g.pts * (last ? rd * f + 2 * sizeof(double2) : (rd + 3) * f));
  }
  {
    const long long o = (long long)j * g.pts;
    r_in += o;
    if constexpr (!START) d_in += o;
    r_out += o;
    d_out += o;
    u_io += o;
    x64 += 2 * o + g.pts;  // the eta-part of amplitude j
  }
  const ChebAmp<T, M>& q_ = c.amp[j];
  const T g0 = q_.g0, gx = q_.gx, gy = q_.gy, ax = q_.ax, ay = q_.ay;
  const T k0 = q_.k0, kx = q_.kx, ky = q_.ky, bx = q_.bx, by = q_.by, ma = q_.ma;
  const T p0 = q_.p0, px = q_.px, py = q_.py;

  const C zero = mkc<T>((T)0, (T)0);
  for (int i = t; i < (int)(SH::ring_elems + SH::keep_elems); i += NT) ring[i] = zero;

  // columns of this thread: V t .. V t + V - 1 of the strip
  const int x_first = sx * g.wv - S;
  int gx0 = (x_first + V * t) % g.nx;
  if (gx0 < 0) gx0 += g.nx;
  [[maybe_unused]] const int gx1 = cheb_wrap(gx0, g.nx);
  // even rows: a pair never straddles the periodic boundary and is 16-byte aligned
  const bool vec = V == 1 || (g.nx & 1) == 0;
  const int xo = sx * g.wv + (V * t - S);  // first owned column
  const bool col_own = V * t >= S && V * t < NC - S && xo < g.nx;
  [[maybe_unused]] const bool own1 = col_own && xo + 1 < g.nx;
  const int y0 = sy * g.Ly;
  const int y_end = min(g.ny, y0 + g.Ly);
  const int steps = (y_end - y0) + 2 * S;

  // row addresses, uniform over the block, advanced by one row per step: fetched rows wrap
  // around the grid, owned rows (u, the outputs) are used only where they lie on it
  auto grow = [&](int lr) {
    int y = (y0 - S + lr) % g.ny;
    return y < 0 ? y + g.ny : y;
  };
  const long long nx = g.nx, wrap = (long long)(g.ny - 1) * nx;
  int fy_in = grow(0);
  [[maybe_unused]] int fy_r = grow(-2);
  const C* f_in = (START ? r_in : d_in) + fy_in * nx;
  [[maybe_unused]] const C* f_r = r_in + fy_r * nx;
  [[maybe_unused]] const C* f_u = u_io + (long long)(y0 - 2 * S) * nx + xo;  // row of the last stage
  auto fetch = [&](C* dst, const C* p) {
    if constexpr (V == 1) {
      cheb_cp_async(dst, p + gx0);
    } else {
      if (vec) {
        cheb_cp_async16(dst, p + gx0);
      } else {
        cheb_cp_async(dst, p + gx0);
        cheb_cp_async(dst + 1, p + gx1);
      }
    }
  };
  auto issue = [&](int tf, int slot) {
    C* st = stg + (size_t)slot * SH::NF * NC + V * t;
    if (tf < steps) {
      fetch(st, f_in);
      if constexpr (!START) {
        fetch(st + NC, f_r);
        if (col_own && tf >= 2 * S) {
          if constexpr (V == 1) {
            cheb_cp_async(st + 2 * NC, f_u);
          } else {
            if (vec) {
              cheb_cp_async16(st + 2 * NC, f_u);
            } else {
              cheb_cp_async(st + 2 * NC, f_u);
              if (own1) cheb_cp_async(st + 2 * NC + 1, f_u + 1);
            }
          }
        }
        f_r += fy_r + 1 == g.ny ? -wrap : nx;
        fy_r = cheb_wrap(fy_r, g.ny);
        f_u += nx;
      }
      f_in += fy_in + 1 == g.ny ? -wrap : nx;
      fy_in = cheb_wrap(fy_in, g.ny);
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

  C* o_r = r_out + (long long)(y0 - S - (S - 2 * M)) * nx + xo;  // row of the stage that forms r'
  C* o_d = d_out + (long long)(y0 - 2 * S) * nx + xo;            // row of the last stage
  C* o_u = u_io + (long long)(y0 - 2 * S) * nx + xo;
  double2* o_x = x64 + (long long)(y0 - 2 * S) * nx + xo;

  // own-column history of every stage input: H[q][k] the row formed k' steps ago, k' = (t - k) mod HD
  C H[S][SH::HD][V];
#pragma unroll
  for (int q = 0; q < S; ++q)
#pragma unroll
    for (int k = 0; k < SH::HD; ++k)
#pragma unroll
      for (int v = 0; v < V; ++v) H[q][k][v] = zero;
  [[maybe_unused]] C XD[S + 1][V], RD[S + 1][V];  // inner Chebyshev x and r of each stage, one step old
  if constexpr (M > 1) {
#pragma unroll
    for (int s = 0; s <= S; ++s)
#pragma unroll
      for (int v = 0; v < V; ++v) XD[s][v] = RD[s][v] = zero;
  }
#pragma unroll
  for (int tf = 0; tf < PF; ++tf) issue(tf, tf);
  __syncthreads();

  int slot = 0, islot = PF, kslot = 0;
  for (int t0 = 0; t0 < steps; t0 += U) {
#pragma unroll
    for (int ph = 0; ph < U; ++ph) {
      const int tt = t0 + ph;
      if (tt >= steps) break;
      if constexpr (U % SH::SLOTS == 0) slot = ph % SH::SLOTS, islot = (ph + PF) % SH::SLOTS;
      if constexpr (U % LM == 0) kslot = ph % LM;
      issue(tt + PF, islot);
      asm volatile("cp.async.wait_group %0;\n" ::"n"(PF));
      const C* st = stg + (size_t)slot * SH::NF * NC + V * t;
      C F[S + 1][V];  // values formed in this step: F[q] the output of stage q (row tt - q)
      C X[S + 1][V], R[S + 1][V];
#pragma unroll
      for (int v = 0; v < V; ++v) F[0][v] = st[v];
      // delayed values: the row formed LM steps ago
      C DL[SH::NDEL][V];
      for_stages<0, S - 1>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        constexpr int di = SH::del_index(q);
        if constexpr (di >= 0) {
#pragma unroll
          for (int v = 0; v < V; ++v) {
            if constexpr (SH::REG)
              DL[di][v] = H[q][ph & 3][v];
            else
              DL[di][v] = keep[((size_t)di * LM + kslot) * NC + V * t + v];
          }
        }
      });
      auto put = [&](int q, const C (&f)[V]) {
        C* w = ring + ((size_t)q * 2 + (ph & 1)) * V * RW + t + 1;
#pragma unroll
        for (int v = 0; v < V; ++v) w[v * RW] = f[v];
      };
      put(0, F[0]);
      for_stages<1, S>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        constexpr int q = s - 1;
        // x-neighbours of row tt - s: written by the neighbouring threads one step ago
        const C* rq = ring + ((size_t)q * 2 + ((ph + 1) & 1)) * V * RW + t + 1;
        const C L = rq[(V - 1) * RW - 1], Rr = rq[1];
        const C(&cc)[V] = H[q][(ph + SH::HD - 1) % SH::HD];
        const C(&uu)[V] = H[q][(ph + SH::HD - 2) % SH::HD];
        const C(&dd)[V] = F[q];
        auto lft = [&](int v) { return v == 0 ? L : cc[v > 0 ? v - 1 : 0]; };
        auto rgt = [&](int v) { return v == V - 1 ? Rr : cc[v < V - 1 ? v + 1 : V - 1]; };
        constexpr int rel = s - 1 - PRE;
        constexpr int it = rel >= 0 ? rel / SI : -1;
        constexpr int pos = rel >= 0 ? rel % SI : 2 + (s - 1);  // START's prefix: the P stages
        constexpr int db = PRE + (it < 0 ? 0 : it) * SI;         // stage whose output is this iteration's d
        if constexpr (pos == 0) {
          // g = G d
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const C l = lft(v), r = rgt(v);
            const C lp = q_fma(gy, q_add(uu[v], dd[v]), q_fma(gx, q_add(l, r), q_mul(g0, cc[v])));
            const C ad = q_fma(ay, q_sub(dd[v], uu[v]), q_mul(ax, q_sub(r, l)));
            F[s][v] = q_addi(lp, ad);
          }
        } else if constexpr (pos == 1) {
          // r' = r - a d - kt G g
          const int lr = tt - s;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            C ro;
            if constexpr (it == 0 && !START)
              ro = st[NC + v];
            else
              ro = DL[SH::del_index(START ? 0 : db - SI + 2)][v];
            const C dc = H[db][(ph + SH::HD - 2) % SH::HD][v];
            const C l = lft(v), r = rgt(v);
            const C lp = q_fma(ky, q_add(uu[v], dd[v]),
                               q_fma(kx, q_add(l, r), q_fma(k0, cc[v], q_fma(ma, dc, ro))));
            const C ad = q_fma(by, q_sub(dd[v], uu[v]), q_mul(bx, q_sub(r, l)));
            F[s][v] = q_addi(lp, ad);
          }
          if constexpr (it == SH::NIT - 1) {
            if (!last && col_own && lr >= S && lr < steps - S) store(o_r, F[s]);
          }
        } else {
          // application k of D in solve 1 or 2 of p
          constexpr int pp = pos - 2;
          constexpr bool second = pp >= M;
          constexpr int k = pp % M;
          constexpr bool fin = k == M - 1;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const C l = lft(v), r = rgt(v);
            const C Dv = q_fma(py, q_add(uu[v], dd[v]), q_fma(px, q_add(l, r), q_mul(p0, cc[v])));
            C out;
            if constexpr (M == 1) {
              out = Dv;
            } else {
              C dn;
              if constexpr (k == 0) {
                X[s][v] = q_mul(q_.ith, cc[v]);
                R[s][v] = q_fma(-q_.ith, Dv, cc[v]);
                dn = q_fma(q_.w1[0], X[s][v], q_mul(q_.w2[0], R[s][v]));
              } else {
                X[s][v] = q_add(XD[s - 1][v], cc[v]);
                R[s][v] = q_sub(RD[s - 1][v], Dv);
                dn = q_fma(q_.w1[k], cc[v], q_mul(q_.w2[k], R[s][v]));
              }
              out = fin ? q_add(X[s][v], dn) : dn;
            }
            if constexpr (fin && second) {
              if constexpr (it < 0)
                out = q_mul(q_.ith_out, out);  // d_0
              else
                out = q_fma(q_.c2[it < 0 ? 0 : it], out, q_mul(q_.c1[it < 0 ? 0 : it], DL[SH::del_index(db)][v]));
            }
            F[s][v] = out;
          }
        }
        if constexpr (s < S) put(s, F[s]);
      });
      // the last stage's row: u and d, or the state
      {
        const int lr = tt - S;
        if (col_own && lr >= S) {
          C un[V];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            if constexpr (START) {
              un[v] = q_add(DL[1][v], F[S][v]);  // d_0 + d_1
            } else {
              un[v] = st[2 * NC + v];
              if constexpr (SH::NIT == 2) un[v] = q_add(un[v], DL[SH::del_index(SI)][v]);
              un[v] = q_add(un[v], F[S][v]);
            }
          }
          if (!last) {
            store(o_d, F[S]);
            store(o_u, un);
          } else {
#pragma unroll
            for (int v = 0; v < V; ++v) {
              if (v > 0 && !own1) break;
              double2 xv = o_x[v];
              if constexpr (sizeof(T) == 4) {  // exact widening by integer operations
                xv.x += f2d(un[v].x);
                xv.y += f2d(un[v].y);
              } else {
                xv.x += un[v].x;
                xv.y += un[v].y;
              }
              o_x[v] = xv;
            }
          }
        }
      }
      // history: the values of this step replace the oldest row
      for_stages<0, S - 1>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        constexpr int di = SH::del_index(q);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          H[q][ph % SH::HD][v] = F[q][v];
          if constexpr (di >= 0 && !SH::REG) keep[((size_t)di * LM + kslot) * NC + V * t + v] = F[q][v];
        }
      });
      if constexpr (M > 1) {
        for_stages<1, S>([&](auto sc) {
          constexpr int s = decltype(sc)::value;
          constexpr int pos = s - 1 - PRE >= 0 ? (s - 1 - PRE) % SI : 2 + (s - 1);
          if constexpr (pos >= 2) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
              XD[s][v] = X[s][v];
              RD[s][v] = R[s][v];
            }
          }
        });
      }
      o_r += nx;
      o_d += nx;
      o_u += nx;
      o_x += nx;
      if constexpr (U % SH::SLOTS != 0) {
        slot = slot + 1 == SH::SLOTS ? 0 : slot + 1;
        islot = islot + 1 == SH::SLOTS ? 0 : islot + 1;
      }
      if constexpr (U % LM != 0) kslot = kslot + 1 == LM ? 0 : kslot + 1;
      __syncthreads();
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
}

inline ChebGeom cheb_geom(int nx, int ny, int S, int NC, int Ly) {
  ChebGeom g;
  g.nx = nx;
  g.ny = ny;
  g.pts = (long long)nx * ny;
  g.Ly = Ly < ny ? Ly : ny;
  g.wv = NC - 2 * S;
  g.nstrips = (nx + g.wv - 1) / g.wv;
  g.nsegs = (ny + g.Ly - 1) / g.Ly;
  return g;
}

// The launch table of runs r0 .. of a batch; returns their count, the most blocks of one in maxblk.
// take: all runs (0), those on tiles (1) or the others (-1; gauge_tiled).
inline int cheb_table(const BatchLaunch& bl, int r0, int S, int NC, int Ly, int J, ChebTab& tab, int& maxblk,
                      int take = 0) {
  const int nr = std::min(kChebRuns, bl.R - r0);
  std::memset(&tab, 0, sizeof(tab));
  maxblk = 0;
  for (int i = 0; i < nr; ++i) {
    const RunGeom& q = bl.host[r0 + i];
    if (take != 0 && (take > 0) != gauge_tiled(q.nx, q.ny, J)) continue;
    const ChebGeom g = cheb_geom(q.nx, q.ny, S, NC, Ly);
    ChebRun& e = tab.run[i];
    e.pts = q.pts;
    e.foff = q.field_off;
    e.xoff = q.elem_off;
    e.nx = q.nx;
    e.ny = q.ny;
    e.Ly = g.Ly;
    e.nstrips = g.nstrips;
    e.nsegs = g.nsegs;
    e.nblk = g.nstrips * g.nsegs * J;
    e.run = r0 + i;
    maxblk = std::max(maxblk, e.nblk);
  }
  return nr;
}

// One pass over one grid or, with bl, over every run of a batch.
template <typename T, int M, int NI, int V, int NT, int PF, bool START>
bool launch_cheb_pass(const OpCoef& c, const ChebStep* w, const ChebPass& cp, int Ly, const ChebBufs<T>& b, int pass,
                      cudaStream_t s, const BatchLaunch* bl) {
  using SH = ChebShape<T, M, NI, V, NT, PF, START>;
  static_assert(SH::S % V == 0 && (SH::NC - 2 * SH::S) % V == 0, "strips start on a pair");
  const int kid = kid_of<T>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  const ChebParam<T, M> in = cheb_param<T, M>(c, w, cp);
  const int cur = pass & 1;
  const cplx<T>* rin = START ? b.r0 : b.r[cur];
  if (bl == nullptr) {
    auto kern = k_cheb2d<T, M, NI, V, NT, PF, START, ChebNoTab>;
    static const cudaError_t attr =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (attr != cudaSuccess) return false;
    const ChebGeom g = cheb_geom(c.nx, c.ny, SH::S, SH::NC, Ly);
    kern<<<dim3(g.nstrips, g.nsegs, c.J), NT, SH::smem, s>>>(in, g, rin, b.d[cur], b.r[1 - cur], b.d[1 - cur],
                                                            b.u, b.x64, b.ks, pass, kid, ChebNoTab{});
    return true;
  }
  if constexpr (sizeof(T) == 8) {
    return false;  // batched runs are FP32
  } else {
    auto kern = k_cheb2d<T, M, NI, V, NT, PF, START, ChebTab>;
    static const cudaError_t attr =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (attr != cudaSuccess) return false;
    for (int r0 = 0; r0 < bl->R; r0 += kChebRuns) {
      ChebTab tab;
      int maxblk = 0;
      const int nr = cheb_table(*bl, r0, SH::S, SH::NC, Ly, c.J, tab, maxblk);
      kern<<<dim3(maxblk, nr), NT, SH::smem, s>>>(in, ChebGeom{0, 0, 0, SH::NC - 2 * SH::S, 0, 0, 0}, rin,
                                                  b.d[cur], b.r[1 - cur], b.d[1 - cur], b.u, b.x64, b.ks, pass, kid,
                                                  tab);
    }
    return true;
  }
}

}  // namespace

}  // namespace apfc
