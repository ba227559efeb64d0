// Chebyshev iteration on the Schur complement S = a + kt G_h^2, 3D grids: the 2D iteration of
// gauge2d.cuh (the same gauge, the same recurrence), one term a pass.
//
// k_gauge3d streams through a chunk of z-planes of an (x, y) tile of TXV x TYV points with a halo
// of two: at step t it forms g' = N v on plane t - 1 and v_(n+1) = v_n + c1 (v_n - v_(n-1)) -
// c2 (a v_n - b + N g') on plane t - 2.  A thread owns V adjacent points of two adjacent rows in
// every plane; z-neighbours are in registers (the plane below has just been formed), x- and
// y-neighbours come from two-plane shared-memory rings, one barrier a plane.  v is fetched PF
// planes ahead (cp.async), v_(n-1) and b, needed at the thread's own points alone, one plane
// ahead into registers.  v_(n+1) replaces v_(n-1) in place.  Reads v, v_(n-1), b, writes
// v_(n+1): 32 bytes a point in FP32.
#pragma once
#include "gauge2d.cuh"

namespace apfc {

namespace {

// A warp spans a row of the tile with its halo (32 lanes of V points), so that shared-memory
// accesses have no bank conflicts (36-column tiles with rows across warps took two wavefronts for
// each) and rows are uniform over a warp.
template <typename T, int V_, int TYV_, int PF_, bool START_>
struct Gauge3Shape {
  static constexpr int V = V_, TYV = TYV_, PF = PF_;
  static constexpr int OX = 32 * V, TXV = OX - 4, OY = TYV + 4;  // tile with its halo
  static constexpr int PX = 32, NT = PX * (OY / 2);
  static constexpr int RW = PX + 2, PLANE = (OY + 2) * RW;  // one part of a ring plane, padded
  static constexpr int SLOTS = PF + 1;
  static constexpr size_t ring_elems = 2ull * 2 * V * PLANE;  // v, g' x two planes
  static constexpr size_t stage_elems = (size_t)SLOTS * NT * 2 * V;
  static constexpr size_t smem = sizeof(cplx<T>) * (ring_elems + stage_elems);
};

struct Gauge3Geom {
  int nx, ny, nz, Lz, ntx;
  long long pts;
};
template <typename T>
struct Gauge3Amp {
  T n0, nx, ny, nz, a, c1, mc2, mith;
};
template <typename T>
struct Gauge3Param {
  Gauge3Amp<T> amp[kMaxJ];
  unsigned long long* prof;
  const cplx<T>* tab;  // [J][tx + ty + tz]
  int J, tx, ty, tz;
};

// Grid (tiles, z-chunks, J).  START: v is the residual; forms b (negated) and v_1, writes both
// and v_2.  vp: v_(n-1) in, v_(n+1) out (START: v_2); v1_out: START's v_1.
template <typename T, int V, int TYV, int PF, int MINB, bool START>
__global__ void __launch_bounds__(Gauge3Shape<T, V, TYV, PF, START>::NT, MINB)
    k_gauge3d(const __grid_constant__ Gauge3Param<T> c, Gauge3Geom g, const cplx<T>* v_in, cplx<T>* vp, cplx<T>* b_io,
              cplx<T>* v1_out, double2* x64, const KScal* ks, int pass, int kid) {
  using SH = Gauge3Shape<T, V, TYV, PF, START>;
  using C = cplx<T>;
  constexpr int NT = SH::NT, TXV = SH::TXV, OX = SH::OX, OY = SH::OY, RW = SH::RW, PLANE = SH::PLANE;
  extern __shared__ __align__(16) unsigned char gauge3_smem[];
  C* ring = reinterpret_cast<C*>(gauge3_smem);  // [v, g'][2 planes][V][PLANE]
  C* stg = ring + SH::ring_elems;               // [SLOTS][NT][2][V]
  const int j = blockIdx.z, t = threadIdx.x;
  const int npass = ks[j].iters;
  if (pass >= npass) return;
  const bool last = pass + 1 == npass;
  if (c.prof != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && t == 0)
    atomicAdd(c.prof + kid, (unsigned long long)g.pts *
                                ((START ? 1 : 3) * sizeof(C) + (last ? 2 * sizeof(double2) : (START ? 3 : 1) * sizeof(C))));
  const Gauge3Amp<T>& q = c.amp[j];
  const T n0 = q.n0, wx = q.nx, wy = q.ny, wz = q.nz, aa = q.a, c1 = q.c1, mc2 = q.mc2;
  const C* tabx = c.tab + (long long)j * (c.tx + c.ty + c.tz);
  const C* taby = tabx + c.tx;
  const C* tabz = taby + c.ty;
  {
    const long long o = (long long)j * g.pts;
    v_in += o;
    vp += o;
    b_io += o;
    if constexpr (START) v1_out += o;
    x64 += 2 * o + g.pts;
  }
  const C zero = mkc<T>((T)0, (T)0), one = mkc<T>((T)1, (T)0);
  for (int i = t; i < (int)SH::ring_elems; i += NT) ring[i] = zero;

  // cells: columns V px .. of rows 2 ry and 2 ry + 1 of the tile; positions beyond the grid are
  // the periodic image times the wraps' phases
  const int ry = __shfl_sync(0xffffffffu, t >> 5, 0), px = t & 31;  // row pair: uniform over the warp
  const int tyi = blockIdx.x / g.ntx, txi = blockIdx.x - tyi * g.ntx;
  const int X0 = txi * TXV - 2 + V * px, Y0 = tyi * TYV - 2 + 2 * ry;
  int gx[V], gyr[2], goff[2];
  bool wrapped = false, xown[V], yown[2];
  C colf[V], rowf[2];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    int x = (X0 + v) % g.nx;
    if (x < 0) x += g.nx;
    gx[v] = x;
    colf[v] = g_pow(tabx[g.nx], (X0 + v - x) / g.nx, one);
    wrapped = wrapped || X0 + v != x;
    xown[v] = V * px + v >= 2 && V * px + v < OX - 2 && X0 + v < g.nx;
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    int y = (Y0 + r) % g.ny;
    if (y < 0) y += g.ny;
    gyr[r] = y;
    goff[r] = y * g.nx;
    rowf[r] = g_pow(taby[g.ny], (Y0 + r - y) / g.ny, one);
    wrapped = wrapped || Y0 + r != y;
    yown[r] = 2 * ry + r >= 2 && 2 * ry + r < OY - 2 && Y0 + r < g.ny;
  }
  const bool rows_own = yown[0] || yown[1];  // stage B's rows: the warps of the halo skip it
  const bool vec = V == 1 || (g.nx & 1) == 0;
  const long long plane = (long long)g.nx * g.ny;
  const int z0 = blockIdx.y * g.Lz, nzc = min(g.nz, z0 + g.Lz) - z0, steps = nzc + 4;
  int fz = (z0 - 2) % g.nz;
  if (fz < 0) fz += g.nz;
  int cz = fz, mz = (z0 - 2 - fz) / g.nz;  // plane of the current step, its wraps
  const C ez = tabz[g.nz];
  C zf = g_pow(ez, mz, one);
  const C* f_v = v_in + fz * plane;
  auto issue = [&](int tf, int slot) {
    if (tf < steps) {
      C* d = stg + ((size_t)slot * NT + t) * 2 * V;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const C* p = f_v + goff[r];
        if constexpr (V == 1) {
          cheb_cp_async(d + r, p + gx[0]);
        } else {
          if (vec) {
            cheb_cp_async16(d + 2 * r, p + gx[0]);
          } else {
            cheb_cp_async(d + 2 * r, p + gx[0]);
            cheb_cp_async(d + 2 * r + 1, p + gx[V - 1]);
          }
        }
      }
      f_v += fz + 1 == g.nz ? -(g.nz - 1) * plane : plane;
      fz = cheb_wrap(fz, g.nz);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  // own points of plane z (elements of the field): loads and stores of pairs where the row allows
  auto load_own = [&](const C* src, long long zo, C (&d)[2][V]) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const C* p = src + zo + goff[r] + gx[0];
      if constexpr (V == 1) {
        if (yown[r] && xown[0]) d[r][0] = p[0];
      } else {
        if (vec) {
          if (yown[r] && xown[0]) {
            const float4 w = *reinterpret_cast<const float4*>(p);
            d[r][0] = make_float2(w.x, w.y);
            d[r][1] = make_float2(w.z, w.w);
          }
        } else {
          if (yown[r] && xown[0]) d[r][0] = p[0];
          if (yown[r] && xown[V - 1]) d[r][1] = src[zo + goff[r] + gx[V - 1]];
        }
      }
    }
  };
  auto store_own = [&](C* dst, long long zo, const C (&d)[2][V]) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      C* p = dst + zo + goff[r] + gx[0];
      if constexpr (V == 1) {
        if (yown[r] && xown[0]) p[0] = d[r][0];
      } else {
        if (vec) {
          if (yown[r] && xown[0]) *reinterpret_cast<float4*>(p) = make_float4(d[r][0].x, d[r][0].y, d[r][1].x, d[r][1].y);
        } else {
          if (yown[r] && xown[0]) p[0] = d[r][0];
          if (yown[r] && xown[V - 1]) dst[zo + goff[r] + gx[V - 1]] = d[r][1];
        }
      }
    }
  };

  // planes formed one and two steps ago
  C v1[2][V], v2[2][V], h1[2][V], h2[2][V];
  // START: b one and two planes old; else v_(n-1) and b fetched for the next step's stage B
  C s1[2][V], s2[2][V];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int v = 0; v < V; ++v) v1[r][v] = v2[r][v] = h1[r][v] = h2[r][v] = s1[r][v] = s2[r][v] = zero;
#pragma unroll
  for (int tf = 0; tf < PF; ++tf) issue(tf, tf);
  __syncthreads();
  int slot = 0, islot = PF;
  const int cell = (2 * ry + 1) * RW + px + 1;  // ring position of the upper row
#pragma unroll 2
  for (int tt = 0; tt < steps; ++tt) {
    issue(tt + PF, islot);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(PF));
    const int par = tt & 1;
    C pv[2][V], bv[2][V];
    const bool outz = tt >= 4;  // stage B's plane tt - 2 is one of the chunk's
    const long long zo = (long long)(z0 + tt - 4) * plane;
    if constexpr (!START) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) pv[r][v] = s1[r][v], bv[r][v] = s2[r][v];
      if (tt >= 3 && tt + 1 < steps) {  // the next step's
        load_own(vp, zo + plane, s1);
        load_own(b_io, zo + plane, s2);
      }
    }
    C F[2][V];
    {
      const C* st = stg + ((size_t)slot * NT + t) * 2 * V;
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) F[r][v] = st[r * V + v];
    }
    C bt[2][V];
    if constexpr (START) {
      const C pz = g_cmul(tabz[cz], zf);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const C pr = g_cmul(pz, g_cmul(taby[gyr[r]], rowf[r]));
          const C w = g_cmul(g_cmul(pr, g_cmul(tabx[gx[v]], colf[v])), F[r][v]);
          bt[r][v] = mkc<T>(-w.x, -w.y);
          F[r][v] = q_mul(q.mith, bt[r][v]);
        }
      if (!last && tt >= 2 && tt < steps - 2) {
        store_own(b_io, zo + 2 * plane, bt);
        store_own(v1_out, zo + 2 * plane, F);
      }
    } else if (wrapped || mz != 0) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) F[r][v] = g_cmul(g_cmul(g_cmul(zf, rowf[r]), colf[v]), F[r][v]);
    }
    auto put = [&](int w, const C (&f)[2][V]) {
      C* d = ring + ((size_t)w * 2 + par) * V * PLANE + cell;
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) d[v * PLANE + r * RW] = f[r][v];
    };
    // n0 c + wx (l + r) + wy (u + d) + wz (below + above) + add at the cells of ring w's previous plane
    auto stencil = [&](int w, const C (&cc)[2][V], const C (&bl)[2][V], const C (&ab)[2][V], const C* add, C (&out)[2][V]) {
      const C* d = ring + ((size_t)w * 2 + (par ^ 1)) * V * PLANE + cell;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const C L = d[(V - 1) * PLANE + r * RW - 1], R = d[r * RW + 1];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const C l = v == 0 ? L : cc[r][v > 0 ? v - 1 : 0], rr = v == V - 1 ? R : cc[r][v < V - 1 ? v + 1 : 0];
          const C o = r == 0 ? d[v * PLANE - RW] : d[v * PLANE + 2 * RW];  // the row outside the pair
          const C s0 = add != nullptr ? q_fma(n0, cc[r][v], add[r * V + v]) : q_mul(n0, cc[r][v]);
          out[r][v] = q_fma(wz, q_add(bl[r][v], ab[r][v]),
                            q_fma(wy, q_add(o, cc[1 - r][v]), q_fma(wx, q_add(l, rr), s0)));
        }
      }
    };
    put(0, F);
    C G[2][V];
    stencil(0, v1, v2, F, nullptr, G);  // plane tt - 1
    put(1, G);
    if (rows_own) {
      // r^ = a v - b + N g' at plane tt - 2
      C av[2 * V], rh[2][V], out[2][V];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) av[r * V + v] = q_fma(aa, v2[r][v], START ? s2[r][v] : bv[r][v]);
      stencil(1, h1, h2, G, av, rh);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const C old = START ? zero : pv[r][v];
          out[r][v] = q_fma(mc2, rh[r][v], q_fma(c1, q_sub(v2[r][v], old), v2[r][v]));
        }
      if (outz) {
        if (!last) {
          store_own(vp, zo, out);
        } else {
          const C pz = tabz[z0 + tt - 4];
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int v = 0; v < V; ++v) {
              if (!(yown[r] && xown[v])) continue;
              const C un = g_cmul(g_conj(g_cmul(g_cmul(pz, taby[gyr[r]]), tabx[gx[v]])), out[r][v]);
              double2* xp = x64 + zo + goff[r] + gx[v];
              double2 xv = *xp;
              if constexpr (sizeof(T) == 4) {
                xv.x += f2d(un.x);
                xv.y += f2d(un.y);
              } else {
                xv.x += un.x;
                xv.y += un.y;
              }
              *xp = xv;
            }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        v2[r][v] = v1[r][v];
        v1[r][v] = F[r][v];
        h2[r][v] = h1[r][v];
        h1[r][v] = G[r][v];
        if constexpr (START) {
          s2[r][v] = s1[r][v];
          s1[r][v] = bt[r][v];
        }
      }
    if (cz + 1 == g.nz) {
      cz = 0;
      ++mz;
      zf = g_cmul(zf, ez);
    } else {
      ++cz;
    }
    slot = slot + 1 == SH::SLOTS ? 0 : slot + 1;
    islot = islot + 1 == SH::SLOTS ? 0 : islot + 1;
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
}

template <typename T, int V, int TYV, int PF, int MINB, bool START>
bool launch_gauge3_pass(const OpCoef& c, const GaugeTab<T>& gt, const GaugeWeights& w, int Lz, const ChebBufs<T>& b,
                        int pass, cudaStream_t s) {
  using SH = Gauge3Shape<T, V, TYV, PF, START>;
  constexpr int TXV = SH::TXV;
  static_assert(SH::OX % V == 0 && SH::OY % 2 == 0 && SH::NT <= 1024, "tile");
  const int kid = kid_of<T>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  Gauge3Param<T> in;
  std::memset(&in, 0, sizeof(in));
  in.prof = c.prof;
  in.tab = gt.tab;
  in.tx = gt.tx;
  in.ty = gt.ty;
  in.tz = gt.tz;
  in.J = c.J;
  for (int j = 0; j < c.J; ++j) {
    Gauge3Amp<T>& a = in.amp[j];
    const double sk = -std::sqrt(c.kt[j]);
    a.n0 = (T)(sk * c.c0);
    a.nx = (T)(sk * gauge_w(c, j, 0));
    a.ny = (T)(sk * gauge_w(c, j, 1));
    a.nz = (T)(sk * gauge_w(c, j, 2));
    a.a = (T)c.a[j];
    a.c1 = (T)w.c1[0][j];
    a.mc2 = (T)(-w.c2[0][j]);
    a.mith = (T)(-w.inv_theta[j]);
  }
  auto kern = k_gauge3d<T, V, TYV, PF, MINB, START>;
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
  if (attr != cudaSuccess) return false;
  // START: v_1 into r[1], v_2 into d[0]; pass p >= 1 reads v from d[0] / r[1] and replaces the other
  cplx<T>* two[2] = {b.r[1], b.d[0]};
  const Gauge3Geom g{c.nx, c.ny, c.nz, Lz, (c.nx + TXV - 1) / TXV, c.pts};
  const dim3 grid((unsigned)(g.ntx * ((c.ny + TYV - 1) / TYV)), (unsigned)((c.nz + Lz - 1) / Lz), (unsigned)c.J);
  kern<<<grid, SH::NT, SH::smem, s>>>(in, g, START ? b.r0 : two[pass & 1], START ? two[1] : two[1 - (pass & 1)], b.u,
                                      START ? two[0] : nullptr, b.x64, b.ks, pass, kid);
  return true;
}

}  // namespace

}  // namespace apfc
