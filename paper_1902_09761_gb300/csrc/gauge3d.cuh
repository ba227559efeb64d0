// Chebyshev iteration on the Schur complement S = a + kt G_h^2, 3D grids: the 2D iteration of
// gauge2d.cuh (the same gauge, the same recurrence), one term a pass.
//
// k_gauge3d streams through a chunk of z-planes of an (x, y) tile of TXV x TYV points with a halo
// of two: at step t it forms g' = N v on plane t - 1 and v_(n+1) = v_n + c1 (v_n - v_(n-1)) -
// c2 (a v_n - b + N g') on plane t - 2.  A thread owns two adjacent columns of R adjacent rows in
// every plane; z-neighbours are in registers (the plane below has just been formed), x-neighbours
// come by shuffles (a warp spans the tile), the rows above and below a warp's from two-plane
// shared-memory rings, one barrier a plane.  v is fetched PF planes ahead (cp.async), v_(n-1) and
// b, needed at the thread's own points alone, one plane ahead into registers.  v_(n+1) replaces
// v_(n-1) in place.  Reads v, v_(n-1), b, writes v_(n+1): 32 bytes a point.
#pragma once
#include "gauge2d.cuh"

namespace apfc {

namespace {

// A warp spans the tile with its halo (32 lanes of two columns) in R adjacent rows.
template <int R_, int NW_, int PF_>
struct Gauge3Shape {
  static constexpr int R = R_, NW = NW_, PF = PF_;
  static constexpr int OX = 64, TXV = OX - 4, OY = R * NW, TYV = OY - 4;  // tile with its halo
  static constexpr int NT = 32 * NW, SLOTS = PF + 1;
  static constexpr size_t ring = 2ull * 2 * NW * 2 * 32;  // v, g' x two planes x each warp's outer rows (float4)
  static constexpr size_t stage = (size_t)SLOTS * R * NT;
  static constexpr size_t smem = sizeof(float4) * (ring + stage);
};

struct Gauge3Geom {
  int nx, ny, nz, Lz, ntx;
  long long pts;
};
struct Gauge3Amp {
  float n0, nx, ny, nz, a, c1, mc2, mith;
};
struct Gauge3Param {
  Gauge3Amp amp[kMaxJ];
  unsigned long long* prof;
  const float2* tab;  // [J][tx + ty + tz]
  int J, tx, ty, tz;
};

// Grid (tiles, z-chunks, J).  START: v is the residual; forms b (negated) and v_1, writes both
// and v_2.  vp: v_(n-1) in, v_(n+1) out (START: v_2); v1_out: START's v_1.
template <int R, int NW, int PF, int MINB, bool START>
__global__ void __launch_bounds__(32 * NW, MINB)
    k_gauge3d(const __grid_constant__ Gauge3Param c, Gauge3Geom g, const float2* v_in, float2* vp, float2* b_io,
              float2* v1_out, double2* x64, const KScal* ks, int pass, int kid) {
  using SH = Gauge3Shape<R, NW, PF>;
  using C = float2;
  constexpr int NT = SH::NT, TXV = SH::TXV, TYV = SH::TYV, OX = SH::OX, OY = SH::OY;
  extern __shared__ __align__(16) unsigned char gauge3_smem[];
  float4* ring = reinterpret_cast<float4*>(gauge3_smem);  // [v, g'][2 planes][NW][first, last row][32]
  float4* stg = ring + SH::ring + threadIdx.x;            // [SLOTS][R][NT]
  const int j = blockIdx.z, t = threadIdx.x;
  dependent_wait();
  const int npass = ks[j].iters;
  if (pass >= npass) return;
  const bool last = pass + 1 == npass;
  if (c.prof != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && t == 0)
    atomicAdd(c.prof + kid, (unsigned long long)g.pts *
                                ((START ? 1 : 3) * sizeof(C) + (last ? 2 * sizeof(double2) : (START ? 3 : 1) * sizeof(C))));
  const Gauge3Amp& q = c.amp[j];
  const float n0 = q.n0, wx = q.nx, wy = q.ny, wz = q.nz, aa = q.a, c1 = q.c1, mc2 = q.mc2;
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
  const C zero = make_float2(0.f, 0.f), one = make_float2(1.f, 0.f);
  for (int i = t; i < (int)SH::ring; i += NT) ring[i] = make_float4(0.f, 0.f, 0.f, 0.f);

  // columns 2 px, 2 px + 1 of rows R w .. of the tile; positions beyond the grid are
  // the periodic image times the wraps' phases
  const int w = __shfl_sync(0xffffffffu, t >> 5, 0), px = t & 31;
  const int tyi = blockIdx.x / g.ntx, txi = blockIdx.x - tyi * g.ntx;
  const int X0 = txi * TXV - 2 + 2 * px, Y0 = tyi * TYV - 2 + R * w;
  int gx[2], gyr[R], goff[R];
  bool wrapped = false, xown[2], yown[R];
  C colf[2], rowf[R];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    int x = (X0 + v) % g.nx;
    if (x < 0) x += g.nx;
    gx[v] = x;
    colf[v] = g_pow(tabx[g.nx], (X0 + v - x) / g.nx, one);
    wrapped = wrapped || X0 + v != x;
    xown[v] = 2 * px + v >= 2 && 2 * px + v < OX - 2 && X0 + v < g.nx;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int y = (Y0 + r) % g.ny;
    if (y < 0) y += g.ny;
    gyr[r] = y;
    goff[r] = y * g.nx;
    rowf[r] = g_pow(taby[g.ny], (Y0 + r - y) / g.ny, one);
    wrapped = wrapped || Y0 + r != y;
    yown[r] = R * w + r >= 2 && R * w + r < OY - 2 && Y0 + r < g.ny;
  }
  const bool vec = (g.nx & 1) == 0;
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
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const C* p = f_v + goff[r];
        C* d = reinterpret_cast<C*>(stg + (slot * R + r) * NT);
        if (vec) {
          cheb_cp_async16(d, p + gx[0]);
        } else {
          cheb_cp_async(d, p + gx[0]);
          cheb_cp_async(d + 1, p + gx[1]);
        }
      }
      f_v += fz + 1 == g.nz ? -(g.nz - 1) * plane : plane;
      fz = cheb_wrap(fz, g.nz);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  // own points of plane z (elements of the field): loads and stores of pairs where the row allows
  auto load_own = [&](const C* src, long long zo, C (&d)[R][2]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const C* p = src + zo + goff[r] + gx[0];
      if (vec) {
        if (yown[r] && xown[0]) {
          const float4 f = *reinterpret_cast<const float4*>(p);
          d[r][0] = make_float2(f.x, f.y);
          d[r][1] = make_float2(f.z, f.w);
        }
      } else {
        if (yown[r] && xown[0]) d[r][0] = p[0];
        if (yown[r] && xown[1]) d[r][1] = src[zo + goff[r] + gx[1]];
      }
    }
  };
  auto store_own = [&](C* dst, long long zo, const C (&d)[R][2]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      C* p = dst + zo + goff[r] + gx[0];
      if (vec) {
        if (yown[r] && xown[0]) *reinterpret_cast<float4*>(p) = make_float4(d[r][0].x, d[r][0].y, d[r][1].x, d[r][1].y);
      } else {
        if (yown[r] && xown[0]) p[0] = d[r][0];
        if (yown[r] && xown[1]) dst[zo + goff[r] + gx[1]] = d[r][1];
      }
    }
  };

  // planes formed one and two steps ago
  C v1[R][2], v2[R][2], h1[R][2], h2[R][2];
  // START: b one and two planes old; else v_(n-1) and b fetched for the next step's stage B
  C s1[R][2], s2[R][2];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int v = 0; v < 2; ++v) v1[r][v] = v2[r][v] = h1[r][v] = h2[r][v] = s1[r][v] = s2[r][v] = zero;
#pragma unroll
  for (int tf = 0; tf < PF; ++tf) issue(tf, tf);
  __syncthreads();
  int slot = 0, islot = PF;
#pragma unroll 2
  for (int tt = 0; tt < steps; ++tt) {
    issue(tt + PF, islot);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(PF));
    const int par = tt & 1;
    C pv[R][2], bv[R][2];
    const bool outz = tt >= 4;  // stage B's plane tt - 2 is one of the chunk's
    const long long zo = (long long)(z0 + tt - 4) * plane;
    if constexpr (!START) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int v = 0; v < 2; ++v) pv[r][v] = s1[r][v], bv[r][v] = s2[r][v];
      if (tt >= 3 && tt + 1 < steps) {  // the next step's
        load_own(vp, zo + plane, s1);
        load_own(b_io, zo + plane, s2);
      }
    }
    C F[R][2];
    {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 f = stg[(slot * R + r) * NT];
        F[r][0] = make_float2(f.x, f.y);
        F[r][1] = make_float2(f.z, f.w);
      }
    }
    C bt[R][2];
    if constexpr (START) {
      const C pz = g_cmul(tabz[cz], zf);
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const C pr = g_cmul(pz, g_cmul(taby[gyr[r]], rowf[r]));
          const C w = g_cmul(g_cmul(pr, g_cmul(tabx[gx[v]], colf[v])), F[r][v]);
          bt[r][v] = make_float2(-w.x, -w.y);
          F[r][v] = q_mul(q.mith, bt[r][v]);
        }
      if (!last && tt >= 2 && tt < steps - 2) {
        store_own(b_io, zo + 2 * plane, bt);
        store_own(v1_out, zo + 2 * plane, F);
      }
    } else if (wrapped || mz != 0) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int v = 0; v < 2; ++v) F[r][v] = g_cmul(g_cmul(g_cmul(zf, rowf[r]), colf[v]), F[r][v]);
    }
    auto put = [&](int q, const C (&f)[R][2]) {
      float4* d = ring + ((q * 2 + par) * NW + w) * 64 + px;
      d[0] = make_float4(f[0][0].x, f[0][0].y, f[0][1].x, f[0][1].y);
      d[32] = make_float4(f[R - 1][0].x, f[R - 1][0].y, f[R - 1][1].x, f[R - 1][1].y);
    };
    // n0 c + wx (l + r) + wy (u + d) + wz (below + above) + add on the previous plane of ring q
    auto stencil = [&](int q, const C (&cc)[R][2], const C (&bl)[R][2], const C (&ab)[R][2], auto first, auto out) {
      const float4* d = ring + (q * 2 + (par ^ 1)) * NW * 64 + px;
      const float4 uf = d[w > 0 ? w * 64 - 32 : 0], df = d[w < NW - 1 ? w * 64 + 64 : 0];
      const C up[2] = {make_float2(uf.x, uf.y), make_float2(uf.z, uf.w)};
      const C dn[2] = {make_float2(df.x, df.y), make_float2(df.z, df.w)};
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const C L = make_float2(__shfl_up_sync(0xffffffffu, cc[r][1].x, 1), __shfl_up_sync(0xffffffffu, cc[r][1].y, 1));
        const C Q = make_float2(__shfl_down_sync(0xffffffffu, cc[r][0].x, 1), __shfl_down_sync(0xffffffffu, cc[r][0].y, 1));
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const C l = v == 0 ? L : cc[r][0], rr = v == 1 ? Q : cc[r][1];
          const C u = r == 0 ? up[v] : cc[r > 0 ? r - 1 : 0][v], b = r == R - 1 ? dn[v] : cc[r < R - 1 ? r + 1 : 0][v];
          out(r, v, q_fma(wz, q_add(bl[r][v], ab[r][v]),
                          q_fma(wy, q_add(u, b), q_fma(wx, q_add(l, rr), first(r, v)))));
        }
      }
    };
    put(0, F);
    C G[R][2];  // plane tt - 1
    stencil(0, v1, v2, F, [&](int r, int v) { return q_mul(n0, v1[r][v]); }, [&](int r, int v, C f) { G[r][v] = f; });
    put(1, G);
    {
      // r^ = a v - b + N g' at plane tt - 2
      C out[R][2];
      stencil(
          1, h1, h2, G,
          [&](int r, int v) { return q_fma(n0, h1[r][v], q_fma(aa, v2[r][v], START ? s2[r][v] : bv[r][v])); },
          [&](int r, int v, C rh) {
            const C old = START ? zero : pv[r][v];
            out[r][v] = q_fma(mc2, rh, q_fma(c1, q_sub(v2[r][v], old), v2[r][v]));
          });
      if (outz) {
        if (!last) {
          store_own(vp, zo, out);
        } else {
          const C pz = tabz[z0 + tt - 4];
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int v = 0; v < 2; ++v) {
              if (!(yown[r] && xown[v])) continue;
              const C un = g_cmul(g_conj(g_cmul(g_cmul(pz, taby[gyr[r]]), tabx[gx[v]])), out[r][v]);
              double2* xp = x64 + zo + goff[r] + gx[v];
              double2 xv = *xp;
              xv.x += f2d(un.x);
              xv.y += f2d(un.y);
              *xp = xv;
            }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
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

template <int R, int NW, int PF, int MINB, bool START>
bool launch_gauge3_pass(const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, int Lz,
                        const ChebBufs<float>& b, int pass, cudaStream_t s) {
  using SH = Gauge3Shape<R, NW, PF>;
  constexpr int TXV = SH::TXV, TYV = SH::TYV;
  const int kid = kid_of<float>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  Gauge3Param in;
  std::memset(&in, 0, sizeof(in));
  in.prof = c.prof;
  in.tab = gt.tab;
  in.tx = gt.tx;
  in.ty = gt.ty;
  in.tz = gt.tz;
  in.J = c.J;
  for (int j = 0; j < c.J; ++j) {
    Gauge3Amp& a = in.amp[j];
    const double sk = -std::sqrt(c.kt[j]);
    a.n0 = (float)(sk * c.c0);
    a.nx = (float)(sk * gauge_w(c, j, 0));
    a.ny = (float)(sk * gauge_w(c, j, 1));
    a.nz = (float)(sk * gauge_w(c, j, 2));
    a.a = (float)c.a[j];
    a.c1 = (float)w.c1[0][j];
    a.mc2 = (float)(-w.c2[0][j]);
    a.mith = (float)(-w.inv_theta[j]);
  }
  auto kern = k_gauge3d<R, NW, PF, MINB, START>;
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
  if (attr != cudaSuccess) return false;
  // START: v_1 into r[1], v_2 into d[0]; pass p >= 1 reads v from d[0] / r[1] and replaces the other
  float2* two[2] = {b.r[1], b.d[0]};
  const Gauge3Geom g{c.nx, c.ny, c.nz, Lz, (c.nx + TXV - 1) / TXV, c.pts};
  const dim3 grid((unsigned)(g.ntx * ((c.ny + TYV - 1) / TYV)), (unsigned)((c.nz + Lz - 1) / Lz), (unsigned)c.J);
  launch_dependent(kern, grid, SH::NT, SH::smem, s, in, g, START ? b.r0 : two[pass & 1], START ? two[1] : two[1 - (pass & 1)], b.u,
                                      START ? two[0] : nullptr, b.x64, b.ks, pass, kid);
  return true;
}

}  // namespace

}  // namespace apfc
