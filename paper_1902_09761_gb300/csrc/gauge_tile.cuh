// Chebyshev iteration on the Schur complement itself, 2D grids: the terms of gauge2d.cuh made on
// tiles held by one block.
//
// The streamed passes are a chain of rows: on small grids each SM holds a block or two whose every
// row waits for the last.  Here a block holds a region of 64 columns and R NW rows, a thread two
// columns of R rows (v, v_(n-1), b in registers), and every stage of a term is one step of the
// whole region: g' = N v, then v_(n+1), x-neighbours by shuffles (a warp spans the region), the
// rows above and below a warp's through shared memory, one barrier a stage.  UNITS x 3 terms need
// a halo of 6 UNITS points, which the region recomputes: (64 - 12 UNITS) x (R NW - 12 UNITS)
// points are the block's own.
//
// Blocks are persistent: while one tile is computed, every thread's own values of the next are on
// their way to its slots in shared memory (cp.async), so a launch of several rounds waits for
// memory once.
//
// Terms are counted in the streamed kernel's passes of three and evaluated by the same operations;
// only values carried across the periodic boundary inside a launch round differently.  What a point
// gets does not depend on the launch's other grids: a run of a batch equals the run alone.
//
// JAC: S = a + d(x) + kt G_h^2 with a Picard iteration's real diagonal d (SchurCoef's bounds widened
// by its range); d commutes with the gauge.  Its values wait in shared memory, two tiles deep.
#pragma once
#include "gauge2d.cuh"

namespace apfc {

namespace {

template <int NW, int R, int UNITS, bool START, bool JAC>
struct TileShape {
  static constexpr int H = 2 * kGaugeNI32 * UNITS, OX = 64, OY = R * NW, TX = OX - 2 * H, TY = OY - 2 * H;
  static constexpr int NF = START ? 1 : 3;  // fields staged: v (START: the residual), v_(n-1), b
  static constexpr size_t xrow = 2 * NW * 2 * 32, stage = (size_t)NF * R * NW * 32,  // in float4
                          diag = JAC ? 2ull * R * NW * 32 : 0;
  static constexpr size_t smem = sizeof(float4) * (xrow + stage + diag);
};

// Tiles of one grid.
struct TileGrid {
  int nx, ny, ns, ng;   // sizes, tiles along x and y
  long long pts, foff, xoff;
  int k0;               // its amplitudes' first entry in the table of units
};

// unit: first unit (three terms) of this launch; ks[].iters units in all.
template <int NW, int R, int UNITS, int MINB, bool START, bool JAC, class TAB>
__global__ void __launch_bounds__(32 * NW, MINB)
    k_gauge_tile(const __grid_constant__ GaugeParam<float> c, ChebGeom g1, int total, const float2* v_in,
                 const float2* vp_in, float2* v_out, float2* vp_out, float2* b_io, double2* x64, const float2* jd, const KScal* ks,
                 int unit, int kid, const __grid_constant__ TAB tab) {
  using SH = TileShape<NW, R, UNITS, START, JAC>;
  using C = float2;
  constexpr bool BATCH = std::is_same<TAB, ChebTab>::value;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  float4* xr = reinterpret_cast<float4*>(tile_smem);       // [v, g'][warp][first, last row][32]
  float4* stg = xr + SH::xrow + threadIdx.x;               // [field][row][thread]
  [[maybe_unused]] float4* dg = stg + SH::stage;           // JAC: [two tiles][row][thread]
  [[maybe_unused]] int dbuf = 0;                           // of the tile fetched last
  __shared__ int its[(BATCH ? kChebRuns : 1) * kMaxJ];
  const int t = threadIdx.x, px = t & 31, w = __shfl_sync(0xffffffffu, t >> 5, 0);
  const C one = make_float2(1.f, 0.f), zero = make_float2(0.f, 0.f);
  dependent_wait();
  if constexpr (BATCH) {
    for (int i = t; i < kChebRuns * c.J; i += 32 * NW) its[i] = ks[(long long)tab.run[i / c.J].run * c.J + i % c.J].iters;
  } else {
    if (t < c.J) its[t] = ks[t].iters;
  }
  __syncthreads();

  // tile `idx` of the launch: its grid, amplitude and first row and column
  TileGrid q;
  int j, X0, Y0, units;
  auto locate = [&](int idx) {
    if constexpr (BATCH) {
      int r = 0;
      while (idx >= tab.run[r].nblk) idx -= tab.run[r].nblk, ++r;
      const ChebRun& e = tab.run[r];
      q = TileGrid{e.nx, e.ny, e.nstrips, e.nsegs, e.pts, e.foff, e.xoff, r * c.J};
    } else {
      q = TileGrid{g1.nx, g1.ny, g1.nstrips, g1.nsegs, g1.pts, 0, 0, 0};
    }
    const int per = q.ns * q.ng;
    j = idx / per;
    idx -= j * per;
    const int sy = idx / q.ns;
    X0 = (idx - sy * q.ns) * SH::TX - SH::H + 2 * px;
    Y0 = sy * SH::TY - SH::H + R * w;
    units = its[q.k0 + j];
  };
  auto wrap_x = [&](int x) {
    x %= q.nx;
    return x < 0 ? x + q.nx : x;
  };
  auto first_row = [&]() {
    const int y = Y0 % q.ny;
    return y < 0 ? y + q.ny : y;
  };
  auto fetch = [&]() {  // the located tile's values of this thread on their way
    if (unit < units) {
      const long long o = q.foff + (long long)j * q.pts;
      const int x0 = wrap_x(X0), x1 = wrap_x(X0 + 1);
      const bool vec = (q.nx & 1) == 0;  // a pair never straddles the boundary and is 16-byte aligned
      int y = first_row();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const long long p = o + (long long)y * q.nx;
#pragma unroll
        for (int f = 0; f < SH::NF + JAC; ++f) {
          const C* src = (f == SH::NF ? jd : f == 0 ? v_in : f == 1 ? vp_in : b_io) + p;
          C* dst = reinterpret_cast<C*>(f == SH::NF ? dg + (dbuf * R + r) * (32 * NW) : stg + (f * R + r) * (32 * NW));
          if (vec) {
            cheb_cp_async16(dst, src + x0);
          } else {
            cheb_cp_async(dst, src + x0);
            cheb_cp_async(dst + 1, src + x1);
          }
        }
        y = y + 1 == q.ny ? 0 : y + 1;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };

  int idx = blockIdx.x;
  if (idx >= total) return;
  locate(idx);
  fetch();
  for (;;) {
    asm volatile("cp.async.wait_group 0;\n" ::);
    const int next = idx + (int)gridDim.x;
    if (unit >= units) {  // this amplitude is done
      if (next >= total) return;
      idx = next;
      locate(idx);
      fetch();
      continue;
    }
    C v[R][2], vp[R][2], b[R][2];
    auto take = [&](int f, C (&d)[R][2]) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 s = stg[(f * R + r) * (32 * NW)];
        d[r][0] = make_float2(s.x, s.y);
        d[r][1] = make_float2(s.z, s.w);
      }
    };
    take(0, v);
    if constexpr (!START) {
      take(1, vp);
      take(2, b);
    }
    const bool last = unit + UNITS >= units;
    const int terms = kGaugeNI32 * min(UNITS, units - unit);
    const TileGrid cq = q;
    const int cj = j, cX = X0, cY = Y0;
    const GaugeAmp<float>& q_ = c.amp[cj];
    const float n0 = q_.n0, nwx = q_.nx, nwy = q_.ny, aa = q_.a;
    const C* tabx = c.tab + (long long)cj * (c.tx + c.ty);
    const C* taby = tabx + c.tx;
    const long long fo = cq.foff + (long long)cj * cq.pts;
    if (c.prof != nullptr && t == 0 && cX == -SH::H && cY == -SH::H) {
      const unsigned long long f = sizeof(C), rd = START ? f : 3 * f, wr = START ? 3 * f : 2 * f;
      atomicAdd(c.prof + kid, (unsigned long long)cq.pts * (rd + (last ? 2 * sizeof(double2) : wr)));
    }
    const bool vec = (cq.nx & 1) == 0;
    const bool cown = 2 * px >= SH::H && 2 * px < SH::OX - SH::H;
    auto own = [&](int r, int k) {
      return cown && cX + k < cq.nx && R * w + r >= SH::H && R * w + r < SH::OY - SH::H && cY + r < cq.ny;
    };
    auto store = [&](C* dst, const C (&d)[R][2]) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        C* p = dst + fo + (long long)(cY + r) * cq.nx + cX;
        if (vec) {
          if (own(r, 0)) *reinterpret_cast<float4*>(p) = make_float4(d[r][0].x, d[r][0].y, d[r][1].x, d[r][1].y);
        } else {
          if (own(r, 0)) p[0] = d[r][0];
          if (own(r, 1)) p[1] = d[r][1];
        }
      }
    };
    // values beyond the grid are the periodic images' times the wraps' phases
    const int x0 = wrap_x(cX), x1 = wrap_x(cX + 1);
    int y = first_row(), my = (cY - y) / cq.ny;
    if constexpr (START) {
      const C cf0 = g_pow(tabx[cq.nx], (cX - x0) / cq.nx, one), cf1 = g_pow(tabx[cq.nx], (cX + 1 - x1) / cq.nx, one);
      const C pc[2] = {g_cmul(tabx[x0], cf0), g_cmul(tabx[x1], cf1)};
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const C pr = g_cmul(taby[y], g_pow(taby[cq.ny], my, one));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const C z = g_cmul(g_cmul(pr, pc[k]), v[r][k]);
          b[r][k] = make_float2(-z.x, -z.y);
          v[r][k] = q_mul(q_.mith, b[r][k]);
          vp[r][k] = zero;
        }
        if (++y == cq.ny) y = 0, ++my;
      }
      if (!last) store(b_io, b);
    } else {
      const int xt = cX - 2 * px, yt = cY - R * w;
      if (xt < 0 || yt < 0 || xt + SH::OX > cq.nx || yt + SH::OY > cq.ny) {
        const C cf[2] = {g_pow(tabx[cq.nx], (cX - x0) / cq.nx, one), g_pow(tabx[cq.nx], (cX + 1 - x1) / cq.nx, one)};
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const C rf = g_pow(taby[cq.ny], my, one);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const C f = g_cmul(rf, cf[k]);
            v[r][k] = g_cmul(f, v[r][k]);
            vp[r][k] = g_cmul(f, vp[r][k]);
            b[r][k] = g_cmul(f, b[r][k]);
          }
          if (++y == cq.ny) y = 0, ++my;
        }
      }
    }
    __syncthreads();  // the slots have been read
    [[maybe_unused]] const float4* dd = dg + dbuf * R * (32 * NW);
    if (next < total) {
      dbuf ^= 1;
      locate(next);
      fetch();
    }
    // out = n0 cc + nwx (l + r) + nwy (u + d) + add, in k_gauge2d's order
    auto exchange = [&](float4* s, const C (&cc)[R][2]) {
      s[(w * 2) * 32 + px] = make_float4(cc[0][0].x, cc[0][0].y, cc[0][1].x, cc[0][1].y);
      s[(w * 2 + 1) * 32 + px] = make_float4(cc[R - 1][0].x, cc[R - 1][0].y, cc[R - 1][1].x, cc[R - 1][1].y);
      __syncthreads();
    };
    auto stencil = [&](const float4* s, const C (&cc)[R][2], auto first, auto out) {
      const float4 uf = s[(w > 0 ? w * 2 - 1 : 0) * 32 + px], df = s[(w < NW - 1 ? w * 2 + 2 : 2 * NW - 1) * 32 + px];
      const C up[2] = {make_float2(uf.x, uf.y), make_float2(uf.z, uf.w)};
      const C dn[2] = {make_float2(df.x, df.y), make_float2(df.z, df.w)};
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const C L = make_float2(__shfl_up_sync(0xffffffffu, cc[r][1].x, 1), __shfl_up_sync(0xffffffffu, cc[r][1].y, 1));
        const C Q = make_float2(__shfl_down_sync(0xffffffffu, cc[r][0].x, 1), __shfl_down_sync(0xffffffffu, cc[r][0].y, 1));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const C l = k == 0 ? L : cc[r][0], rt = k == 1 ? Q : cc[r][1];
          const C u = r == 0 ? up[k] : cc[r > 0 ? r - 1 : 0][k], d = r == R - 1 ? dn[k] : cc[r < R - 1 ? r + 1 : 0][k];
          out(r, k, q_fma(nwy, q_add(u, d), q_fma(nwx, q_add(l, rt), first(r, k))));
        }
      }
    };
    for (int i = 0; i < terms; ++i) {
      C h[R][2];
      exchange(xr, v);
      stencil(xr, v, [&](int r, int k) { return q_mul(n0, v[r][k]); }, [&](int r, int k, C f) { h[r][k] = f; });
      exchange(xr + NW * 64, h);
      const float c1 = q_.c1[i], mc2 = q_.mc2[i];
      stencil(
          xr + NW * 64, h, [&](int r, int k) {
            float a = aa;
            if constexpr (JAC) a += k == 0 ? dd[r * (32 * NW)].x : dd[r * (32 * NW)].z;
            return q_fma(n0, h[r][k], q_fma(a, v[r][k], b[r][k]));
          },
          [&](int r, int k, C rh) {
            const C nv = q_fma(mc2, rh, q_fma(c1, q_sub(v[r][k], vp[r][k]), v[r][k]));
            vp[r][k] = v[r][k];
            v[r][k] = nv;
          });
    }
    if (!last) {
      store(v_out, v);
      store(vp_out, vp);
    } else {
      const C pc[2] = {tabx[x0], tabx[x1]};
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!own(r, 0)) continue;
        const C pr = taby[cY + r];
        double2* xp = x64 + cq.xoff + (2LL * cj + 1) * cq.pts + (long long)(cY + r) * cq.nx + cX;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (!own(r, k)) continue;
          const C un = g_cmul(g_conj(g_cmul(pr, pc[k])), v[r][k]);
          double2 xv = xp[k];
          xv.x += f2d(un.x);
          xv.y += f2d(un.y);
          xp[k] = xv;
        }
      }
    }
    if (next >= total) return;
    idx = next;
  }
}

// Launch `pass` of a solve: units UNITS pass .. UNITS pass + UNITS - 1.
template <int NW, int R, int UNITS, int MINB, bool START, bool JAC = false>
bool launch_tile_pass(const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, const ChebBufs<float>& b,
                      int pass, int sms, cudaStream_t s, const BatchLaunch* bl) {
  using SH = TileShape<NW, R, UNITS, START, JAC>;
  static_assert(kGaugeNI32 * UNITS <= kGaugeMaxNI && SH::H % 2 == 0 && SH::TX > 0 && SH::TY > 0, "tile");
  const int kid = kid_of<float>(KID_FUSED_APINV);
  ProfScope ps_(kid, s);
  const GaugeParam<float> in = gauge_param<float>(c, gt, w, kGaugeNI32 * UNITS);
  const int cur = pass & 1;
  const float2* vin = START ? b.r0 : b.r[cur];
  if (bl == nullptr) {
    auto kern = k_gauge_tile<NW, R, UNITS, MINB, START, JAC, ChebNoTab>;
    static const cudaError_t attr =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
    if (attr != cudaSuccess) return false;
    const ChebGeom g = cheb_geom(c.nx, c.ny, SH::H, SH::OX, SH::TY);
    const int total = g.nstrips * g.nsegs * c.J;
    launch_dependent(kern, std::min(total, MINB * sms), 32 * NW, SH::smem, s, in, g, total, vin, b.d[cur], b.r[1 - cur],
                                                                b.d[1 - cur], b.u, b.x64, c.jd32, b.ks, UNITS * pass,
                                                                kid, ChebNoTab{});
    return true;
  }
  if constexpr (JAC) return false;  // batched runs have no Jacobian
  auto kern = k_gauge_tile<NW, R, UNITS, MINB, START, false, ChebTab>;
  static const cudaError_t attr =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::smem);
  if (attr != cudaSuccess) return false;
  for (int r0 = 0; r0 < bl->R; r0 += kChebRuns) {
    ChebTab tab;
    int maxblk = 0, total = 0;
    const int nr = cheb_table(*bl, r0, SH::H, SH::OX, SH::TY, c.J, tab, maxblk, 1);
    for (int i = 0; i < nr; ++i) total += tab.run[i].nblk;
    if (total == 0) continue;
    kern<<<std::min(total, MINB * sms), 32 * NW, SH::smem, s>>>(in, ChebGeom{}, total, vin, b.d[cur], b.r[1 - cur],
                                                                b.d[1 - cur], b.u, b.x64, nullptr, b.ks, UNITS * pass,
                                                                kid, tab);
  }
  return true;
}

}  // namespace

}  // namespace apfc
