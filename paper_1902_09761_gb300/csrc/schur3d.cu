// The Schur-complement solve on 3D grids: the outer residual r = b - (a + kt G_h^2) eta and the
// passes of the Chebyshev iteration (gauge3d.cuh).
#include "gauge3d.cuh"
#include "resid_point.cuh"

namespace apfc {

namespace {

// Streams through a chunk of z-planes of a tile of 28 columns: a warp spans the columns with a halo of
// two on each side, a thread holds kR3R adjacent rows; at step t zeta = G_h eta is formed on plane
// t - 1 and r on plane t - 2, z-neighbours in registers, x- and y-neighbours from two-plane
// shared-memory rings.  The halo's outer rows only pass eta on, the next ones zeta.  Every double
// is split once (dfloat.cuh); arithmetic and rounding as in the 2D kernel (schur.cu).
// Sixteen warps of two rows, one block per SM: bound by the packed FP32 instructions (about 270 a
// point; with the halo they keep that pipe busy 52 per cent of the time) and the barriers between
// planes.  256^3 x 6: 4.21 ms, twelve warps 4.44, eight
// of two in two blocks 4.61, eight of four 5.02 (with two operations a term more); the 32 x 16 tile of
// 36-column cells before 4.63, with its rows across warps.  Now 3.93.
constexpr int kR3NW = 16, kR3R = 2, kR3B = 1, kR3NT = 32 * kR3NW;
constexpr int kR3X = 28, kR3OY = kR3NW * kR3R, kR3Y = kR3OY - 4;
constexpr int kR3RW = 34, kR3Plane = kR3OY * kR3RW, kR3PF = 1;

// G_h: centre, neighbour sums, neighbour differences (lane signs as in resid_coef); -kt G_h; -a
struct R3Coef {
  LaneC g0, gl[3], ga[3], k0, kl[3], ka[3], ma;
};
constexpr size_t kR3Smem = 2ull * 2 * kR3Plane * 16 + (size_t)(kR3PF + 1) * kR3NT * kR3R * sizeof(double2) + sizeof(R3Coef);

__global__ void __launch_bounds__(kR3NT, kR3B)
    k_resid_schur3d(const double2* b, double2* x, float2* __restrict__ r_out, double2* __restrict__ r64,
                    double* __restrict__ part, const __grid_constant__ OpCoef c, int Lz, int ntx, int want_b) {
  extern __shared__ __align__(16) unsigned char r3_smem[];
  float4* ring = reinterpret_cast<float4*>(r3_smem);  // [eta, zeta][2 planes][kR3Plane]
  double2* stg = reinterpret_cast<double2*>(ring + 4 * kR3Plane);
  R3Coef& q = *reinterpret_cast<R3Coef*>(stg + (kR3PF + 1) * kR3NT * kR3R);
  __shared__ double shn[2][kR3NW];
  constexpr int R = kR3R;
  const int j = blockIdx.z, t = threadIdx.x;
  const int w = __shfl_sync(0xffffffffu, t >> 5, 0), px = t & 31;
  const int tyi = blockIdx.x / ntx, txi = blockIdx.x - tyi * ntx;
  dependent_wait();
  const long long pts = c.pts, plane = (long long)c.nx * c.ny;
  if (c.prof != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && t == 0)
    atomicAdd(c.prof + KID_RESID_REFINE,
              (unsigned long long)pts * (3 * sizeof(double2) + sizeof(float2) +
                                         (r64 != nullptr ? sizeof(double2) : 0)));
  if (t == 0) {
    const ResidCoef<3> rc = resid_coef<3>(c, j);
    q.g0 = rc.g0;
    q.k0 = rc.k0;
    for (int d = 0; d < 3; ++d) q.gl[d] = rc.gl[d], q.ga[d] = rc.ga[d], q.kl[d] = rc.kl[d], q.ka[d] = rc.ka[d];
    q.ma = lane_c(c.a[j], -1.f, -1.f);
  }
  double2* zt = x + 2LL * j * pts;
  const double2* et = zt + pts;
  const double2* bt = b + (2LL * j + 1) * pts;
  const long long fo = (long long)j * pts;
  r_out += fo;
  if (r64 != nullptr) r64 += fo;
  const PDF zero{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  for (int i = t; i < 4 * kR3Plane; i += kR3NT) ring[i] = pdf_pack(zero);

  const int X = txi * kR3X - 2 + px, Y0 = tyi * kR3Y - 2 + R * w;
  int gx = X % c.nx;
  if (gx < 0) gx += c.nx;
  int off[R];
  bool own[R], zrow[R], rrow[R];  // zrow, rrow: zeta and r are formed on the row (uniform over the warp)
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int y = (Y0 + r) % c.ny;
    if (y < 0) y += c.ny;
    off[r] = y * c.nx + gx;
    zrow[r] = R * w + r >= 1 && R * w + r < kR3OY - 1;
    rrow[r] = R * w + r >= 2 && R * w + r < kR3OY - 2 && Y0 + r < c.ny;
    own[r] = px >= 2 && px < 30 && rrow[r] && X < c.nx;
  }
  const int z0 = blockIdx.y * Lz, nzc = min(c.nz, z0 + Lz) - z0, steps = nzc + 4;
  int fz = (z0 - 2) % c.nz;
  if (fz < 0) fz += c.nz;
  auto issue = [&](int tf, int slot) {
    if (tf < steps) {
      double2* d = stg + (size_t)slot * kR3NT * R + t;
      const double2* p = et + fz * plane;
#pragma unroll
      for (int r = 0; r < R; ++r) cheb_cp_async(d + r * kR3NT, p + off[r]);
      fz = cheb_wrap(fz, c.nz);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  PDF e1[R], e2[R], h1[R], h2[R];
  double2 bn[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    e1[r] = e2[r] = h1[r] = h2[r] = zero;
    bn[r] = make_double2(0.0, 0.0);
  }
  float rr = 0.f, bb = 0.f;
#pragma unroll
  for (int tf = 0; tf < kR3PF; ++tf) issue(tf, tf);
  __syncthreads();
  int slot = 0, islot = kR3PF;
  const int cell = R * w * kR3RW + px + 1;
  for (int tt = 0; tt < steps; ++tt) {
    issue(tt + kR3PF, islot);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kR3PF));
    const int par = tt & 1;
    const long long zo = (long long)(z0 + tt - 4) * plane;  // plane tt - 2, where r is formed
    double2 bc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) bc[r] = bn[r];
    if (tt >= 3 && tt + 1 < steps) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (own[r]) bn[r] = bt[zo + plane + off[r]];
    }
    PDF e0[R], h0[R];
    {
      const double2* st = stg + (size_t)slot * kR3NT * R + t;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        e0[r] = pdf_split(st[r * kR3NT]);
        ring[par * kR3Plane + cell + r * kR3RW] = pdf_pack(e0[r]);
      }
    }
    const float4* re = ring + (par ^ 1) * kR3Plane + cell;
    const float4* rz = re + 2 * kR3Plane;
    // zeta at plane tt - 1
#pragma unroll
    for (int r = 0; r < R; ++r) {
      h0[r] = zero;
      if (!zrow[r]) continue;
      const PDF l = pdf_unpack(re[r * kR3RW - 1]), rt = pdf_unpack(re[r * kR3RW + 1]);
      const PDF ym = r == 0 ? pdf_unpack(re[-kR3RW]) : e1[r > 0 ? r - 1 : 0];
      const PDF yp = r == R - 1 ? pdf_unpack(re[R * kR3RW]) : e1[r < R - 1 ? r + 1 : 0];
      double2 zd;
      {
        PAcc a;
        a.init(zero, c.zero);
        a.fma(q.g0.h, q.g0.l, e1[r]);
        a.fma(q.gl[0].h, q.gl[0].l, pdf_add(rt, l));
        a.fma(q.gl[1].h, q.gl[1].l, pdf_add(yp, ym));
        a.fma(q.gl[2].h, q.gl[2].l, pdf_add(e0[r], e2[r]));
        a.fma(q.ga[0].h, q.ga[0].l, pdf_swap(pdf_sub(rt, l)));
        a.fma(q.ga[1].h, q.ga[1].l, pdf_swap(pdf_sub(yp, ym)));
        a.fma(q.ga[2].h, q.ga[2].l, pdf_swap(pdf_sub(e0[r], e2[r])));
        a.result(h0[r].h, h0[r].l);
        zd = make_double2(df_to_d(DF{h0[r].h.x, h0[r].l.x}), df_to_d(DF{h0[r].h.y, h0[r].l.y}));
      }
      ring[(2 + par) * kR3Plane + cell + r * kR3RW] = pdf_pack(h0[r]);
      if (own[r] && tt >= 3 && tt < nzc + 3) zt[zo + plane + off[r]] = zd;
    }
    // r at plane tt - 2
    if (tt >= 4) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!rrow[r] || !own[r]) continue;
        const PDF l = pdf_unpack(rz[r * kR3RW - 1]), rt = pdf_unpack(rz[r * kR3RW + 1]);
        const PDF ym = r == 0 ? pdf_unpack(rz[-kR3RW]) : h1[r > 0 ? r - 1 : 0];
        const PDF yp = r == R - 1 ? pdf_unpack(rz[R * kR3RW]) : h1[r < R - 1 ? r + 1 : 0];
        const long long p = zo + off[r];
        {
          const PDF bp = pdf_split(bc[r]);
          PAcc a;
          a.init(bp, c.zero);
          a.fma(q.k0.h, q.k0.l, h1[r]);
          a.fma(q.kl[0].h, q.kl[0].l, pdf_add(rt, l));
          a.fma(q.kl[1].h, q.kl[1].l, pdf_add(yp, ym));
          a.fma(q.kl[2].h, q.kl[2].l, pdf_add(h0[r], h2[r]));
          a.fma(q.ka[0].h, q.ka[0].l, pdf_swap(pdf_sub(rt, l)));
          a.fma(q.ka[1].h, q.ka[1].l, pdf_swap(pdf_sub(yp, ym)));
          a.fma(q.ka[2].h, q.ka[2].l, pdf_swap(pdf_sub(h0[r], h2[r])));
          a.fma(q.ma.h, q.ma.l, e2[r]);
          float2 f, lo;
          a.result(f, lo);
          r_out[p] = f;
          if (r64 != nullptr) r64[p] = make_double2(df_to_d(DF{f.x, lo.x}), df_to_d(DF{f.y, lo.y}));
          rr = fmaf(f.x, f.x, fmaf(f.y, f.y, rr));
          if (want_b) bb = fmaf(bp.h.x, bp.h.x, fmaf(bp.h.y, bp.h.y, bb));
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      e2[r] = e1[r];
      e1[r] = e0[r];
      h2[r] = h1[r];
      h1[r] = h0[r];
    }
    slot = slot == kR3PF ? 0 : slot + 1;
    islot = islot == kR3PF ? 0 : islot + 1;
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  double rrd = (double)rr, bbd = (double)bb;
  for (int o = 16; o > 0; o >>= 1) {
    rrd += __shfl_xor_sync(0xffffffffu, rrd, o);
    bbd += __shfl_xor_sync(0xffffffffu, bbd, o);
  }
  if (px == 0) shn[0][w] = rrd, shn[1][w] = bbd;
  __syncthreads();
  const int npart = gridDim.x * gridDim.y, blk = blockIdx.y * gridDim.x + blockIdx.x;
  if (t < 2) {
    double v = 0.0;
    for (int i = 0; i < kR3NW; ++i) v += shn[t][i];
    part[(2LL * j + t) * npart + blk] = v;
  }
}

int resid3_planes(int nx, int ny, int nz, int J) {
  const long long tiles = (long long)((nx + kR3X - 1) / kR3X) * ((ny + kR3Y - 1) / kR3Y) * J;
  const long long rows = nz * tiles / 608;  // about four rounds of one block on each of 152 SMs
  return (int)std::min<long long>(nz, std::min<long long>(64, std::max<long long>(8, rows)));
}

}  // namespace

int schur_resid3_parts(int nx, int ny, int nz, int J) {
  const int Lz = resid3_planes(nx, ny, nz, J);
  return ((nx + kR3X - 1) / kR3X) * ((ny + kR3Y - 1) / kR3Y) * ((nz + Lz - 1) / Lz);
}

template <typename T>
bool launch_resid_schur3d(const double2* b, double2* x, cplx<T>* r, double2* r64, double* part, const OpCoef& c,
                          bool want_b, bool f64, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (!f64) {
      static const cudaError_t attr =
          cudaFuncSetAttribute(k_resid_schur3d, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kR3Smem);
      if (attr != cudaSuccess) return false;
      ProfScope ps_(KID_RESID_REFINE, s);
      const int Lz = resid3_planes(c.nx, c.ny, c.nz, c.J), ntx = (c.nx + kR3X - 1) / kR3X;
      launch_dependent(
          k_resid_schur3d, dim3(ntx * ((c.ny + kR3Y - 1) / kR3Y), (c.nz + Lz - 1) / Lz, c.J), kR3NT, kR3Smem, s,
          b, x, r, r64, part, c, Lz, ntx, want_b);
      return true;
    }
  }
  launch_resid64<T>(b, x, r, r64, part, c, want_b, schur_resid3_parts(c.nx, c.ny, c.nz, c.J), s, nullptr);
  return true;
}
template bool launch_resid_schur3d<float>(const double2*, double2*, float2*, double2*, double*, const OpCoef&, bool,
                                          bool, cudaStream_t);
template bool launch_resid_schur3d<double>(const double2*, double2*, double2*, double2*, double*, const OpCoef&, bool,
                                           bool, cudaStream_t);

// Planes per chunk: the blocks of the busiest multiprocessor (in rounds of those resident) times
// the planes each streams, four of them halo.
static int gauge3_planes(const OpCoef& c, int txv, int tyv, int res, int sms) {
  const long long tiles = (long long)((c.nx + txv - 1) / txv) * ((c.ny + tyv - 1) / tyv) * c.J;
  double best = 1e300;
  int bl = c.nz;
  for (int n = 1; n <= c.nz; ++n) {
    const int Lz = (c.nz + n - 1) / n;
    const long long per = (tiles * ((c.nz + Lz - 1) / Lz) + sms - 1) / sms;
    const long long full = per / res, rest = per - full * res;
    const double t = (full * res * 0.6 + (rest > 0 ? std::max(1.0, rest * 0.6) : 0.0)) * (Lz + 5);
    if (t < best) best = t, bl = Lz;
    if (Lz <= 4) break;
  }
  return bl;
}

// Tiles of 60 columns: of 28 rows (eight warps of four, one block per SM) or of 12 (eight warps of
// two, two blocks), one plane ahead.  Measured at 256^3 x 6 (us a term; its 32 bytes a point take
// 481 at the copy rate): 28 rows 670, 12 rows 745 (718 with every x-neighbour from shared memory);
// 26 rows in ten warps of three 727, 28 in sixteen of two 720; v_(n-1) and b through shared memory
// 702 to 816.  A covered row costs the tall tile 0.85 of the short one's; with fewer than two
// rounds of blocks the short one's finer grain wins (70 x 90 x 101: 54 against 58).
bool launch_gauge3d(const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, const ChebBufs<float>& b,
                    int pass, int sms, cudaStream_t s) {
  const long long rows28 = (c.ny + 27) / 28, rows12 = (c.ny + 11) / 12;
  const long long blocks = (c.nx + 59) / 60 * rows28 * ((c.nz + 31) / 32) * c.J;
  if (0.85 * 28 * rows28 < 12.0 * rows12 && blocks >= 2 * sms) {
    const int Lz = gauge3_planes(c, 60, 28, 1, sms);
    return pass == 0 ? launch_gauge3_pass<4, 8, 1, 1, true>(c, gt, w, Lz, b, pass, s)
                     : launch_gauge3_pass<4, 8, 1, 1, false>(c, gt, w, Lz, b, pass, s);
  }
  const int Lz = gauge3_planes(c, 60, 12, 2, sms);
  return pass == 0 ? launch_gauge3_pass<2, 8, 1, 2, true>(c, gt, w, Lz, b, pass, s)
                   : launch_gauge3_pass<2, 8, 1, 2, false>(c, gt, w, Lz, b, pass, s);
}

}  // namespace apfc
