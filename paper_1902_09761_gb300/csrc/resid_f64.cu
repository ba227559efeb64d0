// The outer residual of the Schur-complement solve in FP64 arithmetic: r = b - (a + d) eta - kt G_h zeta
// with zeta = G_h eta, two kernels with a thread per point.
//
// Bound by the FP64 pipe (two operations a clock and multiprocessor; a point costs 18 and about 32):
// the streamed kernels' halos computed 1.1 to 1.5 times the points, so zeta goes through memory,
// where it belongs anyway.  Wrapped neighbours are chosen by index, outside the pipe.  us, three
// amplitudes at 512^2 / six at 64^3: streamed 160 / 413, here 91 / 218.
#include "apfc_internal.cuh"

namespace apfc {

namespace {

template <int DIM>
struct R64Point {
  long long p, xm, xp, ym, yp, zm, zp;
  bool in;
};
template <int DIM>
__device__ __forceinline__ long long r64_tiles(int nx, int ny, int nz) {
  return (long long)((nx + 31) / 32) * ((ny + 7) / 8) * (DIM == 3 ? nz : 1);
}
template <int DIM>
__device__ __forceinline__ R64Point<DIM> r64_point(long long tile, int nx, int ny, int nz) {
  const unsigned ntx = (nx + 31) / 32, nty = (ny + 7) / 8;
  const long long row = tile / ntx;
  const int z = DIM == 3 ? (int)(row / nty) : 0;
  const int x = (int)(tile - row * ntx) * 32 + (threadIdx.x & 31);
  const int y = (int)(row - (long long)z * nty) * 8 + (threadIdx.x >> 5);
  const long long plane = (long long)nx * ny;
  R64Point<DIM> n;
  n.in = x < nx && y < ny;
  n.p = z * plane + (long long)y * nx + x;
  n.xm = x == 0 ? n.p + nx - 1 : n.p - 1;
  n.xp = x + 1 == nx ? n.p - x : n.p + 1;
  n.ym = y == 0 ? n.p + (long long)(ny - 1) * nx : n.p - nx;
  n.yp = y + 1 == ny ? n.p - (long long)y * nx : n.p + nx;
  if constexpr (DIM == 3) {
    n.zm = z == 0 ? n.p + (nz - 1) * plane : n.p - plane;
    n.zp = z + 1 == nz ? n.p - z * plane : n.p + plane;
  }
  return n;
}
template <int DIM>
__device__ __forceinline__ double2 r64_G(const double2* u, double2 uc, const R64Point<DIM>& n, const OpCoef& c, int j) {
  double2 g = make_double2(c.c0 * uc.x, c.c0 * uc.y);
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const double2 m = u[d == 0 ? n.xm : d == 1 ? n.ym : n.zm], p = u[d == 0 ? n.xp : d == 1 ? n.yp : n.zp];
    const double h = c.ih2[d], k = c.kh[j][d];
    g.x = fma(-k, p.y - m.y, fma(h, p.x + m.x, g.x));
    g.y = fma(k, p.x - m.x, fma(h, p.y + m.y, g.y));
  }
  return g;
}

// The run of a batch (blockIdx.z), else the grid of c.
struct R64Geom {
  int nx, ny, nz;
  long long pts, xoff, foff, poff;
  int npart;
};
__device__ __forceinline__ R64Geom r64_geom(const OpCoef& c, const RunGeom* rg) {
  R64Geom g{c.nx, c.ny, c.nz, c.pts, 0, 0, 0, (int)gridDim.x};
  if (rg != nullptr) {
    const RunGeom& q = rg[blockIdx.z];
    g = R64Geom{q.nx, q.ny, 1, q.pts, q.elem_off, q.field_off, q.part_off_r, q.npart_r};
  }
  return g;
}

template <int DIM>
__global__ void __launch_bounds__(256) k_zeta64(double2* x, const __grid_constant__ OpCoef c, const RunGeom* rg) {
  dependent_wait();
  const R64Geom g = r64_geom(c, rg);
  if ((int)blockIdx.x >= g.npart) return;
  const int j = blockIdx.y;
  double2* zt = x + g.xoff + 2LL * j * g.pts;
  const double2* et = zt + g.pts;
  const long long nt = r64_tiles<DIM>(g.nx, g.ny, g.nz);
  for (long long i = blockIdx.x; i < nt; i += g.npart) {
    const R64Point<DIM> n = r64_point<DIM>(i, g.nx, g.ny, g.nz);
    if (n.in) zt[n.p] = r64_G<DIM>(et, et[n.p], n, c, j);
  }
}

template <int DIM, typename RT>
__global__ void __launch_bounds__(256)
    k_resid64(const double2* b, const double2* x, RT* __restrict__ r_out,
              double2* __restrict__ r64, double* __restrict__ part, const __grid_constant__ OpCoef c, int want_b,
              const RunGeom* rg) {
  dependent_wait();
  const R64Geom g = r64_geom(c, rg);
  if ((int)blockIdx.x >= g.npart) return;
  const int j = blockIdx.y;
  if (c.prof != nullptr && blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(c.prof + KID_RESID_REFINE, (unsigned long long)g.pts * (5 * sizeof(double2) + sizeof(RT) +
                                                                     (r64 != nullptr ? sizeof(double2) : 0)));
  const double2* zt = x + g.xoff + 2LL * j * g.pts;
  const double2* et = zt + g.pts;
  const double2* bt = b + g.xoff + (2LL * j + 1) * g.pts;
  const long long fo = g.foff + (long long)j * g.pts;
  const double kt = c.kt[j], a = c.a[j];
  double rr = 0.0, bb = 0.0;
  const long long nt = r64_tiles<DIM>(g.nx, g.ny, g.nz);
  for (long long i = blockIdx.x; i < nt; i += g.npart) {
    const R64Point<DIM> n = r64_point<DIM>(i, g.nx, g.ny, g.nz);
    if (!n.in) continue;
    const double2 G = r64_G<DIM>(zt, zt[n.p], n, c, j), e = et[n.p], bv = bt[n.p];
    const double ap = c.jd != nullptr ? a + c.jd[(long long)j * g.pts + n.p] : a;
    const double2 rv = make_double2(bv.x - fma(kt, G.x, ap * e.x), bv.y - fma(kt, G.y, ap * e.y));
    if constexpr (sizeof(RT) == 16)
      r_out[fo + n.p] = rv;
    else
      r_out[fo + n.p] = make_float2((float)rv.x, (float)rv.y);
    if (r64 != nullptr) r64[fo + n.p] = rv;
    rr = fma(rv.x, rv.x, fma(rv.y, rv.y, rr));
    if (want_b) bb = fma(bv.x, bv.x, fma(bv.y, bv.y, bb));
  }
  __shared__ double sh[2][8];
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
    bb += __shfl_xor_sync(0xffffffffu, bb, o);
  }
  if ((threadIdx.x & 31) == 0) sh[0][threadIdx.x >> 5] = rr, sh[1][threadIdx.x >> 5] = bb;
  __syncthreads();
  if (threadIdx.x < 2) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += sh[threadIdx.x][w];
    part[g.poff + (2LL * j + threadIdx.x) * g.npart + blockIdx.x] = v;
  }
}

}  // namespace

// npart: partial sums per amplitude (batched: the most of a run)
template <typename T>
void launch_resid64(const double2* b, double2* x, cplx<T>* r, double2* r64, double* part, const OpCoef& c, bool want_b,
                    int npart, cudaStream_t s, const BatchLaunch* bl) {
  ProfScope ps_(KID_RESID_REFINE, s);
  const dim3 grid(npart, c.J, bl != nullptr ? bl->R : 1);
  const RunGeom* rg = bl != nullptr ? bl->dev : nullptr;
  if (c.dim == 3) {
    launch_dependent(k_zeta64<3>, grid, 256, 0, s, x, c, rg);
    launch_dependent(k_resid64<3, cplx<T>>, grid, 256, 0, s, b, x, r, r64, part, c, want_b, rg);
  } else {
    launch_dependent(k_zeta64<2>, grid, 256, 0, s, x, c, rg);
    launch_dependent(k_resid64<2, cplx<T>>, grid, 256, 0, s, b, x, r, r64, part, c, want_b, rg);
  }
}
template void launch_resid64<float>(const double2*, double2*, float2*, double2*, double*, const OpCoef&, bool, int,
                                    cudaStream_t, const BatchLaunch*);
template void launch_resid64<double>(const double2*, double2*, double2*, double2*, double*, const OpCoef&, bool, int,
                                     cudaStream_t, const BatchLaunch*);

}  // namespace apfc
