// Complex inner products (u, v) = sum conj(u) v per amplitude (Sec. II.A's L2
// product, conjugate-linear in the first argument) and the per-amplitude
// BiCGStab scalar updates that consume them.
//
// FP64 fields accumulate in FP64.  FP32 fields accumulate in FP32 with
// Neumaier-compensated summation (each partial is a (sum, compensation) pair)
// through the thread, block and final stages; the fixed reduction tree makes
// every result deterministic.
#include "acc.cuh"
#include "apfc_internal.cuh"
#include "bf16pair.cuh"

namespace apfc {

namespace {

template <typename T, int NP>
__global__ void k_dots(DotPairs<T> pr, void* partials, OpCoef c, const KScal* act) {
  const int j = blockIdx.y;
  if (act != nullptr && act[j].active == 0) return;
  const long long n = 2LL * c.pts;
  const long long o = 2LL * j * c.pts;
  if (c.prof != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
    // count each distinct array once
    const void* seen[2 * NP];
    int ns = 0;
    for (int q = 0; q < 2 * NP; ++q) {
      const void* ptr = q < NP ? (const void*)pr.u[q] : (const void*)pr.v[q - NP];
      bool dup = false;
      for (int r = 0; r < ns; ++r) dup = dup || seen[r] == ptr;
      if (!dup) seen[ns++] = ptr;
    }
    atomicAdd(c.prof + kid_of<T>(KID_DOTS), (unsigned long long)ns * n * sizeof(cplx<T>));
  }
  Acc<T> acc[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) acc[q].zero();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int q = 0; q < NP; ++q) acc[q].add(pr.u[q][o + i], pr.v[q][o + i]);
  }
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    block_reduce<T>(acc[q]);
    if (threadIdx.x == 0) acc[q].store(partials, (long long)(j * kDotSlots + q) * kDotBlocks + blockIdx.x);
  }
}

// Reduce the partial sums of amplitude j (slots (j kDotSlots + q) npart + b)
// and apply the scalar update `op` to its Krylov scalars.
template <typename T, int NP>
__device__ void finalize_one(const void* partials, int npart, int j, KScal& k, int op) {
  // a pending final update was applied after the previous OP_OMEGA5: clear the flag
  if (op == OP_ALPHA && threadIdx.x == 0) k.just_done = 0;
  if (op != OP_INIT && op != OP_INIT3 && op != OP_NORMS && op != OP_RNORM && op != OP_BNORM && k.active == 0) return;
  __shared__ double2 res[kDotSlots];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    Acc<T> a;
    a.zero();
    for (int b = threadIdx.x; b < npart; b += blockDim.x) {
      Acc<T> t;
      t.load(partials, (long long)(j * kDotSlots + q) * npart + b);
      a.merge(t);
    }
    block_reduce<T>(a);
    if (threadIdx.x == 0) res[q] = a.value();
  }
  if (threadIdx.x == 0) scalar_update(k, op, res);
}

// Start of an FP32 solve from x0 = 0, in one pass: r = b, rhat = b rounded to bf16 with its
// packed copy rh16 (bf16pair.cuh), and the partial sums of (r, r), (b, b) and (rhat, r) in
// slots 0-2, laid out as k_dots'.
__global__ void __launch_bounds__(kThreads) k_init32(const float2* __restrict__ b, float2* __restrict__ r,
                                                     float2* __restrict__ rhat, uint2* __restrict__ rh16,
                                                     void* partials, OpCoef c) {
  const int j = blockIdx.y;
  const long long pts = c.pts, o1 = 2LL * j * pts, o2 = o1 + pts;
  uint2* q = rh16 + (long long)j * pts;
  if (c.prof != nullptr && blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(c.prof + kid_of<float>(KID_DOTS), (unsigned long long)pts * (6 * sizeof(float2) + sizeof(uint2)));
  Acc<float> a0, a2;
  a0.zero();
  a2.zero();
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < pts; p += (long long)gridDim.x * blockDim.x) {
    const float2 b1 = b[o1 + p], b2 = b[o2 + p];
    r[o1 + p] = b1;
    r[o2 + p] = b2;
    const unsigned h1 = bf16_pack(b1), h2 = bf16_pack(b2);
    const float2 s1 = bf16_unpack(h1), s2 = bf16_unpack(h2);
    rhat[o1 + p] = s1;
    rhat[o2 + p] = s2;
    q[p] = make_uint2(h1, h2);
    a0.add(b1, b1);
    a0.add(b2, b2);
    a2.add(s1, b1);
    a2.add(s2, b2);
  }
  block_reduce<float>(a0);
  if (threadIdx.x == 0) {
    a0.store(partials, (long long)(j * kDotSlots + 0) * kDotBlocks + blockIdx.x);
    a0.store(partials, (long long)(j * kDotSlots + 1) * kDotBlocks + blockIdx.x);  // (b, b) = (r, r)
  }
  block_reduce<float>(a2);
  if (threadIdx.x == 0) a2.store(partials, (long long)(j * kDotSlots + 2) * kDotBlocks + blockIdx.x);
}

template <typename T, int NP>
__global__ void k_finalize(const void* partials, int npart, KScal* ks, int op) {
  finalize_one<T, NP>(partials, npart, blockIdx.x, ks[blockIdx.x], op);
}

}  // namespace

void launch_init32(const float2* b, float2* r, float2* rhat, uint2* rh16, void* partials, const OpCoef& c,
                   cudaStream_t s) {
  ProfScope ps_(kid_of<float>(KID_DOTS), s);
  k_init32<<<dim3(kDotBlocks, c.J), kThreads, 0, s>>>(b, r, rhat, rh16, partials, c);
}

template <typename T>
void launch_dots(int npair, const DotPairs<T>& pr, void* partials, const OpCoef& c, const KScal* act, cudaStream_t s) {
  const dim3 g(kDotBlocks, c.J);
  ProfScope ps_(kid_of<T>(KID_DOTS), s);
  if (npair == 1)
    k_dots<T, 1><<<g, kThreads, 0, s>>>(pr, partials, c, act);
  else if (npair == 2)
    k_dots<T, 2><<<g, kThreads, 0, s>>>(pr, partials, c, act);
  else
    k_dots<T, 3><<<g, kThreads, 0, s>>>(pr, partials, c, act);
}

template <typename T>
void launch_finalize(int npair, const void* partials, KScal* k, int op, int J, cudaStream_t s, int npart) {
  ProfScope ps_(kid_of<T>(KID_FINALIZE), s);
  if (npair == 1)
    k_finalize<T, 1><<<J, kThreads, 0, s>>>(partials, npart, k, op);
  else if (npair == 2)
    k_finalize<T, 2><<<J, kThreads, 0, s>>>(partials, npart, k, op);
  else if (npair == 3)
    k_finalize<T, 3><<<J, kThreads, 0, s>>>(partials, npart, k, op);
  else
    k_finalize<T, 5><<<J, kThreads, 0, s>>>(partials, npart, k, op);
}

void launch_finalize64(int npair, const void* partials, KScal* k, int op, int J, cudaStream_t s) {
  launch_finalize<double>(npair, partials, k, op, J, s);
}

template void launch_dots<double>(int, const DotPairs<double>&, void*, const OpCoef&, const KScal*, cudaStream_t);
template void launch_dots<float>(int, const DotPairs<float>&, void*, const OpCoef&, const KScal*, cudaStream_t);
template void launch_finalize<double>(int, const void*, KScal*, int, int, cudaStream_t, int);
template void launch_finalize<float>(int, const void*, KScal*, int, int, cudaStream_t, int);

}  // namespace apfc
