// Batched independent runs: many 2D simulations of one lattice, parameter set
// and spacing on grids of different sizes, advanced together.  Every stage of
// the step (arXiv:1902.09761, Alg. 1 with the nonlinear term explicit; FP32
// Chebyshev solves of the Schur complement with the Sec. II.B preconditioner in
// FP64 iterative refinement, cheb2d.cuh) is one launch over the work items of
// all runs: the fields of the runs sit one after another in shared arrays, a run
// table maps each block of a launch to (run, strip, row segment, amplitude), and
// each (run, amplitude) takes its own number of passes.  A run that has
// converged idles (its blocks return at once) while the others go on.  The
// passes of a solve can be replayed from captured CUDA graphs.
//
// Where the Chebyshev iteration does not serve (tolerances beneath its residual's noise, more
// terms than max_iter allows) the solves are BiCGStab on the block system (FP32 in FP64
// refinement, fused2d.cuh), batched the same way: each (run, amplitude) keeps its own Krylov
// scalars.  Run by run on contexts of their own, 24 runs of 96^2 to 256^2 took 3 to 10 times as
// long (h = 0.7, dt = 10, tol 1e-12: 71 against 517 ms a step).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "host_common.h"

using namespace apfc;

namespace {

constexpr int kMaxRuns = 65536;
constexpr int kTunePasses = 6;     // Chebyshev passes or BiCGStab iterations timed per autotuner candidate
constexpr int kBlocks = 10;        // BiCGStab: r, rhat, p, v, u, t, r32, p', v', r'
constexpr int kBicgRows = 128;     // its rows per block segment when opts.tile_rows is 0
constexpr int kTuneRows[] = {32, 48, 64, 96, 128, 192, 256};

}  // namespace

struct apfc_batch {
  apfc_lattice lat{};
  apfc_params par{};
  apfc_opts opts{};
  apfc_grid gmax{};  // largest nx, largest ny, and the spacings
  int R = 0, J = 0, flags = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<int> nx, ny;
  std::vector<RunGeom> rg;  // run table
  RunGeom* rg_dev = nullptr;
  BatchLaunch bl{};
  long long elems = 0;   // complex entries of one concatenated block vector
  long long felems = 0;  // and of one concatenated field (each run's start padded to 128 bytes)
  int auto_rows = 0;     // rows per segment when opts.tile_rows is 0
  int sms = 152;
  NonlinTable nt{};
  EnergyTable et{};
  OpCoef coef{};  // sizes of the largest run; kernels take each run's own from the table
  double coef_dt = -1.0;
  std::vector<ChebStep> cw;
  double2* x64 = nullptr;
  double2* b64 = nullptr;
  double2* b64_prev = nullptr;
  double2* r64_prev = nullptr;
  float2* r[2] = {};  // residual and d ping-pong pairs and the sum u (cheb2d.cuh), fields [run][J][pts]
  float2* d[2] = {};
  float2* u = nullptr;
  float2* tab = nullptr;     // phases of the gauge (gauge2d.cuh), for the largest grid
  double* rpart = nullptr;   // residual kernel partials, [run][J][2][npart_r]
  void* part_fix = nullptr;  // right-hand-side kernel partials: R J kDotSlots kDotBlocks slots
  SchurCoef schur{};
  bool schur_ok = false;
  // BiCGStab on the block system (alloc_bicg)
  float2* blk[kBlocks] = {};
  uint2* rh16 = nullptr;         // rhat as packed bf16 pairs, [run][J][pts] (bf16pair.cuh)
  double2* r64_blk = nullptr;    // the last step's residual
  void* part_pipe = nullptr;     // fused-pipeline partials (run table layout)
  long long part_pipe_cap = 0;
  KScal* ks = nullptr;
  KScal* ks_host = nullptr;
  BatchLaunch bl_t{};            // t-kernel partial layout (its own tile variant)
  int layout[4] = {-1, 0, 0, 0}; // tile, rows, tile_t, degree that the run table's partial layouts belong to
  cudaGraphExec_t gblock[2] = {nullptr, nullptr};  // captured iterations, by starting side of the ping-pong buffers
  KScal* ks64 = nullptr;
  KScal* ks64_host = nullptr;
  double* epart = nullptr;
  double* eout = nullptr;
  double* eout_host = nullptr;
  bool have_prev = false;
  bool prev_schur = false;  // r64_prev holds the previous residual, else r64_blk
  double prev_dt = 0.0;
  std::vector<char> has_state;
  std::vector<apfc_stats_t> stats;
  bool failed = false;
  std::string err;
  std::map<int, cudaGraphExec_t> gexec;  // captured solves by their number of passes
  bool ran = false;                      // a solve has run uncaptured (kernels are loaded)
  long long graph_replays = 0;
};

namespace {

apfc_status bfail(apfc_batch* b, apfc_status s, const std::string& msg) {
  if (b) {
    b->err = msg;
    if (s == APFC_ECUDA || s == APFC_ENAN || s == APFC_ENOMEM || s == APFC_ENOCONV) b->failed = true;
  }
  return s;
}

#define BK(call)                                                                              \
  do {                                                                                        \
    cudaError_t e_ = (call);                                                                  \
    if (e_ != cudaSuccess)                                                                    \
      return bfail(b, e_ == cudaErrorMemoryAllocation ? APFC_ENOMEM : APFC_ECUDA,             \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                       \
  } while (0)

int rows_of(const apfc_batch* b) { return b->opts.tile_rows > 0 ? b->opts.tile_rows : b->auto_rows; }

// Offsets of every run in the concatenated arrays.  False when a fused launch could exceed the
// grid limit.
bool make_table(apfc_batch* b) {
  std::vector<RunGeom>& t = b->rg;
  t.resize(b->R);
  long long eoff = 0, foff = 0, poff = 0;
  for (int r = 0; r < b->R; ++r) {
    RunGeom& g = t[r];
    std::memset(&g, 0, sizeof(g));
    g.nx = b->nx[r];
    g.ny = b->ny[r];
    g.pts = (long long)g.nx * g.ny;
    g.elem_off = eoff;
    g.field_off = foff;
    g.part_off_r = poff;
    g.rows_r = schur_resid_rows(g.nx, g.ny, b->J);
    g.npart_r = schur_resid_parts(g.nx, g.ny, b->J);
    eoff += 2LL * b->J * g.pts;
    foff += (b->J * g.pts + 15) / 16 * 16;
    poff += 2LL * b->J * g.npart_r;
    for (int rows : {8, b->opts.tile_rows})
      if (rows > 0 && (long long)((g.nx + 7) / 8) * ((g.ny + rows - 1) / rows) * b->J > 0x7fffffffLL) return false;
  }
  b->elems = eoff;
  b->felems = foff;
  return true;
}

void drop_graphs(apfc_batch* b) {
  for (auto& g : b->gexec) cudaGraphExecDestroy(g.second);
  b->gexec.clear();
  for (auto& g : b->gblock)
    if (g) cudaGraphExecDestroy(g), g = nullptr;
}

// The automatic segment height of the current options and coefficients.
void set_rows(apfc_batch* b) {
  b->auto_rows = schur_auto_rows(b->schur, b->nx.data(), b->ny.data(), b->R, b->J, b->opts.cheb_degree, (int)sizeof(float2),
                                 b->opts.tile, b->sms);
}

bool set_coef(apfc_batch* b, double dt, std::string& e) {
  if (b->coef_dt == dt) return true;
  if (!make_coef(b->lat, b->par, b->gmax, b->opts.tau_mode, dt, b->coef, e)) return false;
  b->cw = cheb_weights_for(b->coef, b->gmax, b->opts.cheb_degree);
  b->schur_ok = schur_build(b->coef, b->gmax, b->opts.cheb_degree, b->schur) && schur_resid_ok(b->schur, b->opts.tol);
  for (int j = 0; j < b->J && b->schur_ok; ++j)
    b->schur_ok = schur_terms(b->opts.tol_inner, b->schur.lnrate[j]) <= 2LL * b->opts.max_iter;
  b->coef_dt = dt;
  set_rows(b);
  drop_graphs(b);  // the captured launches hold the coefficients by value
  return true;
}

OpCoef run_coef(const apfc_batch* b, int r) {
  OpCoef c = b->coef;
  c.nx = b->nx[r];
  c.ny = b->ny[r];
  c.nz = 1;
  c.pts = (long long)c.nx * c.ny;
  return c;
}

// The first np passes of a solve over all runs.
bool issue_passes(apfc_batch* b, int np, int tile, int rows) {
  const int m = b->opts.cheb_degree;
  const GaugeTab<float> gt{b->tab, b->gmax.n[0] + 1, b->gmax.n[1] + 1, 0};
  const ChebBufs<float> bufs{b->r[0], {b->r[0], b->r[1]}, {b->d[0], b->d[1]}, b->u, b->x64, b->ks64};
  return launch_schur_passes<float>(b->schur, m, tile, b->coef, b->cw.data(), gt, rows, bufs, np, b->stream, b->sms, &b->bl);
}

apfc_status sync_ks(apfc_batch* b, KScal* dev, KScal* host) {
  BK(cudaGetLastError());
  BK(cudaMemcpyAsync(host, dev, sizeof(KScal) * b->R * b->J, cudaMemcpyDeviceToHost, b->stream));
  BK(cudaStreamSynchronize(b->stream));
  return APFC_OK;
}

SchurPlan plan_of(const apfc_batch* b) {
  SchurPlan p{};
  const int m = b->opts.cheb_degree, ni = schur_ni<float>(b->schur, 2, m);
  p.tol = b->opts.tol;
  p.tol_inner = b->opts.tol_inner;
  for (int j = 0; j < b->J; ++j) p.lnrate[j] = b->schur.lnrate[j];
  p.t0 = schur_t0<float>(b->schur, 2, m);
  p.ni = ni;
  p.max_pass = (int)std::min<long long>(1 << 30, std::max(1LL, (2LL * b->opts.max_iter - p.t0 + ni - 1) / ni));
  p.J = b->J;
  return p;
}

// One solve of np passes: every (run, amplitude) takes its own ks64[].iters of them and adds
// its correction to the state.
apfc_status solve(apfc_batch* b, int np) {
  const int tile = b->opts.tile, rows = rows_of(b);
  if ((b->flags & APFC_BATCH_GRAPH) && !profiler_on() && b->ran) {
    cudaGraphExec_t& ge = b->gexec[np];
    if (!ge) {
      cudaGraph_t g = nullptr;
      BK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
      const bool ok = issue_passes(b, np, tile, rows);
      const cudaError_t ec = cudaStreamEndCapture(b->stream, &g);
      if (!ok || ec != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        b->gexec.erase(np);
        BK(ec);
        return bfail(b, APFC_ECUDA, "the Chebyshev passes cannot be launched");
      }
      const cudaError_t ei = cudaGraphInstantiate(&ge, g, 0);
      cudaGraphDestroy(g);
      if (ei != cudaSuccess) b->gexec.erase(np);
      BK(ei);
    }
    BK(cudaGraphLaunch(ge, b->stream));
    b->graph_replays += 1;
    return APFC_OK;
  }
  if (!issue_passes(b, np, tile, rows)) return bfail(b, APFC_ECUDA, "the Chebyshev passes cannot be launched");
  b->ran = true;
  return APFC_OK;
}

// ---- BiCGStab on the block system ------------------------------------------
int bicg_rows(const apfc_opts& o) { return o.tile_rows > 0 ? o.tile_rows : kBicgRows; }
int tile_t_of(const apfc_opts& o) { return o.tile_t >= 0 ? o.tile_t : o.tile; }

apfc_status alloc_bicg(apfc_batch* b) {
  if (b->ks_host) return APFC_OK;
  const size_t n = (size_t)b->elems, nks = sizeof(KScal) * (size_t)b->R * b->J;
  for (auto& q : b->blk)
    if (!q) BK(cudaMalloc(&q, sizeof(float2) * n));
  if (!b->rh16) BK(cudaMalloc(&b->rh16, sizeof(uint2) * (n / 2)));
  if (!b->r64_blk) BK(cudaMalloc(&b->r64_blk, sizeof(double2) * n));
  if (!b->ks) BK(cudaMalloc(&b->ks, nks));
  BK(cudaMallocHost(&b->ks_host, nks));
  return APFC_OK;
}

// The partial-sum offsets of (tile, rows) of the v-kernel and tile_t of the t-kernel into the run table.
apfc_status set_layout(apfc_batch* b, int tile, int rows, int tile_t) {
  apfc_status st = alloc_bicg(b);
  if (st != APFC_OK) return st;
  const int m = b->opts.cheb_degree, eb = (int)sizeof(float2), want[4] = {tile, rows, tile_t, m};
  if (std::equal(want, want + 4, b->layout)) return APFC_OK;
  long long poff = 0, poff_t = 0;
  for (RunGeom& g : b->rg) {
    g.part_off = poff;
    g.part_off_t = poff_t;
    fused2d_blocks(g.nx, g.ny, b->J, m, rows, eb, tile, true, &g.npart);
    fused2d_blocks(g.nx, g.ny, b->J, m, rows, eb, tile_t, true, &g.npart_t);
    poff += (long long)b->J * kDotSlots * g.npart;
    poff_t += (long long)b->J * kDotSlots * g.npart_t;
  }
  b->layout[0] = -1;  // until the table is on the device
  const long long need = std::max(poff, poff_t);  // the two kernels use the buffer in turn
  BK(cudaMemcpyAsync(b->rg_dev, b->rg.data(), sizeof(RunGeom) * b->R, cudaMemcpyHostToDevice, b->stream));
  BK(cudaStreamSynchronize(b->stream));
  if (need > b->part_pipe_cap) {
    cudaFree(b->part_pipe);
    b->part_pipe = nullptr;
    b->part_pipe_cap = 0;
    BK(cudaMalloc(&b->part_pipe, 16ull * (size_t)need));
    b->part_pipe_cap = need;
  }
  b->bl_t = b->bl;
  b->bl_t.tlay = 1;
  drop_graphs(b);
  std::copy(want, want + 4, b->layout);
  return APFC_OK;
}

// ping-pong views of the Krylov vectors
struct Vecs {
  float2 *r[2], *p[2], *v[2], *rhat, *u, *t, *r32;
};
Vecs vecs(apfc_batch* b) {
  Vecs v;
  v.r[0] = b->blk[0];
  v.r[1] = b->blk[9];
  v.rhat = b->blk[1];
  v.p[0] = b->blk[2];
  v.p[1] = b->blk[7];
  v.v[0] = b->blk[3];
  v.v[1] = b->blk[8];
  v.u = b->blk[4];
  v.t = b->blk[5];
  v.r32 = b->blk[6];
  return v;
}

// `every` merged BiCGStab iterations over all runs, starting on side `cur`.
bool issue_block(apfc_batch* b, int cur, int every, int tile, int rows, int tile_t) {
  const Vecs x = vecs(b);
  const int m = b->opts.cheb_degree;
  cudaStream_t s = b->stream;
  for (int q = 0; q < every; ++q) {
    if (!launch_fused_merged_v<float>(m, rows, tile, b->coef, b->cw.data(), x.r[cur], x.v[cur], x.t, x.p[cur], x.u,
                                      x.r[1 - cur], x.p[1 - cur], x.v[1 - cur], x.rhat, b->rh16, b->ks, b->part_pipe, s,
                                      &b->bl))
      return false;
    launch_finalize_batch<float>(1, b->part_pipe, 0, b->bl, b->J, b->ks, OP_ALPHA, s);
    if (!launch_fused_merged_t<float>(m, rows, tile_t, b->coef, b->cw.data(), x.r[1 - cur], x.v[1 - cur], x.t,
                                      x.rhat, b->ks, b->part_pipe, s, &b->bl_t))
      return false;
    launch_finalize_batch<float>(5, b->part_pipe, 0, b->bl_t, b->J, b->ks, OP_OMEGA5, s);
    launch_final_update<float>(x.r[1 - cur], x.v[1 - cur], x.p[1 - cur], x.u, b->ks, b->coef, s, &b->bl);
    cur = 1 - cur;
  }
  return true;
}

// Start a BiCGStab solve of A P^{-1} u = r32 for every (run, amplitude); runs with
// skip[r] start converged.  fixed_tol >= 0: that relative tolerance for all; else the
// refinement's per-amplitude choice (inner_tol) from the outer residual norms.
// Leaves the scalars on the host; *any: some are active.
apfc_status krylov_init(apfc_batch* b, const std::vector<char>& skip, int max_iter, bool* any,
                        double fixed_tol = -1.0) {
  const Vecs x = vecs(b);
  cudaStream_t s = b->stream;
  const size_t bytes = sizeof(float2) * (size_t)b->elems;
  for (int r = 0; r < b->R; ++r)
    for (int j = 0; j < b->J; ++j) {
      KScal& k = b->ks_host[r * b->J + j];
      // r0 = b: a relative tolerance >= 1 stops at once; otherwise the run alone's choice
      const KScal& o = b->ks64_host[r * b->J + j];
      const double tj = skip[r]           ? 2.0
                        : fixed_tol >= 0.0 ? fixed_tol
                                           : inner_tol(b->opts.tol, b->opts.tol_inner, o.rnorm2, o.bnorm2);
      std::memset(&k, 0, sizeof(k));
      k.tolrel2 = tj * tj;
      k.max_iter = max_iter;
    }
  BK(cudaMemcpyAsync(b->ks, b->ks_host, sizeof(KScal) * b->R * b->J, cudaMemcpyHostToDevice, s));
  BK(cudaMemsetAsync(x.p[0], 0, bytes, s));
  BK(cudaMemsetAsync(x.v[0], 0, bytes, s));
  BK(cudaMemsetAsync(x.u, 0, bytes, s));
  BK(cudaMemsetAsync(x.t, 0, bytes, s));
  // r = r32 and the shadow residual rounded to bf16, as in a context alone: rho0 = (rhat, r0)
  launch_init32(x.r32, x.r[0], x.rhat, b->rh16, b->part_fix, b->coef, s, &b->bl);
  launch_finalize_batch<float>(3, b->part_fix, kDotBlocks, b->bl, b->J, b->ks, OP_INIT3, s);
  apfc_status st = sync_ks(b, b->ks, b->ks_host);
  if (st != APFC_OK) return st;
  *any = false;
  for (int i = 0; i < b->R * b->J; ++i) {
    if (b->ks_host[i].status == KS_NAN) return bfail(b, APFC_ENAN, "run " + std::to_string(i / b->J) + ": NaN/Inf");
    *any = *any || b->ks_host[i].active;
  }
  return APFC_OK;
}

// Iterate until every (run, amplitude) has stopped.
apfc_status krylov_iterate(apfc_batch* b, int max_iter, int tile, int rows, int tile_t) {
  const int every = std::max(1, b->opts.check_every);
  const bool graph = (b->flags & APFC_BATCH_GRAPH) && !profiler_on();
  int cur = 0;
  long long launched = 0, blocks = 0;
  while (true) {
    if (launched > (long long)max_iter + every) return bfail(b, APFC_ENOCONV, "Krylov iteration cap exceeded");
    launched += every;
    if (graph && blocks > 0) {
      // the first block ran eagerly (kernel attributes are set on first use)
      if (!b->gblock[cur]) {
        cudaGraph_t g = nullptr;
        BK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
        const bool ok = issue_block(b, cur, every, tile, rows, tile_t);
        const cudaError_t ec = cudaStreamEndCapture(b->stream, &g);
        if (!ok) {
          if (g) cudaGraphDestroy(g);
          return bfail(b, APFC_EINVAL, "fused pipeline cannot run these options");
        }
        BK(ec);
        const cudaError_t ei = cudaGraphInstantiate(&b->gblock[cur], g, 0);
        cudaGraphDestroy(g);
        BK(ei);
      }
      BK(cudaGraphLaunch(b->gblock[cur], b->stream));
      b->graph_replays += 1;
    } else if (!issue_block(b, cur, every, tile, rows, tile_t)) {
      return bfail(b, APFC_EINVAL, "fused pipeline cannot run these options");
    }
    ++blocks;
    if (every & 1) cur = 1 - cur;
    apfc_status st = sync_ks(b, b->ks, b->ks_host);
    if (st != APFC_OK) return st;
    bool run = false;
    for (int i = 0; i < b->R * b->J; ++i) run = run || b->ks_host[i].active;
    if (!run) return APFC_OK;
  }
}

// One step of every run by BiCGStab: FP32 solves inside FP64 iterative refinement.
apfc_status bicg_step(apfc_batch* b) {
  cudaStream_t s = b->stream;
  const int tile = b->opts.tile, rows = bicg_rows(b->opts), tile_t = tile_t_of(b->opts);
  const apfc_status sl = set_layout(b, tile, rows, tile_t);
  if (sl != APFC_OK) return sl;
  const Vecs x = vecs(b);
  double* part = reinterpret_cast<double*>(b->part_fix);
  bool resid_ready = false;
  if (b->have_prev && b->prev_dt == b->coef_dt && !b->prev_schur) {
    // r0 = b - b_prev + r_prev; the new RHS goes to the other buffer
    launch_rhs_resid(b->x64, b->b64_prev, b->b64, b->r64_blk, x.r32, part, b->coef, b->nt, false, s, &b->bl);
    std::swap(b->b64, b->b64_prev);
    resid_ready = true;
  } else {
    // the new RHS and ||b||^2 (the same kernel as a context alone), r0 by stencil below
    launch_rhs_resid(b->x64, b->b64, nullptr, nullptr, x.r32, part, b->coef, b->nt, false, s, &b->bl);
  }
  b->have_prev = false;
  const double tol2 = b->opts.tol * b->opts.tol;
  std::vector<char> done(b->R, 0);
  std::vector<int> solves(b->R, 0), iters(b->R, 0);
  int sweep = 0;
  for (;; ++sweep) {
    // the right-hand side's partial sums: ||b||^2 and, with a previous residual, ||r0||^2
    if (sweep == 0) launch_finalize_batch<double>(2, part, kDotBlocks, b->bl, b->J, b->ks64, OP_NORMS, s);
    if (!resid_ready) {
      launch_residual_refine2d(b->b64, b->x64, x.r32, b->r64_blk, part, b->coef, s, b->bl);
      launch_finalize_batch<double>(1, part, kDotBlocks, b->bl, b->J, b->ks64, OP_RNORM, s);
    }
    resid_ready = false;
    apfc_status st = sync_ks(b, b->ks64, b->ks64_host);
    if (st != APFC_OK) return st;
    bool all = true;
    for (int r = 0; r < b->R; ++r) {
      bool ok = true;
      for (int j = 0; j < b->J; ++j) {
        const KScal& k = b->ks64_host[r * b->J + j];
        if (!std::isfinite(k.rnorm2) || !std::isfinite(k.bnorm2))
          return bfail(b, APFC_ENAN, "run " + std::to_string(r) + ": residual norm is not finite");
        if (k.rnorm2 > tol2 * k.bnorm2) ok = false;
      }
      if (ok && !done[r]) done[r] = 1;
      all = all && done[r];
    }
    if (all) {
      // the last check of every run was a stencil residual of its final state
      b->have_prev = sweep > 0;
      b->prev_schur = false;
      b->prev_dt = b->coef_dt;
      break;
    }
    if (sweep >= b->opts.max_refine) {
      for (int r = 0; r < b->R; ++r)
        if (!done[r]) return bfail(b, APFC_ENOCONV, "run " + std::to_string(r) + ": refinement did not converge");
    }
    bool any = false;
    st = krylov_init(b, done, b->opts.max_iter, &any);
    if (st != APFC_OK) return st;
    if (any) {
      st = krylov_iterate(b, b->opts.max_iter, tile, rows, tile_t);
      if (st != APFC_OK) return st;
      // x += P^{-1} u (u = 0 for runs that did not iterate)
      if (!launch_fused_pinv_add<float>(b->opts.cheb_degree, rows, tile, b->coef, b->cw.data(), x.u, b->x64, s,
                                        &b->bl))
        return bfail(b, APFC_EINVAL, "fused pipeline cannot run these options");
    }
    for (int r = 0; r < b->R; ++r) {
      if (done[r]) continue;
      solves[r] += 1;
      int mx = 0;
      for (int j = 0; j < b->J; ++j) {
        const KScal& k = b->ks_host[r * b->J + j];
        if (k.status == KS_NAN) return bfail(b, APFC_ENAN, "run " + std::to_string(r) + ": NaN in the Krylov solve");
        mx = std::max(mx, k.iters);
      }
      iters[r] += mx;
    }
  }
  for (int r = 0; r < b->R; ++r) {
    apfc_stats_t& t = b->stats[r];
    t.steps += 1;
    t.iters_last = iters[r];
    t.iters_total += iters[r];
    t.refine_last = solves[r];
    double rr = 0.0;
    for (int j = 0; j < b->J; ++j) {
      const KScal& k = b->ks64_host[r * b->J + j];
      rr = std::max(rr, std::sqrt(k.rnorm2 / (k.bnorm2 > 0 ? k.bnorm2 : 1.0)));
    }
    t.resid_last = rr;
  }
  return APFC_OK;
}

// One step of every run: FP32 Chebyshev solves inside FP64 iterative refinement.
apfc_status batch_step(apfc_batch* b) {
  if (!b->schur_ok) return bicg_step(b);
  cudaStream_t s = b->stream;
  double* part = reinterpret_cast<double*>(b->part_fix);
  bool resid_ready = false;
  if (b->have_prev && b->prev_dt == b->coef_dt && b->prev_schur) {
    // r0 = b - b_prev + r_prev; the new RHS goes to the other buffer
    launch_rhs_resid(b->x64, b->b64_prev, b->b64, b->r64_prev, b->r[0], part, b->coef, b->nt, true, s, &b->bl);
    std::swap(b->b64, b->b64_prev);
    resid_ready = true;
  } else {
    // the new RHS and ||b||^2 (the same kernel as a context alone), r0 by stencil below
    launch_rhs_resid(b->x64, b->b64, nullptr, nullptr, b->r[0], part, b->coef, b->nt, true, s, &b->bl);
  }
  b->have_prev = false;
  SchurPlan plan = plan_of(b), prhs = plan;
  prhs.part = part;  // (value, 0) pairs [run][J][kDotSlots][kDotBlocks]
  prhs.npart = kDotBlocks;
  prhs.elem = 2;
  prhs.slot_stride = 2 * kDotBlocks;
  prhs.amp_stride = 2 * kDotSlots * kDotBlocks;
  prhs.have = resid_ready ? 3 : 2;
  plan.part = b->rpart;
  plan.elem = 1;
  plan.by_run = 1;
  plan.have = 1;
  const int ni = plan.ni;
  const double tol2 = b->opts.tol * b->opts.tol;
  std::vector<char> done(b->R, 0);
  std::vector<int> solves(b->R, 0), iters(b->R, 0);
  int sweep = 0;
  for (;; ++sweep) {
    if (sweep == 0) launch_schur_plan(prhs, b->ks64, s, &b->bl);
    if (!resid_ready) {
      launch_resid_schur2d<float>(b->b64, b->x64, b->r[0], b->r64_prev, b->rpart, b->coef, false, schur_resid_f64(b->schur, b->opts.tol), s, &b->bl);
      launch_schur_plan(plan, b->ks64, s, &b->bl);
    }
    resid_ready = false;
    apfc_status st = sync_ks(b, b->ks64, b->ks64_host);
    if (st != APFC_OK) return st;
    bool all = true, patch = false;
    int np = 0;
    for (int r = 0; r < b->R; ++r) {
      bool ok = true;
      int most = 0;
      for (int j = 0; j < b->J; ++j) {
        const KScal& k = b->ks64_host[r * b->J + j];
        if (!std::isfinite(k.rnorm2) || !std::isfinite(k.bnorm2))
          return bfail(b, APFC_ENAN, "run " + std::to_string(r) + ": residual norm is not finite");
        if (k.rnorm2 > tol2 * k.bnorm2) ok = false;
        most = std::max(most, k.iters);
      }
      if (done[r] && most > 0) {
        // converged by the pointwise residual of the first check: it waits unchanged, as alone
        for (int j = 0; j < b->J; ++j) b->ks64_host[r * b->J + j].iters = 0;
        patch = true;
        most = 0;
      }
      if (ok) done[r] = 1;
      all = all && done[r];
      if (!done[r]) {
        solves[r] += 1;
        if (most > 0) iters[r] += (plan.t0 + ni * most + 1) / 2;
      }
      np = std::max(np, most);
    }
    if (all) {
      // the last check of every run was a stencil residual of its final state
      b->have_prev = sweep > 0;
      b->prev_schur = true;
      b->prev_dt = b->coef_dt;
      break;
    }
    if (sweep >= b->opts.max_refine) {
      for (int r = 0; r < b->R; ++r)
        if (!done[r]) return bfail(b, APFC_ENOCONV, "run " + std::to_string(r) + ": refinement did not converge");
    }
    if (patch) BK(cudaMemcpyAsync(b->ks64, b->ks64_host, sizeof(KScal) * b->R * b->J, cudaMemcpyHostToDevice, s));
    if (np > 0 && (st = solve(b, np)) != APFC_OK) return st;
  }
  for (int r = 0; r < b->R; ++r) {
    apfc_stats_t& t = b->stats[r];
    t.steps += 1;
    t.iters_last = iters[r];
    t.iters_total += iters[r];
    t.refine_last = solves[r];
    double rr = 0.0;
    for (int j = 0; j < b->J; ++j) {
      const KScal& k = b->ks64_host[r * b->J + j];
      rr = std::max(rr, std::sqrt(k.rnorm2 / (k.bnorm2 > 0 ? k.bnorm2 : 1.0)));
    }
    t.resid_last = rr;
  }
  return APFC_OK;
}

// The autotuner for BiCGStab: merged iterations on the first refinement residual of a step, for every
// tile variant and height of both kernels, then for every variant of the t-kernel alone.
apfc_status bicg_tune(apfc_batch* b, int* tile_out, int* rows_out, double* ms_out) {
  apfc_status st = alloc_bicg(b);
  if (st != APFC_OK) return st;
  cudaStream_t s = b->stream;
  const Vecs x = vecs(b);
  double* part = reinterpret_cast<double*>(b->part_fix);
  launch_rhs(b->x64, b->b64, b->coef, b->nt, s, &b->bl);
  launch_residual_refine2d(b->b64, b->x64, x.r32, nullptr, part, b->coef, s, b->bl);
  b->have_prev = false;
  cudaEvent_t e0, e1;
  BK(cudaEventCreate(&e0));
  BK(cudaEventCreate(&e1));
  int best_tile = b->opts.tile, best_rows = bicg_rows(b->opts), best_t = tile_t_of(b->opts);
  double best = 1e300;
  const std::vector<char> none(b->R, 0);
  auto time_candidate = [&](int tile, int rows, int tile_t, double* ms) -> apfc_status {
    apfc_status s2 = set_layout(b, tile, rows, tile_t);
    if (s2 != APFC_OK) return s2;
    for (int rep = 0; rep < 2; ++rep) {  // the first pass warms up
      bool any = false;
      // a tolerance that no solve reaches within kTunePasses iterations
      if ((s2 = krylov_init(b, none, 1 << 20, &any, 1e-30)) != APFC_OK) return s2;
      BK(cudaEventRecord(e0, s));
      if (!issue_block(b, 0, kTunePasses, tile, rows, tile_t))
        return bfail(b, APFC_EINVAL, "fused pipeline cannot run these options");
      BK(cudaEventRecord(e1, s));
      BK(cudaEventSynchronize(e1));
      float f = 0.f;
      BK(cudaEventElapsedTime(&f, e0, e1));
      *ms = f;
    }
    return APFC_OK;
  };
  double ms = 1e300;
  for (int tile = 0; tile < fused2d_tiles() && st == APFC_OK; ++tile)
    for (int rows : kTuneRows) {
      if ((st = time_candidate(tile, rows, tile, &ms)) != APFC_OK) break;
      if (ms < best) best = ms, best_tile = tile, best_rows = rows, best_t = tile;
    }
  for (int tile_t = 0; tile_t < fused2d_tiles() && st == APFC_OK; ++tile_t) {
    if (tile_t == best_t) continue;
    if ((st = time_candidate(best_tile, best_rows, tile_t, &ms)) == APFC_OK && ms < best) best = ms, best_t = tile_t;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != APFC_OK) return st;
  b->opts.tile = best_tile;
  b->opts.tile_rows = best_rows;
  b->opts.tile_t = best_t;
  if (tile_out) *tile_out = best_tile;
  if (rows_out) *rows_out = best_rows;
  if (ms_out) *ms_out = best / kTunePasses;
  return APFC_OK;
}

bool valid_batch_opts(const apfc_opts& o, std::string& e) {
  if (!valid_opts(o, e)) return false;
  if (o.precision != APFC_FP32_REFINED) e = "batched runs use precision APFC_FP32_REFINED";
  else if (o.fused != 1) e = "batched runs use the fused pipeline (fused = 1)";
  else if (o.picard_iters != 1 || o.jacobian != 0) e = "batched runs take the explicit step (picard_iters 1, jacobian 0)";
  else if (o.guess != APFC_GUESS_PREV) e = "batched runs start each solve from the previous state (guess 0)";
  else if (o.cheb_degree < 1 || o.cheb_degree > fused2d_max_degree((int)sizeof(float2))) e = "cheb_degree";
  else return true;
  return false;
}

void free_batch(apfc_batch* b) {
  if (b->stream) cudaStreamSynchronize(b->stream);
  drop_graphs(b);
  cudaFree(b->rg_dev);
  cudaFree(b->x64);
  cudaFree(b->b64);
  cudaFree(b->b64_prev);
  cudaFree(b->r64_prev);
  for (auto& p : b->r) cudaFree(p);
  for (auto& p : b->d) cudaFree(p);
  cudaFree(b->u);
  cudaFree(b->tab);
  for (auto& p : b->blk) cudaFree(p);
  cudaFree(b->rh16);
  cudaFree(b->r64_blk);
  cudaFree(b->part_pipe);
  cudaFree(b->ks);
  if (b->ks_host) cudaFreeHost(b->ks_host);
  cudaFree(b->rpart);
  cudaFree(b->part_fix);
  cudaFree(b->ks64);
  cudaFree(b->epart);
  cudaFree(b->eout);
  if (b->ks64_host) cudaFreeHost(b->ks64_host);
  if (b->eout_host) cudaFreeHost(b->eout_host);
  if (b->own_stream) cudaStreamDestroy(b->stream);
  delete b;
}

apfc_status check_run(apfc_batch* b, int run) {
  if (run < 0 || run >= b->R) return bfail(b, APFC_EINVAL, "run index out of range");
  return APFC_OK;
}

}  // namespace

// Why the last apfc_batch_init of this thread failed (apfc_batch_last_error(NULL)).
static thread_local std::string g_batch_init_err;

static apfc_status bfail(apfc_status s, const std::string& msg) {
  g_batch_init_err = msg;
  return s;
}

extern "C" {

apfc_status apfc_batch_init(apfc_batch** out, const apfc_lattice* lat, const apfc_params* p, int nruns, const int* nx,
                            const int* ny, double hx, double hy, const apfc_opts* opts, int flags, void* stream) {
  g_batch_init_err.clear();
  if (!out || !lat || !p || !nx || !ny) return bfail(APFC_EINVAL, "null argument");
  *out = nullptr;
  if (!valid_problem(*lat, *p) || lat->dim != 2) return bfail(APFC_EINVAL, "invalid lattice or parameters (batches are 2D)");
  if (nruns < 1 || nruns > kMaxRuns) return bfail(APFC_EINVAL, "run count out of range");
  if (!(hx > 0.0) || !(hy > 0.0) || !std::isfinite(hx) || !std::isfinite(hy))
    return bfail(APFC_EINVAL, "spacings must be positive and finite");
  if (flags & ~APFC_BATCH_GRAPH) return bfail(APFC_EINVAL, "unknown flags");
  long long total = 0;
  int mx = 0, my = 0;
  for (int r = 0; r < nruns; ++r) {
    if (nx[r] < 3 || ny[r] < 3 || nx[r] > (1 << 20) || ny[r] > (1 << 20))
      return bfail(APFC_EINVAL, "run " + std::to_string(r) + ": grid sizes must be in [3, 2^20]");
    total += (long long)nx[r] * ny[r];
    mx = std::max(mx, nx[r]);
    my = std::max(my, ny[r]);
  }
  apfc_opts o;
  apfc_default_opts(&o);
  o.precision = APFC_FP32_REFINED;
  if (opts) o = *opts;
  std::string e;
  if (!valid_batch_opts(o, e)) return bfail(APFC_EINVAL, "invalid option: " + e);
  if (total * 2LL * lat->J > (1LL << 40)) return bfail(APFC_ETOOBIG, "too many points in the batch");
  {
    int ndev = 0;
    const cudaError_t ce = cudaGetDeviceCount(&ndev);
    if (ce != cudaSuccess || ndev == 0)
      return bfail(APFC_ECUDA, std::string("no CUDA device: ") +
                                   (ce != cudaSuccess ? cudaGetErrorString(ce) : "device count 0"));
  }

  apfc_batch* b = new (std::nothrow) apfc_batch();
  if (!b) return bfail(APFC_ENOMEM, "host allocation of the batch failed");
  b->lat = *lat;
  b->par = *p;
  b->opts = o;
  b->R = nruns;
  b->J = lat->J;
  b->flags = flags;
  b->nx.assign(nx, nx + nruns);
  b->ny.assign(ny, ny + nruns);
  b->gmax.n[0] = mx;
  b->gmax.n[1] = my;
  b->gmax.n[2] = 1;
  b->gmax.h[0] = hx;
  b->gmax.h[1] = hy;
  b->gmax.h[2] = 1.0;
  {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0)
      b->sms = sms;
  }
  b->has_state.assign(nruns, 0);
  b->stats.assign(nruns, apfc_stats_t{});
  auto cleanup = [&](apfc_status s) {
    if (g_batch_init_err.empty())
      g_batch_init_err = s == APFC_ENOMEM ? "device allocation failed"
                         : s == APFC_ECUDA   ? std::string("CUDA call failed: ") + cudaGetErrorString(cudaGetLastError())
                         : s == APFC_ETOOBIG ? "the batch exceeds the partial-sum table of the fused kernels"
                                             : "invalid batch";
    free_batch(b);
    return s;
  };
  if (!build_tables(*lat, *p, b->nt, b->et, e)) {
    g_batch_init_err = "nonlinear-term table: " + e;
    return cleanup(APFC_EINVAL);
  }
  b->stream = static_cast<cudaStream_t>(stream);
  if ((flags & APFC_BATCH_GRAPH) && b->stream == nullptr) {
    // graph capture needs a stream other than the legacy default one
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) return cleanup(APFC_ECUDA);
    b->own_stream = true;
  }
  if (!make_table(b)) return cleanup(APFC_ETOOBIG);
  const RunGeom& lastg = b->rg.back();
  const size_t blk64 = sizeof(double2) * (size_t)b->elems, fld32 = sizeof(float2) * (size_t)b->felems;
  const size_t nks = sizeof(KScal) * (size_t)nruns * b->J;
  if (cudaMalloc(&b->rg_dev, sizeof(RunGeom) * nruns) != cudaSuccess) return cleanup(APFC_ENOMEM);
  for (double2** q : {&b->x64, &b->b64, &b->b64_prev})
    if (cudaMalloc(q, blk64) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->r64_prev, sizeof(double2) * (size_t)b->felems) != cudaSuccess) return cleanup(APFC_ENOMEM);
  for (float2** q : {&b->r[0], &b->r[1], &b->d[0], &b->d[1], &b->u})
    if (cudaMalloc(q, fld32) != cudaSuccess) return cleanup(APFC_ENOMEM);
  const int tx = mx + 1, ty = my + 1;
  if (cudaMalloc(&b->tab, sizeof(float2) * b->J * (size_t)(tx + ty)) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->rpart, sizeof(double) * (size_t)(lastg.part_off_r + 2LL * b->J * lastg.npart_r)) != cudaSuccess)
    return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->part_fix, 16ull * kDotSlots * kDotBlocks * (size_t)nruns * b->J) != cudaSuccess)
    return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->ks64, nks) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMallocHost(&b->ks64_host, nks) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->epart, sizeof(double) * kDotBlocks) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMalloc(&b->eout, sizeof(double)) != cudaSuccess) return cleanup(APFC_ENOMEM);
  if (cudaMallocHost(&b->eout_host, sizeof(double)) != cudaSuccess) return cleanup(APFC_ENOMEM);
  std::memset(b->ks64_host, 0, nks);
  // the zeta-parts of the right-hand sides stay zero
  if (cudaMemsetAsync(b->x64, 0, blk64, b->stream) != cudaSuccess) return cleanup(APFC_ECUDA);
  if (cudaMemsetAsync(b->b64, 0, blk64, b->stream) != cudaSuccess) return cleanup(APFC_ECUDA);
  if (cudaMemsetAsync(b->b64_prev, 0, blk64, b->stream) != cudaSuccess) return cleanup(APFC_ECUDA);
  if (cudaMemsetAsync(b->ks64, 0, nks, b->stream) != cudaSuccess) return cleanup(APFC_ECUDA);
  if (cudaMemcpyAsync(b->rg_dev, b->rg.data(), sizeof(RunGeom) * nruns, cudaMemcpyHostToDevice, b->stream) !=
      cudaSuccess)
    return cleanup(APFC_ECUDA);
  b->bl.dev = b->rg_dev;
  b->bl.host = b->rg.data();
  b->bl.R = nruns;
  if (!set_coef(b, 1.0, e)) return cleanup(APFC_EINVAL);
  launch_gauge_table<float>(b->tab, b->coef, tx, ty, 0, b->stream);
  if (cudaStreamSynchronize(b->stream) != cudaSuccess) return cleanup(APFC_ECUDA);
  *out = b;
  return APFC_OK;
}

apfc_status apfc_batch_set_opts(apfc_batch* b, const apfc_opts* opts) {
  if (!b || !opts) return APFC_EINVAL;
  std::string e;
  if (!valid_batch_opts(*opts, e)) return bfail(b, APFC_EINVAL, e);
  b->opts = *opts;
  const double dt = b->coef_dt;
  b->coef_dt = -1.0;  // tau_mode or the degree may have changed
  if (!set_coef(b, dt > 0 ? dt : 1.0, e)) return bfail(b, APFC_EINVAL, e);
  drop_graphs(b);
  b->have_prev = false;
  return APFC_OK;
}

apfc_status apfc_batch_set_amplitudes(apfc_batch* b, int run, const void* eta, int where) {
  if (!b || !eta || (where != APFC_HOST && where != APFC_DEVICE)) return APFC_EINVAL;
  apfc_status st = check_run(b, run);
  if (st != APFC_OK) return st;
  const RunGeom& g = b->rg[run];
  const size_t row = sizeof(double2) * (size_t)g.pts;
  const cudaMemcpyKind k = where == APFC_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  BK(cudaMemcpy2DAsync(b->x64 + g.elem_off + g.pts, 2 * row, eta, row, row, b->J, k, b->stream));
  launch_zeta(b->x64 + g.elem_off, run_coef(b, run), b->stream);
  BK(cudaGetLastError());
  BK(cudaStreamSynchronize(b->stream));
  b->has_state[run] = 1;
  b->have_prev = false;
  b->failed = false;  // as on a context: new amplitudes clear a sticky error
  b->err.clear();
  b->stats[run] = apfc_stats_t{};
  return APFC_OK;
}

apfc_status apfc_batch_get_amplitudes(apfc_batch* b, int run, void* eta, int where) {
  if (!b || !eta || (where != APFC_HOST && where != APFC_DEVICE)) return APFC_EINVAL;
  apfc_status st = check_run(b, run);
  if (st != APFC_OK) return st;
  if (!b->has_state[run]) return bfail(b, APFC_ESTATE, "no amplitudes set for this run");
  const RunGeom& g = b->rg[run];
  const size_t row = sizeof(double2) * (size_t)g.pts;
  const cudaMemcpyKind k = where == APFC_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  BK(cudaMemcpy2DAsync(eta, row, b->x64 + g.elem_off + g.pts, 2 * row, row, b->J, k, b->stream));
  BK(cudaStreamSynchronize(b->stream));
  return APFC_OK;
}

apfc_status apfc_batch_step(apfc_batch* b, double dt, int n) {
  if (!b || n < 0) return APFC_EINVAL;
  if (b->failed) return APFC_ESTATE;
  for (int r = 0; r < b->R; ++r)
    if (!b->has_state[r]) return bfail(b, APFC_ESTATE, "no amplitudes set for run " + std::to_string(r));
  std::string e;
  if (!set_coef(b, dt, e)) return bfail(b, APFC_EINVAL, e);
  for (int i = 0; i < n; ++i) {
    apfc_status st = batch_step(b);
    if (st != APFC_OK) return st;
  }
  return APFC_OK;
}

apfc_status apfc_batch_energy(apfc_batch* b, int run, double* F) {
  if (!b || !F) return APFC_EINVAL;
  apfc_status st = check_run(b, run);
  if (st != APFC_OK) return st;
  if (!b->has_state[run]) return bfail(b, APFC_ESTATE, "no amplitudes set for this run");
  launch_energy(b->x64 + b->rg[run].elem_off, b->epart, b->eout, run_coef(b, run), b->et, b->par.Bx, b->stream);
  BK(cudaGetLastError());
  BK(cudaMemcpyAsync(b->eout_host, b->eout, sizeof(double), cudaMemcpyDeviceToHost, b->stream));
  BK(cudaStreamSynchronize(b->stream));
  *F = b->gmax.h[0] * b->gmax.h[1] * b->eout_host[0];
  return APFC_OK;
}

apfc_status apfc_batch_stats(const apfc_batch* b, int run, apfc_stats_t* out) {
  if (!b || !out || run < 0 || run >= b->R) return APFC_EINVAL;
  *out = b->stats[run];
  return APFC_OK;
}

apfc_status apfc_batch_autotune(apfc_batch* b, double dt, int* tile_out, int* rows_out, double* ms_out) {
  if (!b) return APFC_EINVAL;
  if (b->failed) return APFC_ESTATE;
  for (int r = 0; r < b->R; ++r)
    if (!b->has_state[r]) return bfail(b, APFC_ESTATE, "no amplitudes set for run " + std::to_string(r));
  std::string e;
  if (!set_coef(b, dt, e)) return bfail(b, APFC_EINVAL, e);
  if (!b->schur_ok) return bicg_tune(b, tile_out, rows_out, ms_out);
  cudaStream_t s = b->stream;
  // the first refinement residual of a step from the current state is the right-hand side
  // every candidate iterates on; u is never added to the state (the passes stop before the
  // last of the ks64[].iters set here)
  launch_rhs(b->x64, b->b64, b->coef, b->nt, s, &b->bl);
  launch_resid_schur2d<float>(b->b64, b->x64, b->r[0], nullptr, b->rpart, b->coef, false, schur_resid_f64(b->schur, b->opts.tol), s, &b->bl);
  b->have_prev = false;
  std::memset(b->ks64_host, 0, sizeof(KScal) * b->R * b->J);
  for (int i = 0; i < b->R * b->J; ++i) b->ks64_host[i].iters = kTunePasses + 1;
  BK(cudaMemcpyAsync(b->ks64, b->ks64_host, sizeof(KScal) * b->R * b->J, cudaMemcpyHostToDevice, s));
  cudaEvent_t e0, e1;
  BK(cudaEventCreate(&e0));
  BK(cudaEventCreate(&e1));
  int best_tile = b->opts.tile, best_rows = rows_of(b);
  double best = 1e300;
  apfc_status st = APFC_OK;
  auto time_candidate = [&](int tile, int rows, double* ms) -> apfc_status {
    for (int rep = 0; rep < 2; ++rep) {  // the first pass warms up
      BK(cudaEventRecord(e0, s));
      if (!issue_passes(b, kTunePasses, tile, rows))
        return bfail(b, APFC_ECUDA, "the Chebyshev passes cannot be launched");
      BK(cudaEventRecord(e1, s));
      BK(cudaEventSynchronize(e1));
      float f = 0.f;
      BK(cudaEventElapsedTime(&f, e0, e1));
      *ms = f;
    }
    return APFC_OK;
  };
  for (int tile : {3, 5})  // narrow and wide strips
    for (int rows : kTuneRows) {
      if (st != APFC_OK) break;
      double ms = 1e300;
      if ((st = time_candidate(tile, rows, &ms)) != APFC_OK) break;
      if (ms < best) best = ms, best_tile = tile, best_rows = rows;
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != APFC_OK) return st;
  b->opts.tile = best_tile;
  b->opts.tile_rows = best_rows;
  if (b->opts.tile_t < 0) b->opts.tile_t = best_tile;
  drop_graphs(b);
  if (tile_out) *tile_out = best_tile;
  if (rows_out) *rows_out = best_rows;
  if (ms_out) *ms_out = best / kTunePasses;
  return APFC_OK;
}

apfc_status apfc_batch_get_opts(const apfc_batch* b, apfc_opts* out) {
  if (!b || !out) return APFC_EINVAL;
  *out = b->opts;
  return APFC_OK;
}

long long apfc_batch_graph_replays(const apfc_batch* b) { return b ? b->graph_replays : -1; }

const char* apfc_batch_last_error(const apfc_batch* b) {
  if (b) return b->err.c_str();
  return g_batch_init_err.empty() ? "null batch" : g_batch_init_err.c_str();
}

void apfc_batch_destroy(apfc_batch* b) {
  if (b) free_batch(b);
}

apfc_status apfc_batch_profile_start(apfc_batch* b, int timed_id) {
  if (!b) return APFC_EINVAL;
  std::string e;
  if (!profiler_start(b->stream, timed_id, &b->coef.prof, e)) return bfail(b, APFC_EINVAL, e);
  return APFC_OK;
}

apfc_status apfc_batch_profile_read(apfc_batch* b, int id, double* ms, long long* launches, double* bytes,
                                    long long* all_launches) {
  if (!b) return APFC_EINVAL;
  std::string e;
  if (!profiler_read(b->stream, id, ms, launches, bytes, all_launches, e)) return bfail(b, APFC_EINVAL, e);
  return APFC_OK;
}

apfc_status apfc_batch_profile_stop(apfc_batch* b) {
  if (!b) return APFC_EINVAL;
  profiler_stop();
  b->coef.prof = nullptr;
  return APFC_OK;
}

}  // extern "C"
