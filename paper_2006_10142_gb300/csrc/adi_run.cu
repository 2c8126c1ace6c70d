// adi_run.cu -- handle implementation: creation, the time loop (Algorithm 1)
// as chained launches or replayed step pairs, checkpoints, state access,
// status, tuning and measurement hooks.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "adi_adjoint.h"
#include "adi_internal.h"
#include "adi_run.h"

using namespace adi;

namespace {

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Kernel attributes (dynamic shared memory, cluster sizes) are per device:
// one flag per device, set under a lock.
constexpr int kMaxDevices = 64;
bool g_configured[kMaxDevices] = {};
std::mutex g_config_mu;

bool stream_captures(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return cs != cudaStreamCaptureStatusNone;
}

#define CK(call, what)                                          \
  do {                                                          \
    cudaError_t e_ = (call);                                    \
    if (e_ != cudaSuccess) return cuda_fail(this, e_, what);    \
  } while (0)

}  // namespace

cudaError_t adi::configure_current_device() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_config_mu);
  if (g_configured[dev]) return cudaSuccess;
  e = configure_kernels();
  if (e == cudaSuccess) e = configure_adjoint_kernels();
  if (e == cudaSuccess) e = configure_y_coop_kernels();
  if (e == cudaSuccess) e = configure_model_kernels();
  if (e == cudaSuccess) e = configure_tile_kernels();
  if (e == cudaSuccess) e = configure_patch_kernels();
  if (e == cudaSuccess) g_configured[dev] = true;
  return e;
}

// The grid's and plan's part of the one-pass step's arguments.
TileArgs adi::tile_args(const Grid& G) {
  TileArgs a = {};
  a.nx = G.nx;
  a.ny = G.ny;
  a.ld = G.ld;
  a.band_rows = G.plan.tile_rows;
  a.small = G.plan.small_patch ? 1 : 0;
  a.cx = (float)(G.dt * G.dt / (G.hx * G.hx));
  a.cy = (float)(G.dt * G.dt / (G.hy * G.hy));
  a.scx = (float)(G.dt * G.dt / (2.0 * G.hx * G.hx));
  a.scy = (float)(G.dt * G.dt / (2.0 * G.hy * G.hy));
  a.src_scale = (float)(G.dt * G.dt / (G.hx * G.hy));
  return a;
}

// Scratch of the y sweep without clusters (y_stage 4): segment summaries for
// up to 32 segments per column and two counters per strip, zeroed once.
int adi_wave::ensure_ycoop(Grid& G) {
  if (G.plan.y_stage != ADI_STAGE_COOP) return ADI_OK;
  const int cols = (G.nx + 31) / 32 * 32;
  const int strips = (G.nx + 15) / 16;
  G.yc.C = G.plan.C;
  if (G.yc.tops != nullptr && G.yc.cols >= cols && G.yc.strips >= strips) return ADI_OK;
  cudaFree(G.yc.tops);
  cudaFree(G.yc.sync);
  G.yc.tops = nullptr;
  G.yc.sync = nullptr;
  G.yc.cols = 0;
  G.yc.strips = 0;
  cudaError_t e = cudaMalloc(&G.yc.tops, sizeof(float) * 8 * 32 * (size_t)cols);
  if (e == cudaSuccess) e = cudaMalloc(&G.yc.sync, sizeof(int) * 2 * (size_t)strips);
  if (e == cudaSuccess) e = cudaMemset(G.yc.sync, 0, sizeof(int) * 2 * (size_t)strips);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaFree(G.yc.tops);
    cudaFree(G.yc.sync);
    G.yc.tops = nullptr;
    G.yc.sync = nullptr;
    return fail(this, e == cudaErrorMemoryAllocation ? ADI_ENOMEM : ADI_ECUDA,
                std::string("y sweep scratch: ") + cudaGetErrorString(e));
  }
  G.yc.cols = cols;
  G.yc.strips = strips;
  return ADI_OK;
}

// The grid record goes to the device as a kernel argument: no copy engine
// and no host buffer that must outlive the call.
int adi_wave::upload_gd(Grid& G, cudaStream_t st) {
  G.hgd.kf[0] = G.hgd.k;
  G.hgd.kf[1] = G.hgd.k;
  CK(launch_put_gd(&G.gd, &G.hgd, 1, st), "upload grid state");
  launches += 1;
  return ADI_OK;
}

int adi_wave::create(const adi_wave_desc* desc, int n, const float* const* m,
                     const float* const* phi, const float* const* psi, const adi_source* src,
                     cudaStream_t st) {
  CK(configure_current_device(), "configure kernels");
  CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "create capture stream");
  CK(cudaMalloc(&d_err, 4 * sizeof(int)), "alloc error word and scan");
  scan = reinterpret_cast<unsigned int*>(d_err) + 1;
  CK(cudaMemsetAsync(d_err, 0, sizeof(int), st), "clear error word");
  g.resize(n);
  for (int s = 0; s < n; ++s) {
    Grid& G = g[s];
    const adi_wave_desc& d = desc[s];
    G.nx = d.nx;
    G.ny = d.ny;
    G.ld = round_up(d.nx, 32);
    G.lx = d.lx;
    G.ly = d.ly;
    G.dt = d.dt;
    G.hx = d.lx / (d.nx + 1);
    G.hy = d.ly / (d.ny + 1);
    G.start = d.start;
    G.fp64mode = d.fp64_solve;
    // One allocation and one clear for a grid: an allocation and its release
    // cost the host some 60 us together, whatever the size, which counts
    // where a handle lives for a few dozen steps (301^2, 60 steps through
    // autograd: 2.78 -> 2.51 ms with the checkpoints' and the
    // reverse sweep's allocations merged likewise).
    const size_t field = (sizeof(float) * (size_t)G.ld * G.ny + 255) / 256 * 256;
    cudaError_t e = cudaMalloc(&G.mem, 4 * field + sizeof(GridDev));
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(this, e == cudaErrorMemoryAllocation ? ADI_ENOMEM : ADI_ECUDA,
                  std::string("allocate grid: ") + cudaGetErrorString(e));
    }
    G.m = reinterpret_cast<float*>(G.mem);
    G.buf[0] = reinterpret_cast<float*>(G.mem + field);
    G.buf[1] = reinterpret_cast<float*>(G.mem + 2 * field);
    G.w = reinterpret_cast<float*>(G.mem + 3 * field);
    G.gd = reinterpret_cast<GridDev*>(G.mem + 4 * field);
    CK(cudaMemsetAsync(G.mem, 0, 4 * field, st), "clear fields");
    int rc = start_grid(s, m[s], phi[s], psi ? psi[s] : nullptr, src ? &src[s] : nullptr, st);
    if (rc != ADI_OK) return rc;
  }
  if (n == 1) return ADI_OK;
  const int rc = setup_batch(st);
  return rc == ADI_OK ? ensure_batch_tiles() : rc;
}

// Two steps of every shot (rest: of those the one-launch step leaves) as a
// graph, from the present orientation.
int adi_wave::capture_batch_pair(cudaGraphExec_t* ex, bool rest) {
  std::vector<int> cur0;
  std::vector<long long> k0;
  std::vector<char> init0;
  for (Grid& G : g) {
    cur0.push_back(G.cur);
    k0.push_back(G.k);
    init0.push_back(G.from_init);
  }
  const int64_t l0 = launches;
  CK(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "begin capture");
  int rc = ADI_OK;
  if (batch_mode == 2) {
    rc = enqueue_batch_steps_parallel(2, cap, rest);  // per-shot chains of two steps
  } else {
    rc = enqueue_batch_step(cap);
    if (rc == ADI_OK) rc = enqueue_batch_step(cap);
  }
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(cap, &graph);
  for (size_t s = 0; s < g.size(); ++s) {
    g[s].cur = cur0[s];
    g[s].k = k0[s];
    g[s].from_init = init0[s];
  }
  pair_launches = launches - l0;
  launches = l0;
  if (rc != ADI_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(this, e, "end capture");
  e = cudaGraphInstantiate(ex, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    *ex = nullptr;
    return cuda_fail(this, e, "graph instantiate");
  }
  return ADI_OK;
}

// Batched run: every shot advances `steps` steps, by the form of the batch
// mode (one launch per step for all shots where their plans allow it, the
// persistent kernel, or the plain kernels per shot); step pairs of the latter
// two are replayed from a captured graph.
int adi_wave::run_batch(int steps, const adi_source* src, cudaStream_t st) {
  for (size_t s = 0; s < g.size(); ++s) {
    Grid& G = g[s];
    const adi_source none = {-1, -1, nullptr, 0};
    const adi_source sr = src ? src[s] : none;
    const bool on = sr.ix >= 0 && sr.wavelet != nullptr;
    G.hgd.k = G.k;
    G.hgd.k0 = G.k;
    G.hgd.steps = steps;
    G.hgd.wavelet = on ? sr.wavelet : nullptr;
    G.hgd.n_wavelet = on ? sr.n_wavelet : 0;
    G.hgd.src_ix = on ? sr.ix : -1;
    G.hgd.src_iy = on ? sr.iy : -1;
    G.hgd.n_rec = 0;
    G.hgd.rec = nullptr;
    G.hgd.traces = nullptr;
    G.hgd.kf[0] = G.hgd.kf[1] = G.k;
  }
  {
    std::vector<GridDev*> dst;
    std::vector<GridDev> v;
    for (Grid& G : g) {
      dst.push_back(G.gd);
      v.push_back(G.hgd);
    }
    CK(launch_put_gd(dst.data(), v.data(), (int)g.size(), st), "upload grid states");
    launches += ((int)g.size() + 31) / 32;
  }
  rr.valid = false;
  bool aligned = true;  // a reset that failed half way leaves shots in two orientations
  for (const Grid& G : g) aligned = aligned && G.cur == g[0].cur;
  if (batch_mode == 2 && aligned) {
    const int rc = ensure_batch_tiles();
    if (rc != ADI_OK) return rc;
    if (bt_n > 0) return run_batch_tiles(steps, st);
  }
  bool use_graph = g[0].plan.graph && !profile;
  // Sweeps shot after shot fill the GPU one by one: as launches they overlap a
  // little better than in a graph (us per step at tau = 2h: fifteen shots of 64^2
  // to 1500 x 200 180 and 190, four of 2048^2 153.6 and 155.3).
  if (batch_mode == 1 && tuning.use_graph == 0)
    for (const Grid& G : g) use_graph = use_graph && G.plan.tile != 0;
  int t = 0;
  if (use_graph) {
    while (steps - t >= 2) {
      cudaGraphExec_t& ex = pair[g[0].cur][0];
      if (!ex) {
        const int rc = capture_batch_pair(&ex, false);
        if (rc != ADI_OK) return rc;
      }
      CK(cudaGraphLaunch(ex, st), "graph launch");
      launches += pair_launches;
      for (Grid& G : g) { G.k += 2; G.from_init = false; }
      t += 2;
    }
  }
  while (t < steps) {
    int rc = enqueue_batch_step(st);
    if (rc != ADI_OK) return rc;
    t += 1;
  }
  return ADI_OK;
}

// Copy m (optional), re-plan, and run the start-up of Eq. (CN2) for shot s.
int adi_wave::start_grid(int s, const float* m, const float* phi, const float* psi,
                         const adi_source* sr, cudaStream_t st) {
  Grid& G = g[s];
  if (m) {
    // the caller's medium is scanned before it replaces the handle's, so a
    // rejected one leaves the handle as it was
    if (!scan_host) {
      unsigned int* hp = nullptr;
      CK(cudaHostAlloc((void**)&hp, 4 * sizeof(unsigned int), cudaHostAllocMapped), "alloc scan result");
      scan_host = hp;
      CK(cudaHostGetDevicePointer((void**)&scan_host_dev, hp, 0), "map scan result");
    }
    CK(launch_scan_m(m, G.nx, G.ny, G.nx, scan, scan_host_dev, st), "scan m");
    CK(cudaStreamSynchronize(st), "scan sync");
    unsigned int res3[3] = {scan_host[0], scan_host[1], scan_host[2]};
    launches += 3;
    if (res3[2]) return fail(this, ADI_EINVAL, "m must be finite and > 0 everywhere");
    CopyArgs c = {};
    c.nx = G.nx;
    c.ny = G.ny;
    c.spitch = G.nx;
    c.dpitch = G.ld;
    c.src0 = m;
    c.dst0 = G.m;
    CK(launch_copy_fields(c, GridDev{}, st), "copy m");
    launches += 1;
    float lo, hi;
    memcpy(&lo, &res3[0], 4);
    memcpy(&hi, &res3[1], 4);
    G.mmin = lo;
    G.mmax = hi;
    std::string why;
    GridPlan old = G.plan;
    int rc = plan_grid(G, tuning, why);
    if (rc != ADI_OK) {
      G.plan = old;
      return fail(this, rc, why);
    }
    // the captured steps stay valid while the plan (launch shapes, kernels) is the same
    if (!(G.plan == old)) drop_graphs();
    rc = ensure_ycoop(G);
    if (rc != ADI_OK) return rc;
  }
  G.hgd = GridDev{};
  G.hgd.k = 1;
  G.hgd.k0 = 1;
  G.hgd.src_ix = -1;
  G.hgd.src_iy = -1;
  G.hgd.kf[0] = G.hgd.kf[1] = 1;
  const bool has_src = sr && sr->ix >= 0 && sr->wavelet && sr->n_wavelet > 0;
  InitArgs ia = {};
  ia.nx = G.nx;
  ia.ny = G.ny;
  ia.ld = G.ld;
  ia.m = G.m;
  ia.phi = phi;
  ia.psi = psi;
  ia.u0 = G.buf[0];
  ia.u1 = G.buf[1];
  ia.tau = G.dt;
  ia.cx_half = G.dt * G.dt / (2.0 * G.hx * G.hx);
  ia.cy_half = G.dt * G.dt / (2.0 * G.hy * G.hy);
  ia.taylor = G.start == ADI_START_TAYLOR2 ? 1 : 0;
  ia.sx = has_src ? sr->ix : -1;
  ia.sy = has_src ? sr->iy : -1;
  ia.src_half = G.dt * G.dt / (2.0 * G.hx * G.hy);
  ia.wavelet = has_src ? sr->wavelet : nullptr;
  ia.n_wavelet = has_src ? sr->n_wavelet : 0;
  ia.gd_dst = G.gd;
  CK(launch_init(ia, G.hgd, st), "init kernel");
  launches += 1;
  G.cur = 1;
  G.k = 1;
  G.from_init = true;
  rr.valid = false;
  return ADI_OK;
}

int adi_wave::reset(const float* const* m, const float* const* phi, const float* const* psi,
                    const adi_source* src, cudaStream_t st) {
  for (size_t s = 0; s < g.size(); ++s) {
    if (!phi[s]) return fail(this, ADI_EINVAL, "phi is required");
    if (src && src[s].ix >= 0 &&
        (src[s].ix >= g[s].nx || src[s].iy < 0 || src[s].iy >= g[s].ny))
      return fail(this, ADI_EINVAL, "source node outside the grid");
  }
  for (size_t s = 0; s < g.size(); ++s) {
    int rc = start_grid((int)s, m ? m[s] : nullptr, phi[s], psi ? psi[s] : nullptr,
                        src ? &src[s] : nullptr, st);
    if (rc != ADI_OK) return rc;
  }
  return g.size() > 1 ? ensure_batch_tiles() : ADI_OK;
}

int adi_wave::prof_begin(cudaStream_t st, cudaEvent_t* a) {
  if (ev_pool.empty()) {
    cudaEvent_t e;
    CK(cudaEventCreate(&e), "event create");
    ev_pool.push_back(e);
  }
  *a = ev_pool.back();
  ev_pool.pop_back();
  CK(cudaEventRecord(*a, st), "event record");
  return ADI_OK;
}

int adi_wave::prof_end(cudaStream_t st, cudaEvent_t a, int kind) {
  if (ev_pool.empty()) {
    cudaEvent_t e;
    CK(cudaEventCreate(&e), "event create");
    ev_pool.push_back(e);
  }
  cudaEvent_t b = ev_pool.back();
  ev_pool.pop_back();
  CK(cudaEventRecord(b, st), "event record");
  prof.push_back(ProfRec{a, b, kind});
  return ADI_OK;
}

// Whether the steps are replayed as captured pairs.  Launched one by one they
// overlap, which those on either side of a graph's end do not.  Where the x
// sweep is the band form, which does not overlap, the graph's shorter gaps
// win on small grids (us per step at tau = 2h: 8000 x 64 13.4 and 14.4, 16384
// x 40 19.5 and 20.6, 8000 x 500 50.7 and 51.6; 8192^2 the same either way).
bool adi_wave::graph_steps(const Grid& G, bool one_pass) const {
  if (tuning.use_graph != 0) return tuning.use_graph > 0;
  return !one_pass && !model.active && G.plan.x_stage == ADI_STAGE_BAND && (size_t)G.nx * G.ny <= ((size_t)1 << 22);
}

// In the step as long as that costs less than a launch of its own.  Every CTA
// of the one-pass step goes through the whole list: eight entries per thread
// at most.  The x sweep's CTAs share it; its band form samples none.  us per
// step, in the step and by a launch: 128^2 (2.7 without receivers) 2048
// receivers 4.7, 4096 6.9 and 4.4; 1000^2 (7.5) 2048 9.0, 4096 10.8 and 9.7,
// 65536 62 and 11; 3001 x 1501 (21) 1024 22.9, 2048 24.6 and 22.9, 10^6 1950
// and 29; sweeps at 500 x 400 (10.4) 16384 11.9, 65536 14.9 and 11.9.
adi_wave::Sampling adi_wave::sampling_of(const Grid& G, int n_rec, bool one_pass) const {
  if (n_rec <= 0) return kNone;
  const GridPlan& P = G.plan;
  const int most = one_pass ? 8 * (P.tile_rows > 0 ? tile_threads() : patch_threads())
                            : P.x_stage == ADI_STAGE_BAND ? 0 : 16384;
  return n_rec <= most ? kInStep : kAfterStep;
}

// Samples u^k at the run's receivers (captured: the level is in the record,
// which the sweeps and the one-pass step keep in different words).
int adi_wave::enqueue_gather(Grid& G, cudaStream_t st, bool one_pass) {
  const long long lev = st != cap ? G.k : one_pass ? kRecordLevel + 1 + G.cur : kRecordLevel;
  CK(launch_gather(G.gd, G.buf[G.cur], G.ld, G.hgd.n_rec, lev, st), "gather launch");
  launches += 1;
  return ADI_OK;
}

int adi_wave::enqueue_step(Grid& G, cudaStream_t st, Sampling smp, bool one_pass) {
  float* u_cur = G.buf[G.cur];
  float* u_prev = G.buf[1 - G.cur];
  int rc = one_pass ? launch_fwd_tile(G, u_cur, u_prev, G.gd, G.cur, smp == kInStep, st != cap, st)
                    : launch_fwd(G, u_cur, u_prev, G.w, nullptr, G.gd, smp == kInStep, st);
  if (rc != ADI_OK) return rc;
  G.cur = 1 - G.cur;
  G.k += 1;
  G.from_init = false;
  return smp == kAfterStep ? enqueue_gather(G, st, one_pass) : ADI_OK;
}

// The same step as one launch (adi_tile.cu, adi_patch.cu).  par: which level
// word of gd it reads (it leaves the next level in the other one).  gather:
// sample u_cur at the run's receivers.
// by_value: the level and the source travel with the launch (it is not captured).
int adi_wave::launch_fwd_tile(Grid& G, const float* u_cur, float* u_prev, GridDev* gd, int par, bool gather,
                              bool by_value, cudaStream_t st) {
  const bool patch = G.plan.tile_rows == 0;
  auto encode = [&](CUtensorMap* out, const float* p, bool u) {
    return patch ? encode_patch_map(out, p, G.nx, G.ld, G.ny, u) : encode_tile_map(out, p, G.nx, G.ld, G.ny, false);
  };
  if (G.tt_form != (patch ? 2 : 1)) {
    for (int q = 0; q < 2; ++q) {
      CK(encode(&G.tt_buf[q], G.buf[q], true), "step map u");
      if (!patch) CK(encode_tile_map(&G.tt_strip[q], G.buf[q], G.nx, G.ld, G.ny, true), "step map u");
    }
    CK(encode(&G.tt_m, G.m, false), "step map m");
    G.tt_form = patch ? 2 : 1;
  }
  TileMaps mp;
  mp.m = G.tt_m;
  if (u_cur == G.buf[0] || u_cur == G.buf[1]) mp.u = G.tt_buf[u_cur == G.buf[1]];
  else CK(encode(&mp.u, u_cur, true), "step map");
  if (patch) {
    // u^{k-1} is read and written without a map
  } else if (u_prev == G.buf[0] || u_prev == G.buf[1]) {
    mp.o = G.tt_buf[u_prev == G.buf[1]];
    mp.p = G.tt_strip[u_prev == G.buf[1]];
  } else {
    CK(encode_tile_map(&mp.o, u_prev, G.nx, G.ld, G.ny, false), "step map");
    CK(encode_tile_map(&mp.p, u_prev, G.nx, G.ld, G.ny, true), "step map");
  }
  TileArgs a = tile_args(G);
  a.par = par;
  a.u_prev = u_prev;
  if (by_value) {
    a.by_value = 1;
    a.level = G.k;
    a.alone = G.k == G.hgd.k0;
    a.wavelet = G.hgd.wavelet;
    a.n_wavelet = G.hgd.n_wavelet;
    a.src_ix = G.hgd.src_ix;
    a.src_iy = G.hgd.src_iy;
  }
  a.u_cur = u_cur;
  a.rec = gather ? d_rec : nullptr;
  a.n_rec = gather ? G.hgd.n_rec : 0;
  a.gd = gd;
  a.err = d_err;
  cudaEvent_t ev = nullptr;
  if (profile && prof_begin(st, &ev) != ADI_OK) return ADI_ECUDA;
  CK(patch ? launch_patch(a, G.plan.tile, mp.u, mp.m, st) : launch_tile(a, G.plan.tile, mp, st), "step launch");
  if (profile && prof_end(st, ev, ADI_KERNEL_OTHER) != ADI_OK) return ADI_ECUDA;
  launches += 1;
  return ADI_OK;
}

// One forward step on explicit buffers: x sweep into w, y sweep + update
// writing u^{k+1} over u_prev (and z into z_out when given).  gather: sample
// u_cur at the run's receivers.
int adi_wave::launch_fwd(Grid& G, const float* u_cur, float* u_prev, float* w, float* z_out,
                         GridDev* gd, bool gather, cudaStream_t st) {
  const GridPlan& P = G.plan;
  XArgs xa;
  xa.nx = G.nx;
  xa.ny = G.ny;
  xa.ld = G.ld;
  xa.log2tsys = P.log2tsys;
  xa.spc = P.spc;
  xa.pcr = P.pcr;
  xa.m = G.m;
  xa.u = u_cur;
  xa.w = w;
  xa.cx = G.dt * G.dt / (G.hx * G.hx);
  xa.cy = G.dt * G.dt / (G.hy * G.hy);
  xa.sc = G.dt * G.dt / (2.0 * G.hx * G.hx);
  xa.src_scale = G.dt * G.dt / (G.hx * G.hy);
  xa.gd = gd;
  xa.persist = P.persist;
  xa.stage_mode = P.x_stage;
  xa.stage_off = -1;
  xa.err = d_err;
  xa.xc = P.xc;
  XRec xr;
  if (gather) {
    xr.rec = d_rec;
    xr.n_rec = G.hgd.n_rec;
  }
  YArgs ya;
  ya.nx = G.nx;
  ya.ny = G.ny;
  ya.ld = G.ld;
  ya.log2W = P.log2W;
  ya.log2tcol = P.log2tcol;
  ya.C = P.C;
  ya.pcr = P.pcr;
  ya.m = G.m;
  ya.w = w;
  ya.u_cur = u_cur;
  ya.u_prev = u_prev;
  ya.z_out = z_out;
  ya.stage_mode = P.y_stage;
  ya.persist = P.persist;
  ya.stage_off = 0;
  ya.sc = G.dt * G.dt / (2.0 * G.hy * G.hy);
  ya.gd = gd;
  ya.err = d_err;

  cudaEvent_t a = nullptr;
  if (profile && prof_begin(st, &a) != ADI_OK) return ADI_ECUDA;
  if (P.x_stage == 3 || P.x_stage == 5) {
    const int L = x_pipe_box_lines((1 << P.log2tsys) / P.xc, P.kx);
    if (G.tm_lines != L) {
      CK(encode_row_map(&G.tm_buf[0], G.buf[0], G.ld, G.ny, L), "tensor map u0");
      CK(encode_row_map(&G.tm_buf[1], G.buf[1], G.ld, G.ny, L), "tensor map u1");
      CK(encode_row_map(&G.tm_m, G.m, G.ld, G.ny, L), "tensor map m");
      CK(encode_row_map(&G.tm_w, G.w, G.ld, G.ny, L), "tensor map w");
      G.tm_lines = L;
    }
    CUtensorMap tmp, tmpw;
    const CUtensorMap* tu = u_cur == G.buf[0] ? &G.tm_buf[0] : u_cur == G.buf[1] ? &G.tm_buf[1] : nullptr;
    if (tu == nullptr) {
      CK(encode_row_map(&tmp, u_cur, G.ld, G.ny, L), "tensor map u");
      tu = &tmp;
    }
    const CUtensorMap* tw = &G.tm_w;
    if (w != G.w) {
      CK(encode_row_map(&tmpw, w, G.ld, G.ny, L), "tensor map w");
      tw = &tmpw;
    }
    if (P.x_stage == 5) CK(launch_x_band(xa, P.kx, *tu, G.tm_m, *tw, st), "x sweep launch");
    else CK(launch_x_pipe(xa, xr, P.kx, *tu, G.tm_m, *tw, st), "x sweep launch");
  } else {
    CK(launch_x(xa, xr, P.kx, P.fp64x, P.tree, st), "x sweep launch");
  }
  if (profile && prof_end(st, a, ADI_KERNEL_X) != ADI_OK) return ADI_ECUDA;
  if (profile && prof_begin(st, &a) != ADI_OK) return ADI_ECUDA;
  if (P.y_stage == 3 || P.y_stage == 4) {
    const int BH = y_pipe_box_rows(1 << P.log2tcol, P.ky);
    const int BW = 1 << P.log2W;
    if (G.ts_rows != BH * 64 + BW) {
      CK(encode_strip_map(&G.ts_buf[0], G.buf[0], G.ld, G.ny, BW, BH), "strip map u0");
      CK(encode_strip_map(&G.ts_buf[1], G.buf[1], G.ld, G.ny, BW, BH), "strip map u1");
      CK(encode_strip_map(&G.ts_m, G.m, G.ld, G.ny, BW, BH), "strip map m");
      CK(encode_strip_map(&G.ts_w, G.w, G.ld, G.ny, BW, BH), "strip map w");
      G.ts_rows = BH * 64 + BW;
    }
    YMaps mp;
    mp.m = G.ts_m;
    const float* want[3] = {w, u_cur, u_prev};
    CUtensorMap* outm[3] = {&mp.w, &mp.uc, &mp.up};
    for (int f = 0; f < 3; ++f) {
      const float* p = want[f];
      if (p == G.w) *outm[f] = G.ts_w;
      else if (p == G.buf[0]) *outm[f] = G.ts_buf[0];
      else if (p == G.buf[1]) *outm[f] = G.ts_buf[1];
      else CK(encode_strip_map(outm[f], p, G.ld, G.ny, BW, BH), "strip map");
    }
    if (P.y_stage == 4) CK(launch_y_coop(ya, P.ky, G.yc, mp, st), "y sweep launch");
    else CK(launch_y_pipe(ya, P.ky, mp, st), "y sweep launch");
  } else {
    CK(launch_y(ya, P.ky, P.fp64y, P.tree, st), "y sweep launch");
  }
  if (profile && prof_end(st, a, ADI_KERNEL_Y) != ADI_OK) return ADI_ECUDA;
  launches += 2;
  return ADI_OK;
}

void adi_wave::drop_graphs() {
  for (int o = 0; o < 2; ++o)
    for (int q = 0; q < 4; ++q)
      if (pair[o][q]) {
        cudaGraphExecDestroy(pair[o][q]);
        pair[o][q] = nullptr;
      }
}

int adi_wave::launch_pair_graph(Grid& G, cudaStream_t st, Sampling smp, bool one_pass) {
  cudaGraphExec_t& ex = pair[G.cur][(smp != kNone ? 1 : 0) + (one_pass ? 2 : 0)];
  if (!ex) {
    const int cur0 = G.cur;
    const long long k0 = G.k;
    const int64_t l0 = launches;
    CK(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "begin capture");
    int rc = enqueue_step(G, cap, smp, one_pass);
    if (rc == ADI_OK) rc = enqueue_step(G, cap, smp, one_pass);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(cap, &graph);
    G.cur = cur0;
    G.k = k0;
    launches = l0;
    if (rc != ADI_OK) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return cuda_fail(this, e, "end capture");
    e = cudaGraphInstantiate(&ex, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      ex = nullptr;
      return cuda_fail(this, e, "graph instantiate");
    }
  }
  CK(cudaGraphLaunch(ex, st), "graph launch");
  launches += 2 * ((one_pass ? 1 : 2) + (smp == kAfterStep ? 1 : 0));
  G.k += 2;
  return ADI_OK;
}

int adi_wave::run(int steps, const adi_source* src, const int32_t* rec_xy, int n_rec,
                  float* traces, cudaStream_t st, bool record) {
  if (steps < 0 || n_rec < 0) return fail(this, ADI_EINVAL, "negative steps or receiver count");
  if (n_rec > 0 && (g.size() != 1 || !rec_xy || !traces))
    return fail(this, ADI_EINVAL, "receivers need one grid, rec_xy and traces");
  for (size_t s = 0; s < g.size(); ++s) {
    if (src && src[s].ix >= 0 &&
        (src[s].ix >= g[s].nx || src[s].iy < 0 || src[s].iy >= g[s].ny))
      return fail(this, ADI_EINVAL, "source node outside the grid");
  }
  if (g.size() != 1) return run_batch(steps, src, st);
  Grid& G = g[0];
  for (int r = 0; r < n_rec; ++r) {
    if (rec_xy[2 * r] < 0 || rec_xy[2 * r] >= G.nx || rec_xy[2 * r + 1] < 0 ||
        rec_xy[2 * r + 1] >= G.ny)
      return fail(this, ADI_EINVAL, "receiver node outside the grid");
  }
  if (steps == 0) return ADI_OK;

  // per-run device state: level, source, receivers
  // (a caller's graph that holds the copy reads both ends at every replay)
  const int32_t* rec_host = rec_xy;
  if (n_rec > 0 && stream_captures(st)) {
    graph_recs.emplace_back(rec_xy, rec_xy + 2 * (size_t)n_rec);
    rec_host = graph_recs.back().data();
  }
  if (n_rec > rec_cap) {
    if (d_rec && !graph_recs.empty()) graph_recs_dev.push_back(d_rec);
    else if (d_rec) cudaFree(d_rec);
    d_rec = nullptr;
    rec_cap = 0;
    CK(cudaMalloc(&d_rec, sizeof(int) * 2 * (size_t)n_rec), "alloc receivers");
    rec_cap = n_rec;
  }
  if (n_rec > 0)
    CK(cudaMemcpyAsync(d_rec, rec_host, sizeof(int) * 2 * (size_t)n_rec, cudaMemcpyHostToDevice, st),
       "copy receivers");
  const adi_source none = {-1, -1, nullptr, 0};
  const adi_source sr = src ? src[0] : none;
  G.hgd.k = G.k;
  G.hgd.k0 = G.k;
  G.hgd.steps = steps;
  G.hgd.wavelet = (sr.ix >= 0) ? sr.wavelet : nullptr;
  G.hgd.n_wavelet = (sr.ix >= 0 && sr.wavelet) ? sr.n_wavelet : 0;
  G.hgd.src_ix = (sr.ix >= 0 && sr.wavelet) ? sr.ix : -1;
  G.hgd.src_iy = (sr.ix >= 0 && sr.wavelet) ? sr.iy : -1;
  G.hgd.n_rec = n_rec;
  G.hgd.rec = d_rec;
  G.hgd.traces = traces;
  const int every = record ? ckpt_every : 0;
  // A run that keeps checkpoints is one to be differentiated: its steps are
  // the separate sweeps, whose w and z the reverse sweep recomputes.  The
  // gradient is made of differences of nearly equal FP32 fields (z - w), so
  // its last digits follow the rounding of every forward value.
  const bool one_pass = G.plan.tile != 0 && every == 0 && !model.active;
  // (a graph cannot be launched into a stream that is being captured)
  const bool use_graph = graph_steps(G, one_pass) && !profile && !(tuning.use_graph == 0 && stream_captures(st));
  // chained one-pass steps carry level and source by value: without receivers
  // nothing reads the grid record
  if (!one_pass || use_graph || n_rec > 0)
    if (upload_gd(G, st) != ADI_OK) return ADI_ECUDA;

  rr.kept = 0;
  if (record) {
    rr.valid = true;
    rr.k0 = G.k;
    rr.steps = steps;
    rr.every = every;
    rr.taylor = G.start == ADI_START_TAYLOR2 && G.from_init && G.k == 1;
    rr.src = sr;
    rr.rec.assign(rec_xy ? rec_xy : (const int32_t*)nullptr,
                  rec_xy ? rec_xy + 2 * (size_t)n_rec : (const int32_t*)nullptr);
    const size_t need = every > 0 ? (size_t)((steps + every - 1) / every) : 0;
    const size_t fbytes = sizeof(float) * (size_t)G.ld * G.ny;
    if (rr.ckpt_bytes != fbytes) {
      for (float* p : rr.ckpt_mem) cudaFree(p);
      rr.ckpt_mem.clear();
      rr.ckpt.clear();
      rr.ckpt_bytes = fbytes;
    }
    if (rr.ckpt.size() < need) {
      float* p = nullptr;
      cudaError_t e = cudaMalloc(&p, 2 * fbytes * (need - rr.ckpt.size()));
      if (e != cudaSuccess) {
        cudaGetLastError();
        rr.valid = false;
        return fail(this, ADI_ENOMEM, "allocate checkpoints");
      }
      rr.ckpt_mem.push_back(p);
      for (; rr.ckpt.size() < need; p += 2 * (size_t)G.ld * G.ny) rr.ckpt.push_back(p);
    }
  }

  const bool gather = n_rec > 0;
  const Sampling smp = sampling_of(G, n_rec, one_pass);
  if (gather && (n_rec != graph_rec || d_rec != graph_rec_at)) {  // captured steps hold both
    drop_graphs();
    graph_rec = n_rec;
    graph_rec_at = d_rec;
  }
  const size_t fbytes = sizeof(float) * (size_t)G.ld * G.ny;
  // w and z of the last segments, as many as it has buffers for (two), go
  // straight into the workspace of the reverse sweep that is to come, which
  // then need not recompute them (the gradient at 1024^2, 100 steps in two
  // segments: 5.89 -> 4.83 ms; 301^2, 60 steps in three, with set-up: 2.99 ->
  // 2.78).  Where there is no
  // room the reverse sweep finds that out for itself.  Not while the stream
  // is being captured (the workspace may have to grow), nor ever after: a
  // replay writes the checkpoints behind this handle's back.
  const int nck = every > 0 ? (steps + every - 1) / every : 0;
  int keep = 0;
  if (record && every > 0) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(st, &cs), "capture status");
    if (cs != cudaStreamCaptureStatusNone) rr.captured = true;
  }
  if (record && every > 0 && gather && !model.active && !rr.captured && adj_beside(G)) {
    const std::string err0 = err;
    const int bufs = nck > 1 ? 2 : 1;
    if (adj_room(G, every, bufs) && ensure_adj_work(G, every, n_rec, bufs) == ADI_OK)
      keep = bufs > 1 ? aw.bufs : 1;
    err = err0;
  }
  int s = 0;
  while (s < steps) {
    int seg = steps - s;
    if (every > 0) {
      if (s % every == 0) {
        float* c = rr.ckpt[s / every];
        CK(cudaMemcpyAsync(c, G.buf[1 - G.cur], fbytes, cudaMemcpyDeviceToDevice, st), "checkpoint");
        CK(cudaMemcpyAsync(c + (size_t)G.ld * G.ny, G.buf[G.cur], fbytes, cudaMemcpyDeviceToDevice,
                           st), "checkpoint");
      }
      seg = std::min(seg, every - s % every);
    }
    int t = 0;
    if (keep > 0 && s >= (nck - keep) * every) {
      const size_t ffl = (size_t)G.ld * G.ny;
      const size_t off = ffl * every * (size_t)(s / every % keep);
      for (; t < seg; ++t) {
        int rc = launch_fwd(G, G.buf[G.cur], G.buf[1 - G.cur], aw.wseg + off + ffl * t, aw.zseg + off + ffl * t, G.gd,
                            smp == kInStep, st);
        if (rc != ADI_OK) {
          rr.kept = 0;
          return rc;
        }
        G.cur = 1 - G.cur;
        G.k += 1;
        G.from_init = false;
        if (smp == kAfterStep) {
          rc = enqueue_gather(G, st, false);
          if (rc != ADI_OK) return rc;
        }
      }
      rr.kept += 1;
      rr.kept_bufs = keep;
    }
    if (model.active) {
      while (t < seg) {
        int rc = enqueue_model_step(G, st, gather);
        if (rc != ADI_OK) return rc;
        t += 1;
      }
    }
    if (use_graph) {
      while (seg - t >= 2) {
        int rc = launch_pair_graph(G, st, smp, one_pass);
        if (rc != ADI_OK) return rc;
        t += 2;
      }
    }
    while (t < seg) {
      int rc = enqueue_step(G, st, smp, one_pass);
      if (rc != ADI_OK) return rc;
      t += 1;
    }
    s += seg;
  }
  if (smp == kInStep && !model.active) {  // the steps have sampled the levels before the last
    const int rc = enqueue_gather(G, st, one_pass);
    if (rc != ADI_OK) return rc;
  }
  G.hgd.k = G.k;
  return ADI_OK;
}

int adi_wave::set_state(int shot, const float* u_prev, const float* u_cur, int64_t k,
                        cudaStream_t st) {
  Grid& G = g[shot];
  G.k = k;
  G.from_init = false;
  G.hgd.k = k;
  G.hgd.k0 = k;
  G.hgd.kf[0] = G.hgd.kf[1] = k;
  G.hgd.steps = 0;
  CopyArgs c = {};
  c.nx = G.nx;
  c.ny = G.ny;
  c.spitch = G.nx;
  c.dpitch = G.ld;
  c.src0 = u_prev;
  c.src1 = u_cur;
  c.dst0 = G.buf[1 - G.cur];
  c.dst1 = G.buf[G.cur];
  c.gd_dst = G.gd;
  CK(launch_copy_fields(c, G.hgd, st), "set_state");
  launches += 1;
  rr.valid = false;
  return ADI_OK;
}

int adi_wave::sync_status(cudaStream_t st) {
  CK(cudaStreamSynchronize(st), "synchronize");
  int word = 0;
  CK(cudaMemcpy(&word, d_err, sizeof(int), cudaMemcpyDeviceToHost), "read error word");
  CK(cudaMemset(d_err, 0, sizeof(int)), "clear error word");
  if (word & ERR_TIMEOUT) return fail(this, ADI_ETIMEOUT, "a bounded device wait expired");
  if (word & ERR_NUMERIC) return fail(this, ADI_ENUMERIC, "non-finite value in the wavefield");
  return ADI_OK;
}

int adi_wave::set_tuning(const adi_wave_tuning& t) {
  std::vector<GridPlan> old;
  for (auto& G : g) old.push_back(G.plan);
  for (auto& G : g) {
    std::string why;
    int rc = plan_grid(G, t, why);
    if (rc != ADI_OK) {
      for (size_t s = 0; s < g.size(); ++s) g[s].plan = old[s];
      return fail(this, rc, why);
    }
  }
  for (auto& G : g) {
    int rc = ensure_ycoop(G);
    if (rc != ADI_OK) {
      for (size_t s = 0; s < g.size(); ++s) g[s].plan = old[s];
      return rc;
    }
  }
  tuning = t;
  drop_graphs();
  return g.size() > 1 ? ensure_batch_tiles() : ADI_OK;
}

int adi_wave::profile_read(double* ms, int64_t* counts, int n_kinds) {
  std::vector<double> acc(ADI_KERNEL_KINDS, 0.0);
  std::vector<int64_t> cnt(ADI_KERNEL_KINDS, 0);
  for (const ProfRec& r : prof) {
    CK(cudaEventSynchronize(r.b), "event sync");
    float t = 0.f;
    CK(cudaEventElapsedTime(&t, r.a, r.b), "event elapsed");
    acc[r.kind] += t;
    cnt[r.kind] += 1;
    ev_pool.push_back(r.a);
    ev_pool.push_back(r.b);
  }
  prof.clear();
  for (int k = 0; k < n_kinds && k < ADI_KERNEL_KINDS; ++k) {
    if (ms) ms[k] = acc[k];
    if (counts) counts[k] = cnt[k];
  }
  return ADI_OK;
}

adi_wave::~adi_wave() {
  cudaDeviceSynchronize();
  drop_graphs();
  for (auto& G : g) {
    cudaFree(G.mem);
    cudaFree(G.yc.tops);
    cudaFree(G.yc.sync);
  }
  for (float* p : rr.ckpt_mem) cudaFree(p);
  free_adj_work();
  for (const ProfRec& r : prof) {
    cudaEventDestroy(r.a);
    cudaEventDestroy(r.b);
  }
  for (cudaEvent_t e : ev_pool) cudaEventDestroy(e);
  if (d_err) cudaFree(d_err);
  if (scan_host) cudaFreeHost(const_cast<unsigned int*>(scan_host));
  if (d_rec) cudaFree(d_rec);
  for (int* p : graph_recs_dev) cudaFree(p);
  if (d_shots) cudaFree(d_shots);
  if (d_items) cudaFree(d_items);
  if (d_sync) cudaFree(d_sync);
  if (bt_dev) cudaFree(bt_dev);
  if (bt_items) cudaFree(bt_items);
  for (int b = 0; b < kBranches; ++b) {
    if (branch[b]) cudaStreamDestroy(branch[b]);
    if (join_ev[b]) cudaEventDestroy(join_ev[b]);
  }
  if (fork_ev) cudaEventDestroy(fork_ev);
  if (fork_adj) cudaEventDestroy(fork_adj);
  for (int b = 0; b < 2; ++b) {
    if (rev_ev[b]) cudaEventDestroy(rev_ev[b]);
    if (seg_ev[b]) cudaEventDestroy(seg_ev[b]);
  }
  if (rec_st) cudaStreamDestroy(rec_st);
  if (cap) cudaStreamDestroy(cap);
}


// ---------------------------------------------------------------------------
// problem class beyond the default (adi_models.cu)
// ---------------------------------------------------------------------------
int adi_wave::set_model(const adi_wave_model& mdl) {
  if (g.size() != 1) return fail(this, ADI_EUNSUPPORTED, "models need a single-grid handle");
  if (mdl.scheme < ADI_SCHEME_FACTORED || mdl.scheme > ADI_SCHEME_LISTING1)
    return fail(this, ADI_EINVAL, "unknown scheme");
  if (mdl.n_g < 0 || mdl.n_f < 0 || (mdl.g && mdl.n_g < 1) || (mdl.f && mdl.n_f < 1))
    return fail(this, ADI_EINVAL, "bad g or f length");
  if (mdl.scheme != ADI_SCHEME_FACTORED && (mdl.g || mdl.f))
    return fail(this, ADI_EINVAL, "the half-level schemes take no g or f");
  Model M;
  M.scheme = mdl.scheme;
  M.g = mdl.g;
  M.n_g = mdl.g ? mdl.n_g : 0;
  M.f = mdl.f;
  M.n_f = mdl.f ? mdl.n_f : 0;
  M.active = mdl.scheme != ADI_SCHEME_FACTORED || mdl.g != nullptr || mdl.f != nullptr;
  if (M.active) {
    // one-shot launch geometry: direct row loads, column strips over clusters
    Grid tmp = g[0];
    tmp.fp64mode = ADI_FP64_NEVER;
    adi_wave_tuning t = tuning;
    t.x_stage = ADI_STAGE_DIRECT;
    t.y_stage = ADI_STAGE_L2;
    t.solver = ADI_SOLVER_TREE;
    t.x_cluster = 0;
    std::string why;
    int rc = plan_grid(tmp, t, why);
    if (rc != ADI_OK) return fail(this, rc, "model launch geometry: " + why);
    M.plan = tmp.plan;
  }
  model = M;
  rr.valid = false;
  drop_graphs();
  return ADI_OK;
}

// One step of the active model: an x pass into the scratch field and a y pass,
// then the level advances (and the receivers sample the new field).
int adi_wave::enqueue_model_step(Grid& G, cudaStream_t st, bool gather) {
  const GridPlan& P = model.plan;
  float* A = G.buf[1 - G.cur];  // u^{k-1} (mode 0) or u^{k-1/2}
  float* B = G.buf[G.cur];      // u^k
  float* Wf = G.w;
  const int mode = model.scheme;
  ModelXArgs xa = {};
  xa.nx = G.nx; xa.ny = G.ny; xa.ld = G.ld;
  xa.log2tsys = P.log2tsys; xa.spc = P.spc; xa.mode = mode;
  xa.m = G.m; xa.a = A; xa.b = B; xa.out = Wf;
  xa.cx = G.dt * G.dt / (G.hx * G.hx);
  xa.cy = G.dt * G.dt / (G.hy * G.hy);
  xa.sc = G.dt * G.dt / (2.0 * G.hx * G.hx);
  xa.src_scale = G.dt * G.dt / (G.hx * G.hy);
  xa.tau2 = G.dt * G.dt;
  xa.g = model.g; xa.n_g = model.n_g;
  xa.f = model.f; xa.n_f = model.n_f;
  xa.level = G.k;
  xa.gd = G.gd;
  ModelYArgs ya = {};
  ya.nx = G.nx; ya.ny = G.ny; ya.ld = G.ld;
  ya.log2W = P.log2W; ya.log2tcol = P.log2tcol; ya.C = P.C; ya.mode = mode;
  ya.m = G.m; ya.w = Wf; ya.b = B; ya.io = A;
  ya.sc = G.dt * G.dt / (2.0 * G.hy * G.hy);
  ya.src_scale = G.dt * G.dt / (G.hx * G.hy);
  ya.g = model.g; ya.n_g = model.n_g;
  ya.level = G.k;
  ya.gd = G.gd;
  ya.err = d_err;
  CK(launch_x_model(xa, P.kx, st), "model x pass");
  CK(launch_y_model(ya, P.ky, st), "model y pass");
  launches += 2;
  if (gather) {
    CK(launch_gather(G.gd, A, G.ld, G.hgd.n_rec, kRecordLevel, st), "gather launch");
    launches += 1;
  }
  if (mode == ADI_SCHEME_FACTORED) {
    G.cur = 1 - G.cur;  // u^{k+1} over u^{k-1}: the usual swap
  } else {
    // half levels: u^{k+1/2} is in the scratch field, u^{k+1} over u^{k-1/2},
    // and u^k's buffer becomes the scratch (Algorithm 1's two swaps)
    G.buf[1 - G.cur] = Wf;
    G.buf[G.cur] = A;
    G.w = B;
    G.tm_lines = 0;  // cached tensor maps name the buffers by role
    G.ts_rows = 0;
    G.tt_form = 0;
  }
  G.k += 1;
  G.from_init = false;
  return ADI_OK;
}
