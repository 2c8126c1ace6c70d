// adi_batch_host.cu -- host side of the batched form: the one-launch step
// (tables of tensor maps and CTAs, form and band length) with the shots beside
// it that need the sweeps; per-shot chains of the plain kernels; and for the
// persistent kernel the per-shot geometry (every item is one full CTA of K = 16
// unknowns per thread, so items of different shots carry the same work), the
// work list, and one step.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <string>
#include <vector>

#include "adi_batch.h"
#include "adi_internal.h"
#include "adi_run.h"
#include "adi_sweeps.cuh"

using namespace adi;

#define CKB(call, what)                                          \
  do {                                                           \
    cudaError_t e_ = (call);                                     \
    if (e_ != cudaSuccess) return cuda_fail(this, e_, what);     \
  } while (0)

namespace {
int next_pow2(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}
int ilog2(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}
}  // namespace

int adi_wave::setup_batch(cudaStream_t st) {
  const int n = (int)g.size();
  batch_fp64 = false;
  for (const Grid& G : g) batch_fp64 |= G.plan.fp64x || G.plan.fp64y;
  const int maxT = batch_fp64 ? 512 : 1024;
  const int K = kBatchK;
  std::vector<BatchShot> shots(n);
  std::vector<int2> xitems, yitems;
  size_t smem = 0;
  for (int s = 0; s < n; ++s) {
    Grid& G = g[s];
    const int tsys = next_pow2((G.nx + K - 1) / K);
    const int tcol = next_pow2((G.ny + K - 1) / K);
    if (tsys > maxT || maxT / tcol < 4)
      return fail(this, ADI_EUNSUPPORTED, "grid too large for the batched form (nx, ny <= " +
                                               std::to_string(maxT * K / 4) + ")");
    const int spc = maxT / tsys;
    const int W = maxT / tcol;
    BatchShot& B = shots[s];
    B.x_items = (G.ny + spc - 1) / spc;
    B.y_items = (G.nx + W - 1) / W;
    const size_t ysm = align64(y_smem_bytes(W, 1, tcol, batch_fp64, true));
    smem = std::max(smem, x_smem_bytes(spc, tsys, batch_fp64, true));
    smem = std::max(smem, ysm + y_stage_bytes(maxT, K));
    for (int c = 0; c < 2; ++c) {
      XArgs& xa = B.xa[c];
      xa.nx = G.nx; xa.ny = G.ny; xa.ld = G.ld;
      xa.log2tsys = ilog2(tsys); xa.spc = spc; xa.pcr = 32;
      xa.m = G.m; xa.u = G.buf[c]; xa.w = G.w;
      xa.cx = G.dt * G.dt / (G.hx * G.hx);
      xa.cy = G.dt * G.dt / (G.hy * G.hy);
      xa.sc = G.dt * G.dt / (2.0 * G.hx * G.hx);
      xa.src_scale = G.dt * G.dt / (G.hx * G.hy);
      xa.gd = G.gd;
      xa.persist = 0;
      xa.stage_mode = 2;
      xa.stage_off = -1;
      xa.err = nullptr;
      xa.xc = 1;
      YArgs& ya = B.ya[c];
      ya.nx = G.nx; ya.ny = G.ny; ya.ld = G.ld;
      ya.log2W = ilog2(W); ya.log2tcol = ilog2(tcol); ya.C = 1; ya.pcr = 32;
      ya.m = G.m; ya.w = G.w; ya.u_cur = G.buf[c]; ya.u_prev = G.buf[1 - c]; ya.z_out = nullptr;
      ya.sc = G.dt * G.dt / (2.0 * G.hy * G.hy);
      ya.gd = G.gd; ya.err = d_err;
      ya.stage_off = (int)ysm;
      ya.stage_mode = 1;
      ya.persist = 0;
    }
    for (int i = 0; i < B.x_items; ++i) xitems.push_back(make_int2(s, i << 1));
    for (int i = 0; i < B.y_items; ++i) yitems.push_back(make_int2(s, (i << 1) | 1));
  }
  if (smem + 512 > (size_t)kMaxDynSmem)  // 512: the kernel's static shared variables
    return fail(this, ADI_EUNSUPPORTED, "batched kernel shared memory");
  std::vector<int2> items = xitems;
  items.insert(items.end(), yitems.begin(), yitems.end());
  n_items = (int)items.size();
  CKB(cudaMalloc(&d_shots, sizeof(BatchShot) * n), "alloc shot table");
  CKB(cudaMalloc(&d_items, sizeof(int2) * items.size()), "alloc work list");
  CKB(cudaMalloc(&d_sync, sizeof(int) * (1 + n)), "alloc counters");
  CKB(cudaMemcpyAsync(d_shots, shots.data(), sizeof(BatchShot) * n, cudaMemcpyHostToDevice, st),
      "upload shot table");
  CKB(cudaMemcpyAsync(d_items, items.data(), sizeof(int2) * items.size(), cudaMemcpyHostToDevice, st),
      "upload work list");
  CKB(cudaStreamSynchronize(st), "batch setup sync");
  int dev = 0, nsm = 0, b32 = 0, b64 = 0;
  CKB(cudaGetDevice(&dev), "get device");
  CKB(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev), "SM count");
  CKB(configure_batch_kernels(&b32, &b64, smem, smem), "configure batched kernel");
  const int per_sm = batch_fp64 ? b64 : b32;
  if (per_sm < 1) return fail(this, ADI_EUNSUPPORTED, "batched kernel does not fit an SM");
  batch_grid = nsm * per_sm;
  batch_smem = smem;
  return ADI_OK;
}

// One step of one shot by the single-grid kernels, buf[cur] = u^k.
int adi_wave::launch_batch_fwd(Grid& G, int cur, cudaStream_t st) {
  return G.plan.tile ? launch_fwd_tile(G, G.buf[cur], G.buf[1 - cur], G.gd, cur, false, false, st)
                     : launch_fwd(G, G.buf[cur], G.buf[1 - cur], G.w, nullptr, G.gd, false, st);
}

int adi_wave::enqueue_batch_step(cudaStream_t st) {
  const int n = (int)g.size();
  if (batch_mode == 2) return enqueue_batch_steps_parallel(1, st);
  if (batch_mode == 1) {
    for (Grid& G : g) {
      int rc = launch_batch_fwd(G, G.cur, st);
      if (rc != ADI_OK) return rc;
    }
  } else {
    CKB(cudaMemsetAsync(d_sync, 0, sizeof(int) * (1 + n), st), "clear counters");
    BatchArgs a;
    a.shots = d_shots;
    a.items = d_items;
    a.n_items = n_items;
    a.ticket = d_sync;
    a.x_done = d_sync + 1;
    a.cur = g[0].cur;
    a.err = d_err;
    a.spin_limit = spin_limit;
    a.never_ready_shot = never_ready;
    cudaEvent_t ev = nullptr;
    if (profile && prof_begin(st, &ev) != ADI_OK) return ADI_ECUDA;
    CKB(launch_batch(a, batch_fp64, batch_grid, batch_smem, st), "batched step launch");
    if (profile && prof_end(st, ev, ADI_KERNEL_OTHER) != ADI_OK) return ADI_ECUDA;
    launches += 1;
  }
  for (Grid& G : g) {
    G.cur = 1 - G.cur;
    G.k += 1;
    G.from_init = false;
  }
  return ADI_OK;
}

// Batch mode 2: every shot's steps are a chain of the single-grid kernels on
// one of kBranches streams; the branches fork from `st` and join back into
// it, so shots of different sizes overlap and fill each other's tails, with
// no barrier between shots inside the `nsteps` steps.  Shots go to branches
// largest first, each to the branch with the fewest grid points so far, so
// that the branches end together at the join (for 64 shots of 256^2 to
// 2048^2 the fullest branch holds 1.004 of an even share, against 1.36 with
// shot s on branch s mod kBranches); they are launched in that order too.
int adi_wave::ensure_branches() {
  if (fork_ev) return ADI_OK;
  for (int b = 0; b < kBranches; ++b) {
    CKB(cudaStreamCreateWithFlags(&branch[b], cudaStreamNonBlocking), "create branch stream");
    CKB(cudaEventCreateWithFlags(&join_ev[b], cudaEventDisableTiming), "create join event");
  }
  CKB(cudaEventCreateWithFlags(&fork_ev, cudaEventDisableTiming), "create fork event");
  return ADI_OK;
}

// Tables of the one-launch step: built with the handle and again when a reset
// or a tuning has changed a plan, so that no run allocates (a caller may be
// capturing it).  All such shots take the same form
// and the largest halo any of them needs: patches, or bands of the length
// that gives the shortest step by the times of tile_band_rows(), the longest
// CTAs first.
int adi_wave::ensure_batch_tiles() {
  std::vector<GridPlan> plans;
  for (const Grid& G : g) plans.push_back(G.plan);
  if (plans == bt_plans) return ADI_OK;
  bt_n = 0;
  std::vector<int> shots;
  bt_h = 12;
  for (size_t s = 0; s < g.size(); ++s)
    if (g[s].plan.tile) {
      shots.push_back((int)s);
      bt_h = std::max(bt_h, g[s].plan.tile);
    }
  bt_plans.clear();  // until the tables are in place: a failure below is not taken for them
  if (shots.size() < 2) {
    bt_plans = plans;
    return ADI_OK;
  }
  int dev = 0, nsm = 0;
  CKB(cudaGetDevice(&dev), "get device");
  CKB(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev), "SM count");
  const double slots = 2.0 * nsm;
  double patches = 0;
  int max_blocks = 1;
  bool wide = true;
  for (int s : shots) {
    patches += (double)patch_strips(g[s].nx) * ((g[s].ny + patch_rows(bt_h) - 1) / patch_rows(bt_h));
    max_blocks = std::max(max_blocks, (g[s].ny + 15) / 16);
    wide = wide && g[s].nx >= 224;
  }
  double best = 1.2 + 6.3 * std::max(1.0, std::ceil(patches / slots));
  int best_b = 0;
  // bands of b blocks with their halo: the time of the slot that ends last when the CTAs,
  // longest first, each go to the slot that is free first (even shares alone
  // would choose bands of which a few are left over for a second round: 32
  // shots of 256^2 to 2048^2 174 us per step instead of 130)
  auto band_len = [&](int ny, int rows, int q, int bands) {
    const int own = std::min(rows, ny - q * rows);
    return (own + (q > 0 ? bt_h : 0) + (q + 1 < bands ? bt_h : 0) + 15) / 16;
  };
  // no schedule ends before the longest CTA or an even share: lengths by that
  // bound, until it rules out the rest
  std::vector<std::pair<double, int>> bound;
  for (int b = 4; wide && b < std::min(2 * max_blocks, 128); ++b) {
    const int rows = 16 * b - 2 * bt_h;
    long long total = 0;
    int longest = 0;
    for (int s : shots) {
      const int bands = (g[s].ny + rows - 1) / rows;
      longest = std::max(longest, band_len(g[s].ny, rows, bands > 2 ? 1 : 0, bands));
      total += (long long)tile_strips(g[s].nx) * ((g[s].ny + 2 * (bands - 1) * bt_h + 15) / 16);
    }
    bound.emplace_back(3.5 + 3.05 * std::max((double)longest, total / slots), b);
  }
  std::sort(bound.begin(), bound.end());
  for (const auto& lb : bound) {
    if (lb.first >= best) break;
    const int b = lb.second, rows = 16 * b - 2 * bt_h;
    std::vector<long long> count(b + 1, 0);  // CTAs by blocks
    for (int s : shots) {
      const int bands = (g[s].ny + rows - 1) / rows;
      for (int q = 0; q < bands; ++q) count[band_len(g[s].ny, rows, q, bands)] += tile_strips(g[s].nx);
    }
    std::vector<int> ends(1, (int)slots);  // slots by the time they are free
    size_t now = 0;                        // the first of them: it never goes back
    for (int len = b; len > 0; --len)
      for (long long i = 0; i < count[len]; ++i) {
        while (ends[now] == 0) ++now;
        if (ends.size() <= now + len) ends.resize(now + len + 1, 0);
        ends[now] -= 1;
        ends[now + len] += 1;
      }
    const int last = (int)ends.size() - 1;
    const double t = 3.5 + 3.05 * last;
    if (t < best || (t == best && b < best_b)) {
      best = t;
      best_b = b;
    }
  }
  bt_patch = best_b == 0;
  std::vector<BatchTile> tiles;
  struct Item {
    int cost;
    int2 it;
  };
  std::vector<Item> items;
  for (int s : shots) {
    Grid& G = g[s];
    BatchTile t = {};
    for (int q = 0; q < 2; ++q) {
      if (bt_patch) {
        CKB(encode_patch_map(&t.u[q], G.buf[q], G.nx, G.ld, G.ny, true), "batch map u");
      } else {
        CKB(encode_tile_map(&t.u[q], G.buf[q], G.nx, G.ld, G.ny, false), "batch map u");
        CKB(encode_tile_map(&t.p[q], G.buf[q], G.nx, G.ld, G.ny, true), "batch map u");
      }
      t.buf[q] = G.buf[q];
    }
    if (bt_patch) CKB(encode_patch_map(&t.m, G.m, G.nx, G.ld, G.ny, false), "batch map m");
    else CKB(encode_tile_map(&t.m, G.m, G.nx, G.ld, G.ny, false), "batch map m");
    t.a = tile_args(G);
    t.a.gd = G.gd;
    t.a.err = d_err;
    t.a.band_rows = bt_patch ? patch_rows(bt_h) : 16 * best_b - 2 * bt_h;
    t.a.strips = bt_patch ? patch_strips(G.nx) : tile_strips(G.nx);
    const int bands = (G.ny + t.a.band_rows - 1) / t.a.band_rows;
    for (int b = 0; b < bands; ++b)
      for (int c = 0; c < t.a.strips; ++c) {
        items.push_back(Item{bt_patch ? 0 : -band_len(G.ny, t.a.band_rows, b, bands), make_int2((int)tiles.size(), b * t.a.strips + c)});
      }
    tiles.push_back(t);
  }
  std::stable_sort(items.begin(), items.end(), [](const Item& x, const Item& y) { return x.cost < y.cost; });
  std::vector<int2> list;
  for (const Item& i : items) list.push_back(i.it);
  cudaFree(bt_dev);
  cudaFree(bt_items);
  bt_dev = nullptr;
  bt_items = nullptr;
  CKB(cudaMalloc(&bt_dev, sizeof(BatchTile) * tiles.size()), "alloc batch tables");
  CKB(cudaMalloc(&bt_items, sizeof(int2) * list.size()), "alloc batch tables");
  // On the handle's own stream, and waited for: a copy from pageable memory on
  // the legacy stream may return before it has landed, and a non-blocking
  // stream of the caller's is not ordered behind it.
  CKB(cudaMemcpyAsync(bt_dev, tiles.data(), sizeof(BatchTile) * tiles.size(), cudaMemcpyHostToDevice, cap), "batch tables");
  CKB(cudaMemcpyAsync(bt_items, list.data(), sizeof(int2) * list.size(), cudaMemcpyHostToDevice, cap), "batch tables");
  CKB(cudaStreamSynchronize(cap), "batch tables");
  if (tiles.size() < g.size()) {
    const int rc = ensure_branches();
    if (rc != ADI_OK) return rc;
  }
  bt_n = (int)tiles.size();
  bt_n_items = (int)list.size();
  bt_plans = plans;
  return ADI_OK;
}

// One step of the one-pass shots, the buf[par] = u^k.
int adi_wave::launch_batch_tiles(int par, cudaStream_t st) {
  cudaEvent_t ev = nullptr;
  if (profile && prof_begin(st, &ev) != ADI_OK) return ADI_ECUDA;
  CKB(bt_patch ? launch_patch_batch(bt_dev, bt_items, bt_n_items, par, bt_h, st)
               : launch_tile_batch(bt_dev, bt_items, bt_n_items, par, bt_h, st), "batched step launch");
  if (profile && prof_end(st, ev, ADI_KERNEL_OTHER) != ADI_OK) return ADI_ECUDA;
  launches += 1;
  return ADI_OK;
}

// `steps` steps of every shot: one launch per step for the one-pass shots on
// st and, beside them, the others' sweeps on branches that fork from st
// before the first step and join it after the last: pairs of steps of all of
// them replayed from a graph, or chains of launches, a shot to a branch, where
// graphs are off or st is being captured itself.  (Sweeps launched step by
// step behind the one-pass steps, with a fork and a join each, took 8 strong
// and 24 weak shots of 256^2 from 54 to 94 us a step.)
int adi_wave::run_batch_tiles(int steps, cudaStream_t st) {
  const int cur0 = g[0].cur;  // the shots advance together: one orientation
  const bool rest = bt_n < (int)g.size();
  int t = 0;
  if (rest) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    CKB(cudaStreamIsCapturing(st, &cs), "capture status");
    if (g[0].plan.graph && !profile && cs == cudaStreamCaptureStatusNone && steps >= 2) {
      cudaGraphExec_t& ex = pair[cur0][1];
      if (!ex) {
        const int rc2 = capture_batch_pair(&ex, true);
        if (rc2 != ADI_OK) return rc2;
      }
      CKB(cudaEventRecord(fork_ev, st), "fork");
      CKB(cudaStreamWaitEvent(branch[0], fork_ev, 0), "branch wait");
      for (; steps - t >= 2; t += 2) {
        CKB(cudaGraphLaunch(ex, branch[0]), "graph launch");
        launches += pair_launches;
        for (int q = 0; q < 2; ++q) {
          const int rc2 = launch_batch_tiles(cur0 ^ (q & 1), st);
          if (rc2 != ADI_OK) return rc2;
        }
      }
      for (Grid& G : g)
        if (!G.plan.tile) {
          G.k += t;
          G.from_init = false;
        }
      CKB(cudaEventRecord(join_ev[0], branch[0]), "join");
      CKB(cudaStreamWaitEvent(st, join_ev[0], 0), "join wait");
    }
  }
  if (rest && t < steps) {
    const int t0 = t;
    const int rc = enqueue_batch_steps_parallel(steps - t0, st, true, [&](int q) { return launch_batch_tiles(cur0 ^ ((t0 + q) & 1), st); });
    if (rc != ADI_OK) return rc;
    t = steps;
  }
  for (; t < steps; ++t) {
    const int rc = launch_batch_tiles(cur0 ^ (t & 1), st);
    if (rc != ADI_OK) return rc;
  }
  for (Grid& G : g) {
    if (!G.plan.tile) continue;  // advanced above
    if (steps & 1) G.cur = 1 - G.cur;
    G.k += steps;
    G.from_init = false;
  }
  return ADI_OK;
}

// rest: only the shots that the one-launch step leaves.  beside(t): called as
// step t of the shots is in their branches.
int adi_wave::enqueue_batch_steps_parallel(int nsteps, cudaStream_t st, bool rest,
                                           const std::function<int(int)>& beside) {
  int rc = ensure_branches();
  if (rc != ADI_OK) return rc;
  const int n = (int)g.size();
  const int nb = std::min(n, (int)kBranches);
  if ((int)shot_order.size() != n) {
    shot_order.resize(n);
    shot_branch.assign(n, 0);
    for (int s = 0; s < n; ++s) shot_order[s] = s;
    std::stable_sort(shot_order.begin(), shot_order.end(), [&](int a, int b) {
      return (long long)g[a].nx * g[a].ny > (long long)g[b].nx * g[b].ny;
    });
    std::vector<long long> load(nb, 0);
    for (int s : shot_order) {
      const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
      shot_branch[s] = b;
      load[b] += (long long)g[s].nx * g[s].ny;
    }
  }
  CKB(cudaEventRecord(fork_ev, st), "fork");
  for (int b = 0; b < nb; ++b) CKB(cudaStreamWaitEvent(branch[b], fork_ev, 0), "branch wait");
  // shot by shot, so that a shot's steps find its fields in L2; step by step
  // where other launches are to start before the last of these is issued
  const int rounds = beside ? nsteps : 1, per = nsteps / rounds;
  for (int t = 0; t < rounds; ++t) {
    for (int s : shot_order) {
      Grid& G = g[s];
      if (rest && G.plan.tile) continue;
      for (int q = 0; q < per; ++q) {
        rc = launch_batch_fwd(G, G.cur ^ ((t + q) & 1), branch[shot_branch[s]]);
        if (rc != ADI_OK) return rc;
      }
    }
    if (beside) {
      rc = beside(t);
      if (rc != ADI_OK) return rc;
    }
  }
  for (int b = 0; b < nb; ++b) {
    CKB(cudaEventRecord(join_ev[b], branch[b]), "join");
    CKB(cudaStreamWaitEvent(st, join_ev[b], 0), "join wait");
  }
  for (Grid& G : g) {
    if (rest && G.plan.tile) continue;
    if (nsteps & 1) G.cur = 1 - G.cur;
    G.k += nsteps;
    G.from_init = false;
  }
  return ADI_OK;
}
