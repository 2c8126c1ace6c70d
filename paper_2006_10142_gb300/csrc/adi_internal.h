// adi_internal.h -- host/device structures shared by the library's .cu files.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace adi {

// Per-grid state read by the kernels from device memory, so that a captured
// CUDA graph picks up the current run's source and receivers on replay.
struct GridDev {
  long long k;          // time level of u_cur (u^k); the y sweep advances it
  long long k0;         // level at the start of the current run
  long long steps;      // length of the current run (bounds of traces)
  const float* wavelet; // w(t_k) samples, or null
  int n_wavelet;
  int src_ix, src_iy;   // source node, src_ix < 0 = none
  int n_rec;
  const int* rec;       // [n_rec][2] receiver nodes
  float* traces;        // [steps][n_rec]
  // The one-pass step (adi_tile.cu) has CTAs that read the level while
  // others finish, so the level alternates between two words: a step reads
  // kf[par] and leaves its successor in kf[1 - par].
  long long kf[2];
};

// Device error word bits.
enum : int { ERR_NUMERIC = 1, ERR_TIMEOUT = 2 };

// Arguments of the fused RHS + x-sweep kernel (Eq. fr1's x operator).
struct XArgs {
  int nx, ny, ld;
  int log2tsys;   // threads per row (system) = 1 << log2tsys
  int spc;        // rows per CTA
  int pcr;        // CR -> PCR switch size
  const float* m;
  const float* u;   // u^k
  float* w;         // out: w = X^{-1} r
  double cx, cy;    // tau^2 / h1^2, tau^2 / h2^2
  double sc;        // tau^2 / (2 h1^2): s = sc * m
  double src_scale; // tau^2 / (h1 h2)
  const GridDev* gd;
  int persist;      // 1: persistent CTAs loop over row blocks (grid set by the launcher)
  int stage_mode;   // 1: rows staged through shared memory (FP32), 2: direct loads, 3: TMA pipeline
  int stage_off;    // byte offset of the staging area (set by the launcher), -1: none
  int* err;         // device error word (bounded waits), or null
  int xc;           // TMA pipeline: 2 = each row split over a cluster of two CTAs, else 1
};

// Receivers at which an x sweep samples u^k into gd's traces.  Beside XArgs,
// not in it: the band form, which samples none, ran 6 to 8 % slower with the
// arguments that follow moved (0.707 to 0.762 ms at 16384^2).
struct XRec {
  const int* rec = nullptr;  // [n_rec][2]
  int n_rec = 0;
};

// Arguments of the y-sweep + update kernel (Eq. fr2's y operator).
struct YArgs {
  int nx, ny, ld;
  int log2W;      // columns per strip = 1 << log2W
  int log2tcol;   // threads per column in one CTA
  int C;          // CTAs per cluster along the column
  int pcr;
  const float* m;
  const float* w;      // RHS
  const float* u_cur;  // u^k
  float* u_prev;       // in: u^{k-1}; out: u^{k+1}
  float* z_out;        // optional copy of z = u^{k+1} - 2u^k + u^{k-1} (adjoint recompute)
  double sc;           // tau^2 / (2 h2^2)
  GridDev* gd;         // k is advanced by one CTA
  int* err;
  int stage_off;       // byte offset of the u^k / u^{k-1} staging area in shared memory, -1: L2
  int stage_mode;      // 1: shared-memory staging, 2: L2 prefetch (launchers set stage_off)
  int persist;         // 1: persistent clusters loop over strips (grid set by the launcher)
};

// Launchers (adi_forward.cu).
cudaError_t launch_x(const XArgs& a, const XRec& rec, int K, bool fp64, bool tree, cudaStream_t st);
cudaError_t launch_y(const YArgs& a, int K, bool fp64, bool tree, cudaStream_t st);
// lev: the level of u_new, or kRecordLevel: gd->k, kRecordLevel + 1 + q: gd->kf[q]
constexpr long long kRecordLevel = -0x7fffffffffffffffll;
cudaError_t launch_gather(const GridDev* gd, const float* u_new, int ld, int n_rec, long long lev, cudaStream_t st);
// Fields between the caller's contiguous rows and the handle's pitched ones
// (adi_copy.cu): dst0 <- src0 and, if src1 is given, dst1 <- src1; without
// src1 a given dst1 gets src0 too.  Both launches also write the grid record
// gd to gd_dst if that is given.
struct CopyArgs {
  int nx, ny;
  int spitch, dpitch;  // floats per row
  const float* src0;
  const float* src1;
  float* dst0;
  float* dst1;
  GridDev* gd_dst;
};
cudaError_t launch_copy_fields(const CopyArgs& a, const GridDev& gd, cudaStream_t st);
struct InitArgs {
  int nx, ny, ld;
  const float* m;    // pitched
  const float* phi;  // contiguous, psi too (or null)
  const float* psi;
  float* u0;
  float* u1;
  double tau, cx_half, cy_half;
  int taylor;
  int sx, sy;
  double src_half;
  const float* wavelet;
  int n_wavelet;
  GridDev* gd_dst;
};
cudaError_t launch_init(const InitArgs& a, const GridDev& gd, cudaStream_t st);
// min(m), max(m) bit patterns and a non-finite/non-positive flag into out3
// (device) and then host3 (mapped pinned host memory, device address): three
// launches, no copies.
cudaError_t launch_scan_m(const float* m, int nx, int ny, int ld, unsigned int* out3,
                          unsigned int* host3, cudaStream_t st);
// *dst[i] = v[i] on the stream for i < n (the records travel as kernel arguments).
cudaError_t launch_put_gd(GridDev* const* dst, const GridDev* v, int n, cudaStream_t st);
size_t x_smem_bytes(int spc, int tsys, bool fp64, bool tree);
size_t y_smem_bytes(int W, int C, int tcol, bool fp64, bool tree);
size_t y_stage_bytes(int threads, int K);
size_t x_stage_bytes(int threads, int K);
size_t x_pipe_smem_bytes(int spc, int tsys, int K, int xc);
int x_pipe_box_lines(int tsys, int K);
size_t y_pipe_smem_bytes(int W, int C, int tcol, int K);
int y_pipe_box_rows(int tcol, int K);
cudaError_t encode_strip_map(CUtensorMap* out, const float* base, int ld, int ny, int box_cols,
                             int box_rows);
// Strip maps of the pipelined y sweep: w, m, u^k, u^{k-1}.
struct YMaps {
  CUtensorMap w, m, uc, up;
};
cudaError_t launch_y_pipe(const YArgs& a, int K, const YMaps& mp, cudaStream_t st);
// The same kernel on the reverse step's column systems: wbar (z_out) from
// lam (strip map `lam`) and m (a.m and strip map `m`); u fields unused.
cudaError_t launch_y_pipe_adj(const YArgs& a, int K, const CUtensorMap& lam, const CUtensorMap& m,
                              cudaStream_t st);
// Column solves without clusters (adi_ycoop.cu): persistent co-resident CTAs
// take (strip, segment) items; the C segments of a column meet through
// global memory.  Scratch of one grid:
struct YCoop {
  int C;        // segments per column (1..32)
  int cols;     // columns the summaries hold (nx rounded up to 32)
  int strips;   // strips the counters hold (nx / 16 rounded up)
  float* tops;  // [cols][C] segment summaries, 8 floats each
  int* sync;    // [strips][2] arrival / completion counters, zero between launches
};
size_t y_coop_smem_bytes(int W, int tcol, int K, int C);
int y_coop_segments(int ny, int tcol, int K);
cudaError_t launch_y_coop(const YArgs& a, int K, const YCoop& yc, const YMaps& mp, cudaStream_t st);
cudaError_t launch_y_coop_adj(const YArgs& a, int K, const YCoop& yc, const CUtensorMap& lam,
                              const CUtensorMap& m, cudaStream_t st);
cudaError_t configure_y_coop_kernels();

// One whole step in one pass, for systems whose couplings decay fast enough
// (adi_tile.cu, adi_patch.cu): x and y solves are local, with halos of H
// unknowns.
struct TileArgs {
  int nx, ny, ld;
  int strips;          // set by the launcher
  int band_rows;       // rows of a band
  int small;           // patches of 32 columns instead of 96
  int par;             // which of gd->kf holds the level
  float cx, cy;        // tau^2 / h1^2, tau^2 / h2^2
  float scx, scy;      // tau^2 / (2 h1^2), tau^2 / (2 h2^2)
  float src_scale;     // tau^2 / (h1 h2)
  float* u_prev;       // in: u^{k-1}; out: u^{k+1}
  // The step's level and source: by value, so that the wavelet's
  // sample is fetched before the step before is done, or from gd (by_value = 0:
  // captured steps and batches, whose arguments outlive a run).  The first
  // step of a run waits for all that is before it (alone): the wavelet may be
  // the work of the caller's last kernel.
  int by_value, alone;
  long long level;
  const float* wavelet;
  int n_wavelet, src_ix, src_iy;
  const float* u_cur;  // u^k, for the receivers
  const int* rec;      // [n_rec][2] receivers to sample u^k at
  int n_rec;           // 0 = none
  GridDev* gd;
  int* err;
};
struct TileMaps {
  CUtensorMap u, m;  // u^k, m (panel boxes)
  CUtensorMap p, o;  // u^{k-1}: strip boxes to read, panel boxes to write
};
// Halo the local solves need for off-diagonals up to s_max (12 or 16), 0 =
// the couplings decay too slowly.
int tile_halo(double s_max);
int tile_strips(int nx);
int tile_threads();  // per CTA
// rows of a band, or 0 = by patches
int tile_band_rows(int nx, int ny, int H, int nsm);
cudaError_t encode_tile_map(CUtensorMap* out, const float* base, int nx, int ld, int ny, bool strip);
cudaError_t launch_tile(const TileArgs& a, int H, const TileMaps& mp, cudaStream_t st);
cudaError_t configure_tile_kernels();
// The same step patch by patch (adi_patch.cu).
int patch_rows(int H);
int patch_strips(int nx);
int patch_threads();
int small_patch_strips(int nx);
cudaError_t encode_patch_map(CUtensorMap* out, const float* base, int nx, int ld, int ny, bool u);
cudaError_t launch_patch(const TileArgs& a, int H, const CUtensorMap& u, const CUtensorMap& m, cudaStream_t st);
cudaError_t configure_patch_kernels();
// One grid of a batch advanced by one launch per step: arguments (par and
// u_prev from the launch) and tensor maps, in device memory.
struct alignas(128) BatchTile {
  CUtensorMap u[2], p[2], m;  // of buf[0], buf[1] (panel and strip boxes) and m
  TileArgs a;
  float* buf[2];
};
cudaError_t launch_tile_batch(const BatchTile* tiles, const int2* items, int n_items, int par, int H,
                              cudaStream_t st);
cudaError_t launch_patch_batch(const BatchTile* tiles, const int2* items, int n_items, int par, int H,
                               cudaStream_t st);
// 2D tensor map {nx, ny} of a field of row pitch ld with boxes of {box_cols,
// box_rows}, zero fill outside, optionally in the 128-byte swizzle
// (box_cols = 32).
cudaError_t encode_box_map(CUtensorMap* out, const float* base, int nx, int ld, int ny, int box_cols,
                           int box_rows, bool swizzle);

// The wider problem class and the literal half-level schemes (adi_models.cu).
// mode 0: Eq. CN1 with m^k = g_k m and a source field; 1: Eqs. fr1 / fr2 over
// half levels; 2: Listing 1's systems over half levels.
struct ModelXArgs {
  int nx, ny, ld, log2tsys, spc, mode;
  const float* m;
  const float* a;     // mode 0: u^{k-1}; modes 1, 2: u^{k-1/2}
  const float* b;     // u^k
  float* out;         // mode 0: w; modes 1, 2: u^{k+1/2}
  double cx, cy;      // tau^2 / h1^2, tau^2 / h2^2
  double sc;          // tau^2 / (2 h1^2)
  double src_scale;   // tau^2 / (h1 h2)
  double tau2;        // tau^2
  const float* g;     // [n_g] per-level factor of m (mode 0), or null
  int n_g;
  const float* f;     // [n_f][ny][nx] per-level source field (mode 0), or null
  int n_f;
  long long level;    // k
  const GridDev* gd;  // point source
};
struct ModelYArgs {
  int nx, ny, ld, log2W, log2tcol, C, mode;
  const float* m;
  const float* w;     // mode 0: the x pass's result; modes 1, 2: u^{k+1/2}
  const float* b;     // u^k
  float* io;          // mode 0: u^{k-1} in, u^{k+1} out; modes 1, 2: u^{k+1} out
  double sc;          // tau^2 / (2 h2^2)
  double src_scale;
  const float* g;
  int n_g;
  long long level;
  GridDev* gd;
  int* err;
};
cudaError_t launch_x_model(const ModelXArgs& a, int K, cudaStream_t st);
cudaError_t launch_y_model(const ModelYArgs& a, int K, cudaStream_t st);
cudaError_t configure_model_kernels();
// Row tensor map for the pipelined x sweep (see adi_tma.cuh).
cudaError_t encode_row_map(CUtensorMap* out, const float* base, int ld, int ny, int box_lines);
cudaError_t launch_x_pipe(const XArgs& a, const XRec& rec, int K, const CUtensorMap& tu, const CUtensorMap& tm,
                          const CUtensorMap& tw, cudaStream_t st);
// Band form of the x sweep (x_stage 5): clusters of xc = 2, 4 or 8 CTAs walk
// bands of consecutive rows with a ring of three rows of u^k in shared memory.
size_t x_band_smem_bytes(int tsys, int K, int xc);
cudaError_t launch_x_band(const XArgs& a, int K, const CUtensorMap& tu, const CUtensorMap& tm,
                          const CUtensorMap& tw, cudaStream_t st);
constexpr int kMaxDynSmem = 227 * 1024;
cudaError_t configure_kernels();
// Kernel attributes of every kernel of the library on the current device,
// once per device (thread-safe); adi_run.cu.
cudaError_t configure_current_device();

}  // namespace adi
