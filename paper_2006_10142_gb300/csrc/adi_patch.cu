// adi_patch.cu -- the one-pass step of adi_tile.cu for grids that fit the
// caches, where a step is a chain of latencies rather than a stream.
//
// adi_tile.cu marches down a band block by block; on a small grid the blocks
// of the one band a CTA has (two of them halo) follow one another at about
// 2 us each.  Here a CTA takes a patch of 64 x 128 staged points (96 columns
// and 64 - 2H rows of its own) all at once: the row solves of all 64 rows run
// side by side, then the column solves, four chunks of 16 rows to a column,
// with the same hand-over between chunks as along the rows.  The halo rows
// cost 64 / (64 - 2H) of the work, which the idle SMs have to spare.
//   x phase: 256 threads = 4 groups of 16 rows x 8 chunks of 16 unknowns x 8
//     row pairs (r, r + 8), one pair in packed arithmetic per thread;
//   y phase: 192 threads = 4 chunks of 16 rows x 48 column pairs.
// Two CTAs per SM; consecutive steps overlap their launches (adi_local.cuh),
// and m, which no step writes, is fetched before the previous step is done.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "adi_bodies.cuh"
#include "adi_device.cuh"
#include "adi_internal.h"
#include "adi_local.cuh"
#include "adi_sweeps.cuh"
#include "adi_tma.cuh"

namespace adi {

namespace {

constexpr int kPX = 96;                 // columns of a patch
constexpr int kPH = 16;                 // halo columns on either side
constexpr int kPR = 64;                 // staged rows
constexpr int kPN = 256;                // threads
constexpr int kPCols = kPX + 2 * kPH;   // staged columns
constexpr int kPChunks = kPCols / 16;
constexpr int kUPanel = 72 * 128;       // u: rows -1 .. 64 of a 32-column panel (66), to a multiple of 8
constexpr int kMPanel = kPR * 128;
constexpr int kPairs = kPX / 2;
// shared memory: u | m | w | XT[9][32] 16 B | X0[9][32] 8 B | YT[5][48] 16 B | Y0[5][48] 8 B | mbarrier
constexpr int kPOffM = (kPCols / 32) * kUPanel;
constexpr int kPOffW = kPOffM + (kPCols / 32) * kMPanel;
constexpr int kPOffXT = kPOffW + (kPX / 32) * kMPanel;
constexpr int kPOffX0 = kPOffXT + (kPChunks + 1) * 32 * 16;
constexpr int kPOffYT = kPOffX0 + (kPChunks + 1) * 32 * 8;
constexpr int kPOffY0 = kPOffYT + 5 * kPairs * 16;
constexpr int kPOffBar = kPOffY0 + 5 * kPairs * 8;
constexpr int kPatchSmem = kPOffBar + 8 + 1016;  // the base is aligned to 1024

}  // namespace

// Patch `blk` of one grid (REC: with receivers).
template <int H, bool REC>
__device__ __forceinline__ void patch_body(const TileArgs& a, const CUtensorMap* tm_u, const CUtensorMap* tm_m,
                                           int blk, int par, float* u_prev) {
  constexpr int PY = kPR - 2 * H;  // rows of a patch
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sa0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t sa = (sa0 + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (sa - sa0);
  ulonglong2* XT = reinterpret_cast<ulonglong2*>(smem + kPOffXT);
  f2* X0 = reinterpret_cast<f2*>(smem + kPOffX0);
  ulonglong2* YT = reinterpret_cast<ulonglong2*>(smem + kPOffYT);
  f2* Y0 = reinterpret_cast<f2*>(smem + kPOffY0);
  const uint32_t bar = sa + kPOffBar;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int strip = blk % a.strips;
  const int band = blk / a.strips;
  const int r0 = band * PY - H;         // first staged row
  const int c0 = strip * kPX - kPH;     // first staged column

  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  if (tid < 32) {
    XT[tid] = make_ulonglong2(0ull, 0ull);
    X0[kPChunks * 32 + tid] = 0ull;
  }
  if (tid >= 64 && tid < 64 + kPairs) {
    YT[tid - 64] = make_ulonglong2(0ull, 0ull);
    Y0[4 * kPairs + tid - 64] = 0ull;
  }
  __syncthreads();
  Source src;
  src.early(a);
  Sampler rec;
  if (REC && a.n_rec > 0) rec.look(a, c0 + kPH, c0 + kPH + kPX, r0 + H, r0 + H + PY);
  if (tid < 32) {
    if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)((kPCols / 32) * (66 + kPR) * 128));
    __syncwarp();
    if (lane < 4) tma_load_2d(sa + kPOffM + (uint32_t)(lane * kMPanel), tm_m, c0 + 32 * lane, r0, bar);
    chain_wait();
    if (lane < 4) tma_load_2d(sa + (uint32_t)(lane * kUPanel), tm_u, c0 + 32 * lane, r0 - 1, bar);
  } else {
    chain_wait();
  }
  chain_release();

  // x phase: rows xr and xr + 8 of the patch, chunk ch (see adi_tile.cu for
  // the swizzled addresses); row r of the patch is row r + 1 of the u stage
  const int xr = (tid >> 6) * 16 + (tid & 7);
  const int ch = (tid >> 3) & 7;
  const int xs = (tid >> 6) * 8 + (tid & 7);  // slot of the row pair
  auto unit0 = [](int panel, int r, int c) {
    return (uint32_t)((c >> 1) * panel + r * 128 + (((c & 1) * 64) ^ ((r & 7) << 4)));
  };
  const uint32_t pu = sa + unit0(kUPanel, xr, ch), pc = sa + unit0(kUPanel, xr + 1, ch),
                 pd = sa + unit0(kUPanel, xr + 2, ch), pm = sa + kPOffM + unit0(kMPanel, xr, ch);
  const uint32_t pL = ch > 0 ? sa + (unit0(kUPanel, xr + 1, ch - 1) ^ 48u) + 12u : sa;
  const uint32_t pR = ch < kPChunks - 1 ? sa + unit0(kUPanel, xr + 1, ch + 1) : sa;
  const uint32_t ow = sa + kPOffW + unit0(kMPanel, xr, ch - 1);
  const int gx0 = c0 + 16 * ch;
  const float sg = ((xr & 3) == 1 || (xr & 3) == 2) ? -1.f : 1.f;
  const f2 cx2 = dup2(sg * a.cx), cy2 = dup2(sg * a.cy);
  const float scx = a.scx;
  src.late(a, par, blk == 0 && tid == 0);
  const GridDev* gd = a.gd;
  const int sx = src.sx, sy = src.sy;
  const float fsrc = sg * src.f;
  if (REC && a.n_rec > 0) rec.sample(a, gd, src.lev, c0 + kPH, c0 + kPH + kPX, r0 + H, r0 + H + PY);

  // y phase: chunk yc of columns 2 cp, 2 cp + 1; its rows that are the patch's
  const bool ythread = tid < 4 * kPairs;
  const int yc = tid / kPairs, cp = tid - yc * kPairs;
  const int yi = strip * kPX + 2 * cp;
  const bool ok0 = ythread && yi < a.nx, ok1 = ythread && yi + 1 < a.nx;
  const int ylo = max(0, H - 16 * yc), yhi = min(16, min(kPR - H - 16 * yc, a.ny - r0 - 16 * yc));
  const size_t ld = (size_t)a.ld;
  float* const orow = u_prev + ((ptrdiff_t)(r0 + 16 * yc) * (ptrdiff_t)ld + yi);

  bool timed_out = false;
  if (!mbar_wait_bounded(bar, 0u, 1000000000ull)) timed_out = true;
  // ---------------- x phase ----------------
  {
    float d[2][16], s[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      f2 c2[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const ulonglong2 t = lds4((pc ^ (16u * q)) + 1024u * h);
        c2[2 * q] = t.x;
        c2[2 * q + 1] = t.y;
      }
      const float uL = lds(pL + 1024u * h), uR = lds(pR + 1024u * h);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const ulonglong2 t4 = lds4((pu ^ (16u * q)) + 1024u * h);
        const ulonglong2 b4 = lds4((pd ^ (16u * q)) + 1024u * h);
        const ulonglong2 m4 = lds4((pm ^ (16u * q)) + 1024u * h);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = 2 * q + e, k = 2 * j;
          const f2 vs = add2(e ? t4.y : t4.x, e ? b4.y : b4.x);
          const f2 mm = e ? m4.y : m4.x;
          const float l = j > 0 ? hi2(c2[j > 0 ? j - 1 : 0]) : uL;
          const float r = j < 7 ? lo2(c2[j < 7 ? j + 1 : 7]) : uR;
          const f2 lr = pk(l + hi2(c2[j]), lo2(c2[j]) + r);
          const f2 t1 = fma2(dup2(-2.f), c2[j], lr);
          const f2 t2 = fma2(dup2(-2.f), c2[j], vs);
          const f2 lap = fma2(cy2, t2, mul2(cx2, t1));
          d[h][k] = sgn_d(k) * lo2(mm) * lo2(lap);
          d[h][k + 1] = sgn_d(k + 1) * hi2(mm) * hi2(lap);
          s[h][k] = scx * lo2(mm);
          s[h][k + 1] = -scx * hi2(mm);
        }
      }
      if (r0 + xr + 8 * h == sy && sx >= gx0 && sx < gx0 + 16) {
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (gx0 + k == sx) d[h][k] += sgn_d(k) * fsrc;
      }
      // the stage's outermost columns lack a neighbour: zero there, as beyond
      if (ch == 0) { d[h][0] = 0.f; s[h][0] = 0.f; }
      if (ch == kPChunks - 1) { d[h][15] = 0.f; s[h][15] = 0.f; }
    }
    f2 D[16], S[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      D[k] = pk(d[0][k], d[1][k]);
      S[k] = pk(s[0][k], s[1][k]);
    }
    Elim2 e;
    e.begin(0ull, 0ull);
    e.tail<H>(S, D);
    {
      const f2 r = pk(rcp_t(lo2(e.p)), rcp_t(hi2(e.p)));
      XT[(ch + 1) * 32 + xs] = make_ulonglong2(mul2(e.a, r), mul2(e.N, r));
    }
    __syncthreads();
    {
      const ulonglong2 t = XT[ch * 32 + xs];
      e.begin(t.x, t.y);
    }
    e.chunk(S, D);
    f2 X = 0ull;
#pragma unroll
    for (int k = H - 1; k >= 0; --k) X = fma2(S[k], X, D[k]);
    X0[ch * 32 + xs] = X;
    __syncthreads();
    X = X0[(ch + 1) * 32 + xs];
    float xa = -lo2(X), xb = -hi2(X);  // x itself from here on
#pragma unroll
    for (int k = 15; k >= 0; --k) {
      xa = fmaf((k & 1) ? lo2(S[k]) : -lo2(S[k]), xa, -sgn_d(k) * lo2(D[k]));
      xb = fmaf((k & 1) ? hi2(S[k]) : -hi2(S[k]), xb, -sgn_d(k) * hi2(D[k]));
      d[0][k] = xa;
      d[1][k] = xb;
    }
    if (ch >= 1 && ch <= kPChunks - 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(__cvta_shared_to_generic((ow ^ (16u * q)) + 1024u * h)) =
              make_float4(d[h][4 * q], d[h][4 * q + 1], d[h][4 * q + 2], d[h][4 * q + 3]);
    }
  }
  __syncthreads();
  // ---------------- y phase ----------------
  {
    f2 up[16], D[16], S[16];
    auto colbyte = [](int panel, int c) { return (uint32_t)((c >> 5) * panel + ((c & 31) << 2)); };
    const uint32_t row = (uint32_t)(16 * yc * 128);
    const uint32_t ym = sa + kPOffM + row + colbyte(kMPanel, 2 * cp + kPH);
    const uint32_t yw = sa + kPOffW + row + colbyte(kMPanel, 2 * cp);
    const uint32_t yu = sa + row + colbyte(kUPanel, 2 * cp + kPH);
    Elim2 e;
    if (ythread) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        up[i] = 0ull;
        if (i >= ylo && i < yhi) {
          if (ok1) up[i] = __ldcg(reinterpret_cast<const f2*>(orow + i * ld));
          else if (ok0) up[i] = pk(__ldcg(orow + i * ld), 0.f);
        }
      }
      const f2 scy_p = dup2(a.scy), scy_n = dup2(-a.scy);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint32_t key = (uint32_t)((i & 7) << 4);
        S[i] = mul2((i & 1) ? scy_n : scy_p, lds2((ym ^ key) + i * 128));
        D[i] = lds2((yw ^ key) + i * 128);
      }
      e.begin(0ull, 0ull);
      e.tail<H>(S, D);
      const f2 r = pk(rcp_t(lo2(e.p)), rcp_t(hi2(e.p)));
      YT[(yc + 1) * kPairs + cp] = make_ulonglong2(mul2(e.a, r), mul2(e.N, r));
    }
    __syncthreads();
    if (ythread) {
      const ulonglong2 t = YT[yc * kPairs + cp];
      e.begin(t.x, t.y);
      e.chunk(S, D);
      f2 X = 0ull;
#pragma unroll
      for (int k = H - 1; k >= 0; --k) X = fma2(S[k], X, D[k]);
      Y0[yc * kPairs + cp] = X;
      // q = +-(2u^k - u^{k-1})
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const f2 u = lds2((yu ^ (uint32_t)(((i + 1) & 7) << 4)) + (i + 1) * 128);
        if (sgn_d(i) > 0.f) up[i] = pk(fmaf(2.f, lo2(u), -lo2(up[i])), fmaf(2.f, hi2(u), -hi2(up[i])));
        else up[i] = fma2(dup2(-2.f), u, up[i]);
      }
    }
    __syncthreads();
    f2 chk = 0ull;
    if (ythread) {
      f2 X = Y0[(yc + 1) * kPairs + cp];
#pragma unroll
      for (int i = 15; i >= 0; --i) {
        X = fma2(S[i], X, D[i]);
        if (i >= ylo && i < yhi) {
          const f2 un = updated(i, up[i], X);
          float* o = orow + i * ld;
          if (ok1) *reinterpret_cast<f2*>(o) = un;
          else if (ok0) o[0] = lo2(un);
          if (ok0) chk = fma2(un, 0ull, chk);
        }
      }
    }
    const bool bad = lo2(chk) != 0.f || (ok1 && hi2(chk) != 0.f);
    if (__any_sync(0xffffffffu, bad) && lane == 0 && a.err) atomicOr(a.err, ERR_NUMERIC);
    if (timed_out && lane == 0 && a.err) atomicOr(a.err, ERR_TIMEOUT);
  }
}

template <int H>
__global__ void __launch_bounds__(kPN, 2)
    patch_step_kernel(const TileArgs a, const __grid_constant__ CUtensorMap tm_u,
                      const __grid_constant__ CUtensorMap tm_m) {
  patch_body<H, true>(a, &tm_u, &tm_m, blockIdx.x, a.par, a.u_prev);
}

// A step of many grids: items[b] = (grid, patch) of CTA b.
template <int H>
__global__ void __launch_bounds__(kPN, 2)
    patch_batch_kernel(const BatchTile* __restrict__ tiles, const int2* __restrict__ items, int par) {
  const int2 it = __ldg(items + blockIdx.x);
  const BatchTile& t = tiles[it.x];
  if (threadIdx.x < 32) {  // the warp that issues the tensor copies
    tensormap_acquire(&t.u[par]);
    tensormap_acquire(&t.m);
  }
  const TileArgs a = t.a;
  patch_body<H, false>(a, &t.u[par], &t.m, it.y, par, t.buf[par ^ 1]);
}

// ---------------------------------------------------------------------------
// Small patches: 64 x 64 staged points, 32 columns of its own, one row or
// column per thread in scalar arithmetic.  On a grid of few patches the time
// of a step is that of one patch (its two phases, about 3.6 us above, where
// two warps per scheduler share the issue slots), and here each thread has
// half the work and an SM half the points: 128^2 3.4 against 6.1 us per step,
// 512^2 4.5 against 6.1 (2.7 and 3.7 since the launch carries level and
// source by value).  The operations on an unknown and the chunks are
// the same, so with H = 12 the results are too, bit for bit (H = 16 reaches
// the stage's outermost column, which the two kinds cut elsewhere).  Taken
// while two per SM hold the grid: 640 x 600 (300 patches) 4.6 against 6.3,
// 700^2 (396) 7.9 against 7.0.
// ---------------------------------------------------------------------------
namespace {

constexpr int kSX = 32;                 // columns of a small patch
constexpr int kSChunks = (kSX + 2 * kPH) / 16;
// shared memory: u | m | w | XT[5][64] 8 B | X0[5][64] 4 B | YT[5][32] 8 B | Y0[5][32] 4 B | mbarrier
constexpr int kSOffM = 2 * kUPanel;
constexpr int kSOffW = kSOffM + 2 * kMPanel;
constexpr int kSOffXT = kSOffW + kMPanel;
constexpr int kSOffX0 = kSOffXT + (kSChunks + 1) * kPR * 8;
constexpr int kSOffYT = kSOffX0 + (kSChunks + 1) * kPR * 4;
constexpr int kSOffY0 = kSOffYT + 5 * kSX * 8;
constexpr int kSOffBar = kSOffY0 + 5 * kSX * 4;
constexpr int kSmallSmem = kSOffBar + 8 + 1016;  // the base is aligned to 1024

__device__ __forceinline__ float4 lds4f(uint32_t a) {
  return *reinterpret_cast<const float4*>(__cvta_shared_to_generic(a));
}

}  // namespace

template <int H>
__global__ void __launch_bounds__(kPN, 2)
    small_patch_kernel(const TileArgs a, const __grid_constant__ CUtensorMap tm_u,
                       const __grid_constant__ CUtensorMap tm_m) {
  constexpr int PY = kPR - 2 * H;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sa0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t sa = (sa0 + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (sa - sa0);
  float2* XT = reinterpret_cast<float2*>(smem + kSOffXT);
  float* X0 = reinterpret_cast<float*>(smem + kSOffX0);
  float2* YT = reinterpret_cast<float2*>(smem + kSOffYT);
  float* Y0 = reinterpret_cast<float*>(smem + kSOffY0);
  const uint32_t bar = sa + kSOffBar;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int strip = blockIdx.x % a.strips;
  const int band = blockIdx.x / a.strips;
  const int r0 = band * PY - H;
  const int c0 = strip * kSX - kPH;

  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  if (tid < kPR) {
    XT[tid] = make_float2(0.f, 0.f);
    X0[kSChunks * kPR + tid] = 0.f;
  } else if (tid < kPR + kSX) {
    YT[tid - kPR] = make_float2(0.f, 0.f);
    Y0[4 * kSX + tid - kPR] = 0.f;
  }
  __syncthreads();
  Source src;
  src.early(a);
  Sampler rec;
  if (a.n_rec > 0) rec.look(a, c0 + kPH, c0 + kPH + kSX, r0 + H, r0 + H + PY);
  if (tid < 32) {
    if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)(2 * (66 + kPR) * 128));
    __syncwarp();
    if (lane < 2) tma_load_2d(sa + kSOffM + (uint32_t)(lane * kMPanel), &tm_m, c0 + 32 * lane, r0, bar);
    chain_wait();
    if (lane < 2) tma_load_2d(sa + (uint32_t)(lane * kUPanel), &tm_u, c0 + 32 * lane, r0 - 1, bar);
  } else {
    chain_wait();
  }
  chain_release();

  // x phase: row xr of the patch, chunk ch
  const int xr = (tid >> 6) * 16 + (tid & 15);
  const int ch = (tid >> 4) & 3;
  auto unit0 = [](int panel, int r, int c) {
    return (uint32_t)((c >> 1) * panel + r * 128 + (((c & 1) * 64) ^ ((r & 7) << 4)));
  };
  const uint32_t pu = sa + unit0(kUPanel, xr, ch), pc = sa + unit0(kUPanel, xr + 1, ch),
                 pd = sa + unit0(kUPanel, xr + 2, ch), pm = sa + kSOffM + unit0(kMPanel, xr, ch);
  const uint32_t pL = ch > 0 ? sa + (unit0(kUPanel, xr + 1, ch - 1) ^ 48u) + 12u : sa;
  const uint32_t pR = ch < kSChunks - 1 ? sa + unit0(kUPanel, xr + 1, ch + 1) : sa;
  const uint32_t ow = sa + kSOffW + unit0(kMPanel, xr, ch - 1);
  const int gx0 = c0 + 16 * ch;
  const float cx = a.cx, cy = a.cy, scx = a.scx, scy = a.scy;
  src.late(a, a.par, blockIdx.x == 0 && tid == 0);
  const GridDev* gd = a.gd;
  const int sx = src.sx, sy = src.sy;
  const float fsrc = src.f;
  if (a.n_rec > 0) rec.sample(a, gd, src.lev, c0 + kPH, c0 + kPH + kSX, r0 + H, r0 + H + PY);

  // y phase: chunk yc (a warp) of column `lane`; its rows that are the patch's
  const int yc = tid >> 5;
  const bool ythread = tid < 4 * kSX;
  const int yi = strip * kSX + lane;
  const bool ok = ythread && yi < a.nx;
  const int ylo = max(0, H - 16 * yc), yhi = min(16, min(kPR - H - 16 * yc, a.ny - r0 - 16 * yc));
  const size_t ld = (size_t)a.ld;
  float* const orow = a.u_prev + ((ptrdiff_t)(r0 + 16 * yc) * (ptrdiff_t)ld + yi);

  bool timed_out = false;
  if (!mbar_wait_bounded(bar, 0u, 1000000000ull)) timed_out = true;
  // ---------------- x phase ----------------
  {
    float D[16], S[16], c[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = lds4f(pc ^ (16u * q));
      c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
    }
    const float uL = lds(pL), uR = lds(pR);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 t4 = lds4f(pu ^ (16u * q)), b4 = lds4f(pd ^ (16u * q)), m4 = lds4f(pm ^ (16u * q));
      const float vs[4] = {t4.x + b4.x, t4.y + b4.y, t4.z + b4.z, t4.w + b4.w};
      const float mv[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 4 * q + e;
        const float l = k > 0 ? c[k > 0 ? k - 1 : 0] : uL;
        const float r = k < 15 ? c[k < 15 ? k + 1 : 15] : uR;
        const float t1 = fmaf(-2.f, c[k], l + r), t2 = fmaf(-2.f, c[k], vs[e]);
        D[k] = mv[e] * fmaf(cy, t2, cx * t1);
        S[k] = scx * mv[e];
      }
    }
    if (r0 + xr == sy && sx >= gx0 && sx < gx0 + 16) {
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (gx0 + k == sx) D[k] += fsrc;
    }
    // the stage's outermost columns lack a neighbour: zero there, as beyond
    if (ch == 0) { D[0] = 0.f; S[0] = 0.f; }
    if (ch == kSChunks - 1) { D[15] = 0.f; S[15] = 0.f; }
    Elim1 e;
    e.begin(0.f, 0.f);
    e.tail<H>(S, D);
    {
      const float r = rcp_t(e.p);
      XT[(ch + 1) * kPR + xr] = make_float2(e.a * r, e.N * r);
    }
    __syncthreads();
    {
      const float2 t = XT[ch * kPR + xr];
      e.begin(t.x, t.y);
    }
    e.chunk(S, D);
    float x = 0.f;
#pragma unroll
    for (int k = H - 1; k >= 0; --k) x = fmaf(S[k], x, D[k]);
    X0[ch * kPR + xr] = x;
    __syncthreads();
    x = X0[(ch + 1) * kPR + xr];
#pragma unroll
    for (int k = 15; k >= 0; --k) {
      x = fmaf(S[k], x, D[k]);
      D[k] = x;
    }
    if (ch >= 1 && ch <= kSChunks - 2) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(__cvta_shared_to_generic(ow ^ (16u * q))) =
            make_float4(D[4 * q], D[4 * q + 1], D[4 * q + 2], D[4 * q + 3]);
    }
  }
  __syncthreads();
  // ---------------- y phase ----------------
  float up[16], D[16], S[16];
  Elim1 e;
  if (ythread) {
    const uint32_t row = (uint32_t)(16 * yc * 128);
    const uint32_t ym = sa + kSOffM + row + (uint32_t)(((lane + kPH) >> 5) * kMPanel + (((lane + kPH) & 31) << 2));
    const uint32_t yw = sa + kSOffW + row + (uint32_t)(lane << 2);
#pragma unroll
    for (int i = 0; i < 16; ++i) up[i] = ok && i >= ylo && i < yhi ? __ldcg(orow + i * ld) : 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t key = (uint32_t)((i & 7) << 4);
      S[i] = scy * lds((ym ^ key) + i * 128);
      D[i] = lds((yw ^ key) + i * 128);
    }
    e.begin(0.f, 0.f);
    e.tail<H>(S, D);
    const float r = rcp_t(e.p);
    YT[(yc + 1) * kSX + lane] = make_float2(e.a * r, e.N * r);
  }
  __syncthreads();
  if (ythread) {
    const float2 t = YT[yc * kSX + lane];
    e.begin(t.x, t.y);
    e.chunk(S, D);
    float x = 0.f;
#pragma unroll
    for (int k = H - 1; k >= 0; --k) x = fmaf(S[k], x, D[k]);
    Y0[yc * kSX + lane] = x;
    const uint32_t yu = sa + (uint32_t)(16 * yc * 128) +
                        (uint32_t)(((lane + kPH) >> 5) * kUPanel + (((lane + kPH) & 31) << 2));
#pragma unroll
    for (int i = 0; i < 16; ++i)
      up[i] = fmaf(2.f, lds((yu ^ (uint32_t)(((i + 1) & 7) << 4)) + (i + 1) * 128), -up[i]);
  }
  __syncthreads();
  float chk = 0.f;
  if (ythread) {
    float x = Y0[(yc + 1) * kSX + lane];
#pragma unroll
    for (int i = 15; i >= 0; --i) {
      x = fmaf(S[i], x, D[i]);
      if (ok && i >= ylo && i < yhi) {
        const float un = up[i] + x;
        orow[i * ld] = un;
        chk = fmaf(un, 0.f, chk);
      }
    }
  }
  if (__any_sync(0xffffffffu, chk != 0.f) && lane == 0 && a.err) atomicOr(a.err, ERR_NUMERIC);
  if (timed_out && lane == 0 && a.err) atomicOr(a.err, ERR_TIMEOUT);
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
int patch_rows(int H) { return kPR - 2 * H; }
int patch_threads() { return kPN; }
int patch_strips(int nx) { return (nx + kPX - 1) / kPX; }
int small_patch_strips(int nx) { return (nx + kSX - 1) / kSX; }

cudaError_t encode_patch_map(CUtensorMap* out, const float* base, int nx, int ld, int ny, bool u) {
  return encode_box_map(out, base, nx, ld, ny, 32, u ? kPR + 2 : kPR, true);
}

cudaError_t launch_patch(const TileArgs& a_in, int H, const CUtensorMap& u, const CUtensorMap& m, cudaStream_t st) {
  TileArgs a = a_in;
  if (H != 12 && H != 16) return cudaErrorInvalidValue;
  const int bands = (a.ny + patch_rows(H) - 1) / patch_rows(H);
  if (a.small) {
    a.strips = small_patch_strips(a.nx);
    return launch_after(!a.alone, H == 12 ? small_patch_kernel<12> : small_patch_kernel<16>, a.strips * bands, kPN, kSmallSmem,
                          st, a, u, m);
  }
  a.strips = patch_strips(a.nx);
  return launch_after(!a.alone, H == 12 ? patch_step_kernel<12> : patch_step_kernel<16>, a.strips * bands, kPN, kPatchSmem, st,
                        a, u, m);
}

cudaError_t launch_patch_batch(const BatchTile* tiles, const int2* items, int n_items, int par, int H,
                               cudaStream_t st) {
  return launch_chained(H == 12 ? patch_batch_kernel<12> : patch_batch_kernel<16>, n_items, kPN, kPatchSmem, st,
                        tiles, items, par);
}

cudaError_t configure_patch_kernels() {
  cudaError_t e = cudaSuccess;
#define ADI_PATCH_CFG(K) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, kPatchSmem);
  ADI_PATCH_CFG(patch_step_kernel<12>)
  ADI_PATCH_CFG(patch_step_kernel<16>)
  ADI_PATCH_CFG(patch_batch_kernel<12>)
  ADI_PATCH_CFG(patch_batch_kernel<16>)
#undef ADI_PATCH_CFG
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(small_patch_kernel<12>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(small_patch_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
  return e;
}

}  // namespace adi
