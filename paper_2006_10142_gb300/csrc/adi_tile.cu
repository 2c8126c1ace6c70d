// adi_tile.cu -- one whole time step of the factored scheme in one pass over
// the fields: RHS assembly, row solves, column solves and update.
//
// The systems of a step, -s_{i} x_{i-1} + (1 + 2 s_i) x_i - s_i x_{i+1} = d_i,
// are strictly diagonally dominant, and the elimination x_i = delta_i +
// gamma_i x_{i+1} has 0 <= gamma_i <= lambda(s_max) with
//     lambda(s) = (1 + 2s - sqrt(1 + 4s)) / (2s)
// (gamma_i grows with s_i and gamma_{i-1}, and lambda is its fixed point), so
// a value H unknowns away enters with a factor of at most lambda^H.  At
// tau = 0.5 h / max c lambda is 0.101: across 12 unknowns 1e-12.  Where
// lambda^H is below 2^-30 -- a fraction of a unit in the last place of the
// FP32 result -- both sweeps are solved locally: an elimination that starts
// H unknowns before the part it is for, with a zero value in front, gives
// that part's unknowns as the elimination of the whole line does, and a
// back substitution that starts H unknowns behind it likewise.  No interface
// systems, no exchange between CTAs, and w never leaves the SM: a step reads
// u^k, m and u^{k-1} once and writes u^{k+1} (16 B per point and one launch,
// against 32 B and two launches for the separate sweeps).  Weakly dominant
// systems keep the separate sweeps (tile_halo() decides).
//
// A CTA owns a strip of TX = 224 columns and a band of rows.  It stages 256
// columns (16 of halo on either side) and marches down the band in blocks of
// 16 rows:
//   x phase: 16 rows x 16 chunks of 16 unknowns over 128 threads, a chunk of
//     rows r and r + 8 per thread in packed arithmetic (lanes along the rows,
//     so that the 128-byte-swizzled stage is read without bank conflicts).
//     Each thread eliminates the last H unknowns of its chunk from zero, hands
//     (gamma, delta) to the next chunk through shared memory, eliminates its
//     chunk from the exact state it was handed, back-substitutes the first H
//     unknowns from zero, hands x_0 to the previous chunk and back-substitutes
//     the chunk.  The outermost column on either side lacks a neighbour for
//     its RHS and is set to zero: it lies 16 from the strip's own columns, so
//     that with H = 16 too no factor above lambda^16 is left out.
//   y phase: two columns per thread (112 threads, the strip's own columns):
//     the elimination of a column runs on from block to block in registers;
//     after each block the back substitution starts from its last row and
//     yields the 16 rows that lie H behind.  Whole blocks leave by TMA, the
//     rows of a band's edge one by one.
// Blocks of u^k (three slots, shifted by one row so that a block carries its
// lower neighbour row) and m (two) arrive by TMA two blocks ahead, u^{k-1} one
// block ahead from L2, into which it is prefetched with them.  Rows and columns outside the grid arrive as
// zeros with s = 0, which is the Dirichlet ring.  Bands start H rows early
// and end H rows late (the halo of the column solves), and their rows are
// chosen so that halo and all fill whole blocks (3001 x 1501: 21 bands of 72
// rows in 6 blocks instead of 19 of 80 in 7).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "adi_bodies.cuh"
#include "adi_device.cuh"
#include "adi_internal.h"
#include "adi_local.cuh"
#include "adi_sweeps.cuh"
#include "adi_tile_stage.h"
#include "adi_tma.cuh"

namespace adi {

namespace {

constexpr int kOut = (kTX / 32) * kPanel;   // bytes of a block of the strip's own columns
// shared memory: u slots 0..2 | m slots 0..1 | w, then the block's u^{k+1} |
// u^{k-1} [16][224] | XT[17][8] float4 | X0[17][8] float2 | 3 mbarriers
constexpr int kOffM = kUSlots * kSlot;
constexpr int kOffW = kOffM + 2 * kSlot;
constexpr int kOffP = kOffW + kOut;
constexpr int kOffXT = kOffP + kOut;
constexpr int kOffX0 = kOffXT + 17 * 8 * 16;
constexpr int kOffBar = kOffX0 + 17 * 8 * 8;
constexpr int kTileSmem = kOffBar + 24 + 1000;  // the base is aligned to 1024

// One block of two columns: X_i = G_i X_{i+1} + D_i, and q = +-(2u^k -
// u^{k-1}), negative where sigma is.
struct Col {
  f2 g[kTB], d[kTB], q[kTB];
};

}  // namespace

// CTA `blk` of one grid (REC: with receivers).
template <int H, bool REC>
__device__ __forceinline__ void tile_body(const TileArgs& a, const CUtensorMap* tm_u, const CUtensorMap* tm_m,
                                          const CUtensorMap* tm_p, const CUtensorMap* tm_o, int blk, int par, float* u_prev) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sa0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t sa = (sa0 + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (sa - sa0);
  ulonglong2* XT = reinterpret_cast<ulonglong2*>(smem + kOffXT);
  f2* X0 = reinterpret_cast<f2*>(smem + kOffX0);
  const uint32_t bar = sa + kOffBar;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int strip = blk % a.strips;
  const int band = blk / a.strips;
  const int y0 = band * a.band_rows;
  const int y1 = min(a.ny, y0 + a.band_rows);
  const int rs = max(0, y0 - H);                   // first row processed
  const int re = min(a.ny, y1 + H);                // rows at and beyond re are not needed
  const int nblk = (re - rs + kTB - 1) / kTB;
  const int c0 = strip * kTX - kTH;                // first staged column

  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 8u, 1);
    mbar_init(bar + 16u, 1);
    mbar_fence_init();
  }
  if (tid < 8) {
    XT[tid] = make_ulonglong2(0ull, 0ull);
    X0[16 * 8 + tid] = 0ull;
  }
  __syncthreads();

  // warp 0: block b of u^k (rows rs + 16 b + 1 ..) and m, a 32-column panel
  // per lane, and an L2 prefetch of its u^{k-1}
  auto issue = [&](int b) {
    const uint32_t mb = bar + 8u * (uint32_t)(b & 1);
    if (lane == 0) mbar_arrive_expect_tx(mb, (uint32_t)(b == 0 ? 3 * kSlot : 2 * kSlot));
    __syncwarp();
    const int p = lane & 7, f = lane >> 3;
    const int col = c0 + 32 * p, row = rs + kTB * b;
    if (f == 0) {
      tma_load_2d(sa + (uint32_t)((b % 3) * kSlot + p * kPanel), tm_u, col, row + 1, mb);
      if (b == 0) tma_load_2d(sa + (uint32_t)(2 * kSlot + p * kPanel), tm_u, col, row + 1 - kTB, mb);
    } else if (f == 1) {
      tma_load_2d(sa + (uint32_t)(kOffM + (b & 1) * kSlot + p * kPanel), tm_m, col, row, mb);
    } else if (lane == 16) {
      tma_prefetch_2d(tm_p, strip * kTX, row);
    }
  };
  // one thread: block b of u^{k-1}, the strip's own columns
  auto issue_prev = [&](int b) {
    mbar_arrive_expect_tx(bar + 16u, (uint32_t)kOut);
    tma_load_2d(sa + (uint32_t)kOffP, tm_p, strip * kTX, rs + kTB * b, bar + 16u);
  };
  Source src;
  src.early(a);
  Sampler rec;
  if (REC && a.n_rec > 0) rec.look(a, strip * kTX, strip * kTX + kTX, y0, y1);
  chain_wait();
  chain_release();
  if (tid < 32) {
    issue(0);
    if (lane == 0) issue_prev(0);
    if (nblk > 1) issue(1);
  }

  // x phase: rows xr and xr + 8 of the block, chunk ch (offsets: adi_tile_stage.h)
  const int xr = tid & 7;
  const int ch = tid >> 3;
  const TileRow at = tile_row(xr, ch);
  const uint32_t ow = sa + kOffW + tile_unit(xr, ch - 1);  // w holds the strip's own columns
  const int gx0 = c0 + 16 * ch;                        // column of the chunk's first unknown
  // w is wanted as sigma w by the column solves (rows xr and xr + 8 have the same sigma)
  const float sg = ((xr & 3) == 1 || (xr & 3) == 2) ? -1.f : 1.f;
  const f2 cx2 = dup2(sg * a.cx), cy2 = dup2(sg * a.cy);
  const float scx = a.scx;
  src.late(a, par, blk == 0 && tid == 0);
  const int sx = src.sx, sy = src.sy;
  const float fsrc = sg * src.f;
  if (REC && a.n_rec > 0) rec.sample(a, a.gd, src.lev, strip * kTX, strip * kTX + kTX, y0, y1);

  // y phase: columns 2 tid, 2 tid + 1 of the strip, 16 columns into the stage
  const bool ywarp = tid < kTX / 2;
  const int yi = strip * kTX + 2 * tid;
  const bool ok0 = ywarp && yi < a.nx, ok1 = ywarp && yi + 1 < a.nx;
  auto colbyte = [](int c) { return (uint32_t)((c >> 5) * kPanel + ((c & 31) << 2)); };
  const uint32_t ym = colbyte(2 * tid + kTH);
  const uint32_t yw = sa + kOffW + colbyte(2 * tid);
  const uint32_t yp = sa + kOffP + 8u * (uint32_t)tid;
  const size_t ld = (size_t)a.ld;
  const f2 scy_p = dup2(a.scy), scy_n = dup2(-a.scy);

  f2 chk = 0ull;
  bool timed_out = false;

  // one row of a band edge (a block whose rows leave one by one)
  auto store_row = [&](int i, int j, f2 q, f2 X) {
    if (j < y0 || j >= y1) return;
    const f2 un = updated(i, q, X);
    float* o = u_prev + (size_t)j * ld + yi;
    if (ok0) o[0] = lo2(un);
    if (ok1) o[1] = hi2(un);
    if (ok0) chk = fma2(un, 0ull, chk);
  };

  auto block = [&](int n, Col& P, Col& C) {
    if (!mbar_wait_bounded(bar + 8u * (uint32_t)(n & 1), (uint32_t)(n >> 1) & 1u, 1000000000ull)) timed_out = true;
    const uint32_t Ucur = sa + (uint32_t)((n % 3) * kSlot);
    const uint32_t Uprev = sa + (uint32_t)(((n + 2) % 3) * kSlot);
    const uint32_t Mb = sa + kOffM + (uint32_t)((n & 1) * kSlot);
    const int row0 = rs + kTB * n;
    // ---------------- x phase ----------------
    {
      float d[2][16], s[2][16];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // bases of the slots that hold rows r (centre) and r - 1 (above)
        const uint32_t bc = tile_row_base(Ucur, Uprev, xr, h, 0);
        const uint32_t bu = tile_row_base(Ucur, Uprev, xr, h, 1);
        const uint32_t pc = bc + at.centre, pu = bu + at.above;
        const uint32_t pd = Ucur + at.below, pm = Mb + at.below;
        f2 c2[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const ulonglong2 t = lds4(pc ^ (16u * q));
          c2[2 * q] = t.x;
          c2[2 * q + 1] = t.y;
        }
        const float uL = lds(bc + at.left), uR = lds(bc + at.right);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const ulonglong2 t4 = lds4(pu ^ (16u * q));
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
        if (row0 + xr + 8 * h == sy && sx >= gx0 && sx < gx0 + 16) {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (gx0 + k == sx) d[h][k] += sgn_d(k) * fsrc;
        }
        // the stage's outermost columns lack a neighbour: zero there, as beyond
        if (ch == 0) { d[h][0] = 0.f; s[h][0] = 0.f; }
        if (ch == 15) { d[h][15] = 0.f; s[h][15] = 0.f; }
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
        XT[(ch + 1) * 8 + xr] = make_ulonglong2(mul2(e.a, r), mul2(e.N, r));
      }
      __syncthreads();
      {
        const ulonglong2 t = XT[ch * 8 + xr];
        e.begin(t.x, t.y);
      }
      e.chunk(S, D);
      f2 X = 0ull;
#pragma unroll
      for (int k = H - 1; k >= 0; --k) X = fma2(S[k], X, D[k]);
      X0[ch * 8 + xr] = X;
      if (tid < 32) bulk_wait_read();  // the last block's u^{k+1} has left the w area
      __syncthreads();
      X = X0[(ch + 1) * 8 + xr];
      float xa = -lo2(X), xb = -hi2(X);  // x itself from here on
#pragma unroll
      for (int k = 15; k >= 0; --k) {
        xa = fmaf((k & 1) ? lo2(S[k]) : -lo2(S[k]), xa, -sgn_d(k) * lo2(D[k]));
        xb = fmaf((k & 1) ? hi2(S[k]) : -hi2(S[k]), xb, -sgn_d(k) * hi2(D[k]));
        d[0][k] = xa;
        d[1][k] = xb;
      }
      if (ch >= 1 && ch <= 14) {
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
    // the 16 rows that end H rows before the block's end leave by TMA when
    // all of them are the band's
    const int r0 = row0 - H;
    const bool full = r0 >= y0 && r0 + kTB <= y1;
    if (ywarp) {
      const uint32_t pm = Mb + ym;
      Elim2 e;
      {
        const f2 g = P.g[kTB - 1], dl = P.d[kTB - 1];  // = -(a, N) / p
        e.begin(pk(-lo2(g), -hi2(g)), pk(-lo2(dl), -hi2(dl)));
      }
#pragma unroll
      for (int i = 0; i < kTB; ++i) {
        const uint32_t key = (uint32_t)((i & 7) << 4);
        const f2 s = mul2((i & 1) ? scy_n : scy_p, lds2((pm ^ key) + i * 128));
        const f2 w = lds2((yw ^ key) + i * 128);
        if (i & 1) e.add<1>(s, w);
        else e.add<0>(s, w);
        e.solve(C.g[i], C.d[i]);
      }
      if (!mbar_wait_bounded(bar + 16u, (uint32_t)n & 1u, 1000000000ull)) timed_out = true;
#pragma unroll
      for (int i = 0; i < kTB; ++i) {
        const int idx = (i + 15) & 15;  // row row0 + i of u^k: index i - 1 of its block
        const f2 u = lds2((((i >= 1 ? Ucur : Uprev) + ym) ^ (uint32_t)((idx & 7) << 4)) + idx * 128);
        const f2 up = lds2(yp + i * (kTX * 4));
        if (sgn_d(i) > 0.f) C.q[i] = pk(fmaf(2.f, lo2(u), -lo2(up)), fmaf(2.f, hi2(u), -hi2(up)));
        else C.q[i] = fma2(dup2(-2.f), u, up);
      }
      f2 X = 0ull;
#pragma unroll
      for (int i = kTB - 1; i >= kTB - H; --i) X = fma2(C.g[i], X, C.d[i]);
      if (full) {
#pragma unroll
        for (int e2 = kTB - 1; e2 >= 0; --e2) {
          const bool cur = e2 >= H;
          const int i = cur ? e2 - H : e2 + kTB - H;
          X = fma2(cur ? C.g[i] : P.g[i], X, cur ? C.d[i] : P.d[i]);
          const f2 un = updated(i, cur ? C.q[i] : P.q[i], X);
          *reinterpret_cast<f2*>(__cvta_shared_to_generic((yw ^ (uint32_t)((e2 & 7) << 4)) + e2 * 128)) = un;
          chk = fma2(un, 0ull, chk);
        }
      } else {
#pragma unroll
        for (int e2 = kTB - 1; e2 >= 0; --e2) {
          const bool cur = e2 >= H;
          const int i = cur ? e2 - H : e2 + kTB - H;
          X = fma2(cur ? C.g[i] : P.g[i], X, cur ? C.d[i] : P.d[i]);
          store_row(i, r0 + e2, cur ? C.q[i] : P.q[i], X);
        }
      }
      fence_proxy_async_smem();
    }
    __syncthreads();  // the block's stage is consumed, its u^{k+1} in place
    if (tid < 32) {
      if (full) {
        const int col = strip * kTX + 32 * lane;
        if (lane < kTX / 32 && col < a.nx) tma_store_2d(tm_o, col, r0, sa + kOffW + (uint32_t)(lane * kPanel));
        bulk_commit();
      }
      fence_proxy_async_smem();
      if (lane == 0 && n + 1 < nblk) issue_prev(n + 1);
      if (n + 2 < nblk) issue(n + 2);
    }
  };
  // the rows still pending after the last block: only the band at the end of
  // the grid has any of its own (x = 0 beyond the grid)
  auto flush = [&](int n, const Col& C) {
    if (!ywarp) return;
    f2 X = 0ull;
#pragma unroll
    for (int i = kTB - 1; i >= kTB - H; --i) {
      X = fma2(C.g[i], X, C.d[i]);
      store_row(i, rs + kTB * n + i, C.q[i], X);
    }
  };

  Col A, B;
#pragma unroll
  for (int i = 0; i < kTB; ++i) {
    A.g[i] = A.d[i] = A.q[i] = 0ull;
    B.g[i] = B.d[i] = B.q[i] = 0ull;
  }
  int n = 0;
  for (; n + 1 < nblk; n += 2) {
    block(n, A, B);
    block(n + 1, B, A);
  }
  if (n < nblk) {
    block(n, A, B);
    flush(n, B);
  } else if (n > 0) {
    flush(n - 1, A);
  }
  if (tid < 32) bulk_wait_all();
  const bool bad = lo2(chk) != 0.f || hi2(chk) != 0.f;
  if (__any_sync(0xffffffffu, bad) && lane == 0 && a.err) atomicOr(a.err, ERR_NUMERIC);
  if (timed_out && lane == 0 && a.err) atomicOr(a.err, ERR_TIMEOUT);
}

template <int H>
__global__ void __launch_bounds__(kTN, 2)
    tile_step_kernel(const TileArgs a, const __grid_constant__ CUtensorMap tm_u,
                     const __grid_constant__ CUtensorMap tm_m, const __grid_constant__ CUtensorMap tm_p,
                     const __grid_constant__ CUtensorMap tm_o) {
  tile_body<H, true>(a, &tm_u, &tm_m, &tm_p, &tm_o, blockIdx.x, a.par, a.u_prev);
}

// A step of many grids: items[b] = (grid, CTA of that grid) of CTA b.
template <int H>
__global__ void __launch_bounds__(kTN, 2)
    tile_batch_kernel(const BatchTile* __restrict__ tiles, const int2* __restrict__ items, int par) {
  const int2 it = __ldg(items + blockIdx.x);
  const BatchTile& t = tiles[it.x];
  if (threadIdx.x < 32) {  // the warp that issues the tensor copies
    tensormap_acquire(&t.u[par]);
    tensormap_acquire(&t.m);
    tensormap_acquire(&t.p[par ^ 1]);
    tensormap_acquire(&t.u[par ^ 1]);
  }
  const TileArgs a = t.a;
  tile_body<H, false>(a, &t.u[par], &t.m, &t.p[par ^ 1], &t.u[par ^ 1], it.y, par, t.buf[par ^ 1]);
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------

int tile_halo(double s_max) {
  if (!(s_max > 0) || !std::isfinite(s_max)) return 0;
  const double lam = (1.0 + 2.0 * s_max - std::sqrt(1.0 + 4.0 * s_max)) / (2.0 * s_max);
  const double eps = std::ldexp(1.0, -30);
  if (std::pow(lam, 12) <= eps) return 12;
  if (std::pow(lam, 16) <= eps) return 16;
  return 0;
}

int tile_threads() { return kTN; }
int tile_strips(int nx) { return (nx + kTX - 1) / kTX; }

// Bands or patches (of 96 columns), and the rows of a band.  Times in us as measured on 152
// SMs: a block of a band takes 2.2 alone on its SM and 3.05 beside a second
// CTA (4096^2 to 16384^2), a wave of two patches per SM 6.3 (7.5 for one
// wave at 1024^2, 14.1 for two at 1500^2, 25.9 for four at 2048^2, where
// bands take 17.6, 22.8 and 33.0); from about 4 million points up the bands'
// smaller halo wins (3000^2: 37 against 58, 4096^2: 58 against 102).
int tile_band_rows(int nx, int ny, int H, int nsm) {
  const int strips = tile_strips(nx);
  double best = 0;
  int best_rows = 0;
  // bands of as many rows as fill nb blocks with their halo of 2H rows
  for (int nb = 2 * H / kTB + 1;; ++nb) {
    const bool whole = nb * kTB >= ny;
    const int rows = whole ? (ny + kTB - 1) / kTB * kTB : nb * kTB - 2 * H;
    const long long ctas = (long long)strips * ((ny + rows - 1) / rows);
    const long long per_sm = (ctas + nsm - 1) / nsm;
    const double t = 3.5 + (per_sm <= 1 ? 2.2 : 3.05 * (double)((per_sm + 1) / 2)) * std::min(nb, (ny + kTB - 1) / kTB);
    if (best == 0 || t < best) {
      best = t;
      best_rows = rows;
    }
    if (whole) break;
  }
  const long long patches = (long long)patch_strips(nx) * ((ny + patch_rows(H) - 1) / patch_rows(H));
  const double tp = 1.2 + 6.3 * (double)((patches + 2 * nsm - 1) / (2 * nsm));
  return nx < kTX || tp < best ? 0 : best_rows;
}

// Tensor maps of a pitched [ny][ld] FP32 field of nx columns, zeros outside
// (the padding columns too: they are neither read nor written): boxes of 32
// columns x 16 rows with 128-byte swizzle (u^k, m, and the stores of
// u^{k+1}), or of a strip's 224 columns x 16 rows (u^{k-1}).
cudaError_t encode_tile_map(CUtensorMap* out, const float* base, int nx, int ld, int ny, bool strip) {
  return encode_box_map(out, base, nx, ld, ny, strip ? kTX : 32, kTB, !strip);
}

cudaError_t launch_tile(const TileArgs& a_in, int H, const TileMaps& mp, cudaStream_t st) {
  TileArgs a = a_in;
  a.strips = tile_strips(a.nx);
  if (a.band_rows < 1 || (H != 12 && H != 16)) return cudaErrorInvalidValue;
  const int bands = (a.ny + a.band_rows - 1) / a.band_rows;
  return launch_after(!a.alone, H == 12 ? tile_step_kernel<12> : tile_step_kernel<16>, a.strips * bands, kTN, kTileSmem, st,
                        a, mp.u, mp.m, mp.p, mp.o);
}

cudaError_t launch_tile_batch(const BatchTile* tiles, const int2* items, int n_items, int par, int H,
                              cudaStream_t st) {
  return launch_chained(H == 12 ? tile_batch_kernel<12> : tile_batch_kernel<16>, n_items, kTN, kTileSmem, st, tiles,
                        items, par);
}

cudaError_t configure_tile_kernels() {
  cudaError_t e = cudaSuccess;
#define ADI_TILE_CFG(K) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem);
  ADI_TILE_CFG(tile_step_kernel<12>)
  ADI_TILE_CFG(tile_step_kernel<16>)
  ADI_TILE_CFG(tile_batch_kernel<12>)
  ADI_TILE_CFG(tile_batch_kernel<16>)
#undef ADI_TILE_CFG
  return e;
}

}  // namespace adi
