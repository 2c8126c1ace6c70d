// adi_local.cuh -- building blocks of the local line solves (adi_tile.cu,
// adi_patch.cu): packed FP32 arithmetic and the division-free elimination.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "adi_chain.cuh"
#include "adi_device.cuh"
#include "adi_internal.h"

namespace adi {

__device__ __forceinline__ float lds(uint32_t a) { return *reinterpret_cast<const float*>(__cvta_shared_to_generic(a)); }

// Two FP32 numbers in one 64-bit register pair: one packed instruction does
// the work of two, which halves the issue slots of the elimination.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo2(f2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 dup2(float v) { return pk(v, v); }
__device__ __forceinline__ f2 lds2(uint32_t a) { return *reinterpret_cast<const f2*>(__cvta_shared_to_generic(a)); }
__device__ __forceinline__ ulonglong2 lds4(uint32_t a) {
  return *reinterpret_cast<const ulonglong2*>(__cvta_shared_to_generic(a));
}

// Elimination of -s x_{k-1} + (1 + 2s) x_k - s x_{k+1} = d without a
// reciprocal in its chain.  With gamma_k = a_k / p_k and delta_k = N_k / p_k,
//     a_k = s_k p_{k-1},  p_k = p_{k-1} + s_k (2 p_{k-1} - a_{k-1}),
//     N_k = s_k N_{k-1} + d_k p_{k-1}
// (every term of p is positive, so nothing cancels): two dependent FMAs per
// unknown, and the reciprocals of the p_k are independent of one another.  p
// grows by at most 1 + 2s per unknown, 2^16 over a block at s = 1/2, the
// largest s the halo of 16 allows; every block starts again from p = 1.  N is
// p times a solution value, so that fields may be as large as 2^111 (2.6e33).
//
// The packed instructions take no negated operands, so signs are carried by
// the data instead, in a fixed pattern of period 4: s enters as (-1)^k s_k,
// d as sigma_k d_k with sigma = + - - +, and with them a as (-1)^k a_k, N as
// sigma_k N_k; solve() takes the reciprocal of -p, and then
//     X_k = -sigma_k x_k  obeys  X_k = G_k X_{k+1} + D_k.
__device__ __forceinline__ constexpr float sgn_d(int k) { return ((k & 3) == 1 || (k & 3) == 2) ? -1.f : 1.f; }
struct Elim2 {
  f2 p, a, N;
  __device__ __forceinline__ void begin(f2 a0, f2 n0) {
    p = dup2(1.f);
    a = a0;
    N = n0;
  }
  template <int KP>  // parity of k
  __device__ __forceinline__ void add(f2 s, f2 d) {
    const f2 t = fma2(dup2(KP ? -2.f : 2.f), p, a);  // +-(2 p - a)
    a = mul2(s, p);
    N = fma2(s, N, mul2(d, p));
    p = fma2(s, t, p);
  }
  // the last H of a chunk's unknowns
  template <int H>
  __device__ __forceinline__ void tail(const f2 (&S)[16], const f2 (&D)[16]) {
#pragma unroll
    for (int k = 16 - H; k < 16; ++k) {
      if (k & 1) add<1>(S[k], D[k]);
      else add<0>(S[k], D[k]);
    }
  }
  // the chunk: S, D become G, D of the back substitution
  __device__ __forceinline__ void chunk(f2 (&S)[16], f2 (&D)[16]) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (k & 1) add<1>(S[k], D[k]);
      else add<0>(S[k], D[k]);
      solve(S[k], D[k]);
    }
  }
  __device__ __forceinline__ void solve(f2& G, f2& D) const {
    f2 r = pk(rcp_t(-lo2(p)), rcp_t(-hi2(p)));
    r = fma2(fma2(p, r, dup2(1.f)), r, r);  // one Newton step on the approximate reciprocal
    G = mul2(a, r);
    D = mul2(N, r);
  }
};

// u^{k+1} = q + z from X (z = -sigma X)
__device__ __forceinline__ f2 updated(int i, f2 q, f2 X) {
  return sgn_d(i) > 0.f ? fma2(dup2(-1.f), X, q) : fma2(dup2(-1.f), q, X);
}


// The same elimination of one system in scalar arithmetic, operation for
// operation: x_k = G x_{k+1} + D.
struct Elim1 {
  float p, a, N;
  __device__ __forceinline__ void begin(float a0, float n0) {
    p = 1.f;
    a = a0;
    N = n0;
  }
  __device__ __forceinline__ void add(float s, float d) {
    const float t = fmaf(2.f, p, -a);
    a = s * p;
    N = fmaf(s, N, d * p);
    p = fmaf(s, t, p);
  }
  template <int H>
  __device__ __forceinline__ void tail(const float (&S)[16], const float (&D)[16]) {
#pragma unroll
    for (int k = 16 - H; k < 16; ++k) add(S[k], D[k]);
  }
  __device__ __forceinline__ void chunk(float (&S)[16], float (&D)[16]) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      add(S[k], D[k]);
      float r = rcp_t(p);
      r = fmaf(fmaf(-p, r, 1.f), r, r);
      S[k] = a * r;
      D[k] = N * r;
    }
  }
};

// tau^2 f^k of a step's point source, f^k = w(t_k) / (h1 h2) at one node, and
// the level.  early() before chain_wait(), late() behind it.
struct Source {
  int sx, sy;
  float f;
  long long lev;
  __device__ __forceinline__ void set(const float* wavelet, int n, int ix, int iy, float scale) {
    const bool on = ix >= 0 && wavelet != nullptr && lev >= 0 && lev < n;
    sx = on ? ix : -1;
    sy = on ? iy : -1;
    f = on ? scale * wavelet[lev] : 0.f;
  }
  __device__ __forceinline__ void early(const TileArgs& a) {
    lev = a.level;
    if (a.by_value) set(a.wavelet, a.n_wavelet, a.src_ix, a.src_iy, a.src_scale);
  }
  // advance: this thread leaves the next level in the record's other word
  __device__ __forceinline__ void late(const TileArgs& a, int par, bool advance) {
    if (a.by_value) return;
    lev = a.gd->kf[par];
    set(a.gd->wavelet, a.gd->n_wavelet, a.gd->src_ix, a.gd->src_iy, a.src_scale);
    if (advance) a.gd->kf[par ^ 1] = lev + 1;
  }
};

// Receiver sampling inside the step that starts from u^k: traces[k - k0 - 1][r]
// = u^k(rec r) of the receivers in columns [x0, x1), rows [y0, y1).  (The last
// level of a run is sampled by a launch of its own.)  Sampling the field a
// step reads rather than the one it writes keeps it off the end of the step,
// which the next step waits for: look() finds the receivers of the CTA before
// chain_wait() -- their list is not written during a run -- and sample()
// copies the values while the stage is on its way.  1000^2 with 64 receivers:
// 8.0 against 10.1 us per step.  Long lists are left to a launch after the step
// (adi_wave::sampling_of).
struct Sampler {
  int at;  // the node of receiver threadIdx.x, -1 = none of this CTA's
  static __device__ __forceinline__ int node(const TileArgs& a, int r, int x0, int x1, int y0, int y1) {
    const int2 p = reinterpret_cast<const int2*>(a.rec)[r];
    return p.x >= x0 && p.x < x1 && p.y >= y0 && p.y < y1 ? (p.y - y0) * (x1 - x0) + (p.x - x0) : -1;
  }
  __device__ __forceinline__ void look(const TileArgs& a, int x0, int x1, int y0, int y1) {
    at = (int)threadIdx.x < a.n_rec ? node(a, threadIdx.x, x0, x1, y0, y1) : -1;
  }
  __device__ __forceinline__ void sample(const TileArgs& a, const GridDev* gd, long long lev, int x0, int x1, int y0,
                                         int y1) const {
    if (at < 0 && a.n_rec <= (int)blockDim.x) return;
    const long long s = lev - gd->k0 - 1;
    float* tr = gd->traces;
    if (tr == nullptr || s < 0 || s >= gd->steps) return;
    const int w = x1 - x0;
    for (int r = threadIdx.x; r < a.n_rec; r += blockDim.x) {
      const int q = r < (int)blockDim.x ? at : node(a, r, x0, x1, y0, y1);
      if (q >= 0) tr[s * a.n_rec + r] = __ldcg(a.u_cur + (size_t)(y0 + q / w) * a.ld + x0 + q % w);
    }
  }
};

}  // namespace adi
