// adi_copy.cu -- fields crossing the ABI: contiguous [ny][nx] arrays of the
// caller to and from the handle's pitched [ny][ld] rows, and the start-up
// of Eq. (CN2).
//
// All of these are bound by HBM.  A thread moves four columns of eight rows,
// its loads issued together: 16-byte groups where both sides' rows start on
// 16 bytes, single floats otherwise.  Both levels of a state go in one
// launch, and the start-up reads phi once for its two.  At 16384^2 a restart
// and a read-out (7 GiB of traffic) take 1.3 ms; the row-by-row copies and a
// start-up of one node per thread took 3.0.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "adi_internal.h"

namespace adi {

namespace {

constexpr int kRows = 8;
constexpr int kThreads = 128;

template <bool VEC>
__device__ __forceinline__ float4 get4(const float* p, int n) {
  if (VEC) return __ldcs(reinterpret_cast<const float4*>(p));
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  const int s = kThreads;  // a warp's lanes stay next to one another
  if (0 * s < n) v.x = __ldcs(p);
  if (1 * s < n) v.y = __ldcs(p + s);
  if (2 * s < n) v.z = __ldcs(p + 2 * s);
  if (3 * s < n) v.w = __ldcs(p + 3 * s);
  return v;
}

template <bool VEC>
__device__ __forceinline__ void put4(float* p, const float4& v, int n) {
  if (VEC) {
    *reinterpret_cast<float4*>(p) = v;
    return;
  }
  const int s = kThreads;
  if (0 * s < n) p[0] = v.x;
  if (1 * s < n) p[s] = v.y;
  if (2 * s < n) p[2 * s] = v.z;
  if (3 * s < n) p[3 * s] = v.w;
}

// dst0 <- src0 and dst1 <- src1 (blockIdx.z: one of the two), or with both a
// dst1 and no src1, dst0 and dst1 <- src0.  VEC: nx, both pitches and all
// pointers are multiples of 16 bytes.  gd_dst <- gd if given.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) copy_fields_kernel(const CopyArgs a, const GridDev gd) {
  if (a.gd_dst != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *a.gd_dst = gd;
  const float* src = blockIdx.z ? a.src1 : a.src0;
  float* dst = blockIdx.z ? a.dst1 : a.dst0;
  float* dup = a.src1 == nullptr ? a.dst1 : nullptr;
  const int c = VEC ? 4 * (blockIdx.x * kThreads + threadIdx.x) : 4 * blockIdx.x * kThreads + threadIdx.x;
  const int n = a.nx - c;  // floats from column c to the row's end
  if (n <= 0) return;
  for (int j0 = blockIdx.y * kRows; j0 < a.ny; j0 += gridDim.y * kRows) {
    float4 v[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
      if (j0 + r < a.ny) v[r] = get4<VEC>(src + (size_t)(j0 + r) * a.spitch + c, n);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (j0 + r < a.ny) {
        put4<VEC>(dst + (size_t)(j0 + r) * a.dpitch + c, v[r], n);
        if (dup != nullptr) put4<VEC>(dup + (size_t)(j0 + r) * a.dpitch + c, v[r], n);
      }
    }
  }
}

// Eq. (CN2) with a velocity or to second order: u^0 = phi, u^1 = phi + tau
// psi (+ tau^2/2 (m Lap phi + f^0)), formed in FP64, whose rate bounds it: at
// 4096^2 the second-order start takes 533 us and a velocity 132, 629 and 165
// where the two are told apart per node.
template <bool PSI>
__global__ void init_kernel(const InitArgs a, const GridDev gd) {
  if (a.gd_dst != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *a.gd_dst = gd;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= a.nx || j >= a.ny) return;
  const size_t c = (size_t)j * a.nx + i;
  const double ph = a.phi[c];
  double v = PSI ? ph + a.tau * (double)a.psi[c] : ph;
  if (a.taylor) {
    const double l = (i > 0) ? a.phi[c - 1] : 0.0;
    const double r = (i + 1 < a.nx) ? a.phi[c + 1] : 0.0;
    const double dn = (j > 0) ? a.phi[c - a.nx] : 0.0;
    const double up = (j + 1 < a.ny) ? a.phi[c + a.nx] : 0.0;
    const double mm = a.m[(size_t)j * a.ld + i];
    v += mm * (a.cx_half * (l + r - 2.0 * ph) + a.cy_half * (dn + up - 2.0 * ph));
    if (i == a.sx && j == a.sy && a.wavelet != nullptr && a.n_wavelet > 0) v += a.src_half * a.wavelet[0];
  }
  a.u0[(size_t)j * a.ld + i] = (float)ph;
  a.u1[(size_t)j * a.ld + i] = (float)v;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

cudaError_t launch_copy_fields(const CopyArgs& a, const GridDev& gd, cudaStream_t st) {
  const bool vec = a.nx % 4 == 0 && a.spitch % 4 == 0 && a.dpitch % 4 == 0 && aligned16(a.src0) &&
                   aligned16(a.dst0) && aligned16(a.src1) && aligned16(a.dst1);
  const dim3 grid((a.nx + 4 * kThreads - 1) / (4 * kThreads), std::min((a.ny + kRows - 1) / kRows, 65535),
                  a.src1 != nullptr ? 2 : 1);
  if (vec) copy_fields_kernel<true><<<grid, kThreads, 0, st>>>(a, gd);
  else copy_fields_kernel<false><<<grid, kThreads, 0, st>>>(a, gd);
  return cudaGetLastError();
}

cudaError_t launch_init(const InitArgs& a, const GridDev& gd, cudaStream_t st) {
  if (!a.psi && !a.taylor) {  // u^1 = u^0 = phi: no arithmetic
    CopyArgs c = {};
    c.nx = a.nx;
    c.ny = a.ny;
    c.spitch = a.nx;
    c.dpitch = a.ld;
    c.src0 = a.phi;
    c.dst0 = a.u0;
    c.dst1 = a.u1;
    c.gd_dst = a.gd_dst;
    return launch_copy_fields(c, gd, st);
  }
  dim3 block(256, 1, 1);
  dim3 grid((a.nx + 255) / 256, a.ny, 1);
  if (a.psi) init_kernel<true><<<grid, block, 0, st>>>(a, gd);
  else init_kernel<false><<<grid, block, 0, st>>>(a, gd);
  return cudaGetLastError();
}

}  // namespace adi
