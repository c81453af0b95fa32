// CIC weights, gathers and the kick-drift update shared by the particle
// kernels (particles.cu, plain.cu); fixed operation order, so every kernel
// gives the same bits for the same particle.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "particles.cuh"

namespace pm {

// Lower and upper node and their CIC weights along one periodic axis.
__device__ __forceinline__ void cic_axis(float x, int n, int& i0, int& i1, float& w0, float& w1) {
  float f = floorf(x);
  w1 = __fsub_rn(x, f);
  w0 = __fsub_rn(1.0f, w1);
  i0 = (int)f;
  if (i0 >= n) i0 -= n;
  if (i0 < 0) i0 += n;
  i1 = (i0 + 1 == n) ? 0 : i0 + 1;
}

// Fixed point: weights a1 = floor(f 2^20), mass split hi = (M a1 + 2^19) >> 20, lo = M - hi.
__device__ __forceinline__ void fixed_axis(float x, int n, int& i0, int& i1, long long& a1) {
  float f = floorf(x);
  float fr = __fsub_rn(x, f);
  a1 = (long long)__fmul_rn(fr, 1048576.0f);
  i0 = (int)f;
  if (i0 >= n) i0 -= n;
  if (i0 < 0) i0 += n;
  i1 = (i0 + 1 == n) ? 0 : i0 + 1;
}
__device__ __forceinline__ void fixed_split(long long M, long long a1, long long& lo, long long& hi) {
  hi = (M * a1 + (1LL << 19)) >> 20;
  lo = M - hi;
}
__device__ __forceinline__ void fixed_corners(long long M, const long long a[3], long long out[8]) {
  long long mx[2], my[2], mz[2];
  fixed_split(M, a[0], mx[0], mx[1]);
#pragma unroll
  for (int dx = 0; dx < 2; ++dx) {
    fixed_split(mx[dx], a[1], my[0], my[1]);
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      fixed_split(my[dy], a[2], mz[0], mz[1]);
      out[dx + 2 * dy + 0] = mz[0];
      out[dx + 2 * dy + 4] = mz[1];
    }
  }
}

// CIC gather of a [3][n^3] field; fixed operation order so recomputation is bit-identical.
__device__ __forceinline__ void gather(const float* __restrict__ F, int n, float px, float py, float pz, float a[3]) {
  int ix[2], iy[2], iz[2];
  float wx[2], wy[2], wz[2];
  cic_axis(px, n, ix[0], ix[1], wx[0], wx[1]);
  cic_axis(py, n, iy[0], iy[1], wy[0], wy[1]);
  cic_axis(pz, n, iz[0], iz[1], wz[0], wz[1]);
  const int64_t n3 = (int64_t)n * n * n;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    float w = __fmul_rn(__fmul_rn(wx[dx], wy[dy]), wz[dz]);
    int64_t idx = ((int64_t)iz[dz] * n + iy[dy]) * n + ix[dx];
    s0 = __fmaf_rn(w, __ldg(F + idx), s0);
    s1 = __fmaf_rn(w, __ldg(F + n3 + idx), s1);
    s2 = __fmaf_rn(w, __ldg(F + 2 * n3 + idx), s2);
  }
  a[0] = s0;
  a[1] = s1;
  a[2] = s2;
}

// gather() from the interleaved form of the mesh, (x, y, z, unused) per node:
// one 16-byte load per corner, the two x neighbours mostly in one sector.
__device__ __forceinline__ void gather4(const float4* __restrict__ F, int n, float px, float py, float pz, float a[3]) {
  int ix[2], iy[2], iz[2];
  float wx[2], wy[2], wz[2];
  cic_axis(px, n, ix[0], ix[1], wx[0], wx[1]);
  cic_axis(py, n, iy[0], iy[1], wy[0], wy[1]);
  cic_axis(pz, n, iz[0], iz[1], wz[0], wz[1]);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const float w = __fmul_rn(__fmul_rn(wx[dx], wy[dy]), wz[dz]);
    const float4 f = __ldg(F + ((int64_t)iz[dz] * n + iy[dy]) * n + ix[dx]);
    s0 = __fmaf_rn(w, f.x, s0);
    s1 = __fmaf_rn(w, f.y, s1);
    s2 = __fmaf_rn(w, f.z, s2);
  }
  a[0] = s0;
  a[1] = s1;
  a[2] = s2;
}

// acc4: the interleaved fine mesh, used in place of acc_f when set.
__device__ __forceinline__ void accel_at(const Geo& g, const float* acc_c, const float* acc_f, const float4* acc4,
                                         float px, float py, float pz, float a[3]) {
  if (acc4) gather4(acc4, g.nf, px, py, pz, a);
  else gather(acc_f, g.nf, px, py, pz, a);
  if (g.two) {
    float s = 1.0f / (float)g.rc;
    float b[3];
    gather(acc_c, g.nc, __fmul_rn(px, s), __fmul_rn(py, s), __fmul_rn(pz, s), b);
    a[0] = __fadd_rn(b[0], a[0]);
    a[1] = __fadd_rn(b[1], a[1]);
    a[2] = __fadd_rn(b[2], a[2]);
  }
}

// A position at most one box length outside [0, nf), brought back in; then
// (wrap_far) one that moved further, or was rounded onto nf, or is no number.
__device__ __forceinline__ float wrap_near(float x, float nf) {
  x = x < 0.f ? __fadd_rn(x, nf) : x;
  return x >= nf ? __fsub_rn(x, nf) : x;
}
__device__ __forceinline__ float wrap_far(float x, float nf) {
  if (x >= 0.f && x < nf) return x;
  x = __fsub_rn(x, __fmul_rn(nf, floorf(__fdiv_rn(x, nf))));
  return x >= 0.f && x < nf ? x : 0.f;
}
__device__ __forceinline__ float wrap_pos(float x, float nf) { return wrap_far(wrap_near(x, nf), nf); }

// v' = v + c_k a ; x' = wrap(x + c_d v')
__device__ __forceinline__ void kick_drift(float x[3], float v[3], const float a[3], float ck, float cd, float nf) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    v[d] = __fmaf_rn(ck, a[d], v[d]);
    x[d] = wrap_pos(__fmaf_rn(cd, v[d], x[d]), nf);
  }
}

// Sums v[] over runs of consecutive lanes holding the same key (the particle
// stream is cell ordered, so a warp's particles form few runs); returns true
// on the last lane of each run, which then holds the run's totals.
template <int K, typename T>
__device__ __forceinline__ bool run_reduce(unsigned key, T (&v)[K]) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned prev = __shfl_up_sync(FULL, key, 1);
  const unsigned next = __shfl_down_sync(FULL, key, 1);
  const bool head = lane == 0 || prev != key;
  const bool tail = lane == 31 || next != key;
  const unsigned heads = __ballot_sync(FULL, head);
  const int start = 31 - __clz(heads & (FULL >> (31 - lane)));
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      T u = __shfl_up_sync(FULL, v[k], o);
      if (lane - start >= o) v[k] += u;
    }
  }
  return tail;
}

}  // namespace pm
