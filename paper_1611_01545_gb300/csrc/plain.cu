// Kernels over float particles (the plain, one-call-per-stage path):
// decompress (Sec. 2.4), CIC deposit in float32 or int64 fixed point, deposit
// of per-particle weights, CIC force interpolation, kick and drift.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "cic.cuh"
#include "particles.cuh"

namespace pm {

// ---- decompress -----------------------------------------------------------
//
// A block owns kDecChunk consecutive particles (cells differ in weight by
// orders of magnitude on clustered sets, chunks do not), finds the cells of
// the first and the last of them by a 32-way search, and keeps the offsets
// and coordinates of the cells between in shared memory, where a particle
// finds its cell in a few reads.  (One thread per particle with a search over
// all cells' offsets in global memory, 18 dependent loads on a 64^3 mesh, took
// 367 us for 16.8M particles with 16-bit codes; this takes 182 us,
// against 91 us for the bytes alone.)  Positions and velocities go through
// shared memory so that a warp writes whole 128-byte lines where 12-byte
// records would touch each line three times.

constexpr int kDecThreads = 256;
constexpr int kDecChunk = 2048;
constexpr int kDecCells = 512;   // cells of a chunk kept in shared memory; sparser chunks search global memory

// The last cell c in [lo, hi] with off[c] <= p (off[lo] <= p), by a warp.
__device__ __forceinline__ int64_t warp_find_cell(const int64_t* off, int64_t lo, int64_t hi, int64_t p) {
  while (lo < hi) {
    const int64_t step = (hi - lo) / 32 + 1;
    const int64_t c = lo + step * ((threadIdx.x & 31) + 1);
    const int k = __popc(__ballot_sync(0xffffffffu, c <= hi && off[c] <= p));
    const int64_t end = lo + step * (k + 1) - 1;
    lo += step * k;
    hi = end < hi ? end : hi;
  }
  return lo;
}

__global__ void __launch_bounds__(kDecThreads) k_decompress(PCodes in, const int64_t* off, Geo g, float* x, float* v) {
  __shared__ int64_t ends[2];
  __shared__ int64_t ro[kDecCells];
  __shared__ ushort4 at[kDecCells];
  __shared__ float sx[3 * kDecThreads], sv[3 * kDecThreads];
  const float pscale = (float)g.rcmp / 256.0f;
  const int half = in.vel16 ? 32768 : 128;
  const float step = __fmul_rn(*in.vmax, 1.0f / (float)half);
  const uint32_t nc = (uint32_t)g.ncmp;
  for (int64_t p0 = (int64_t)blockIdx.x * kDecChunk; p0 < in.n; p0 += (int64_t)gridDim.x * kDecChunk) {
    const int64_t p1 = p0 + kDecChunk < in.n ? p0 + kDecChunk : in.n;
    const int wid = threadIdx.x >> 5;
    if (wid < 2) {
      const int64_t c = warp_find_cell(off, 0, g.ncell - 1, wid ? p1 - 1 : p0);
      if ((threadIdx.x & 31) == 0) ends[wid] = c;
    }
    __syncthreads();
    const int64_t c0 = ends[0], c1 = ends[1];
    const bool local = c1 - c0 < kDecCells;
    const int cells = local ? (int)(c1 - c0) + 1 : 0;
    int top = 1;   // power of two, at least cells / 2
    while (2 * top < cells) top *= 2;
    for (int i = threadIdx.x; i < cells; i += kDecThreads) {
      ro[i] = off[c0 + i];
      const uint32_t c = (uint32_t)(c0 + i);
      at[i] = make_ushort4((unsigned short)(c % nc), (unsigned short)(c / nc % nc), (unsigned short)(c / nc / nc), 0);
    }
    __syncthreads();
    for (int64_t pb = p0; pb < p1; pb += kDecThreads) {
      const int64_t p = pb + threadIdx.x;
      if (p < p1) {
        ushort4 c;
        if (local) {
          int lo = 0;
          for (int d = top; d > 0; d >>= 1)
            if (lo + d < cells && ro[lo + d] <= p) lo += d;
          c = at[lo];
        } else {
          int64_t lo = c0, hi = c1;
          while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (off[mid] <= p) lo = mid; else hi = mid - 1;
          }
          const uint32_t k = (uint32_t)lo;
          c = make_ushort4((unsigned short)(k % nc), (unsigned short)(k / nc % nc), (unsigned short)(k / nc / nc), 0);
        }
        int q[3], qv[3];
        unpack_pos(in.pos[p], q);
        load_vel(in.vel, in.vel16, p, qv);
        sx[3 * threadIdx.x] = decode_pos(c.x, q[0], pscale);
        sx[3 * threadIdx.x + 1] = decode_pos(c.y, q[1], pscale);
        sx[3 * threadIdx.x + 2] = decode_pos(c.z, q[2], pscale);
#pragma unroll
        for (int d = 0; d < 3; ++d) sv[3 * threadIdx.x + d] = decode_vel(qv[d], half, step);
      }
      __syncthreads();
      const int m = 3 * (int)(p1 - pb < kDecThreads ? p1 - pb : kDecThreads);
      for (int i = threadIdx.x; i < m; i += kDecThreads) {
        x[3 * pb + i] = sx[i];
        v[3 * pb + i] = sv[i];
      }
      __syncthreads();
    }
  }
}

// ---- deposits of float particles --------------------------------------
//
// A particle order that follows the mesh (the cell order that decompression
// leaves, a lattice) puts the particles of a warp into a few neighbouring
// cells, so adding every CIC corner to the global mesh sends most of a warp's
// atomics to the same few addresses, which L2 serialises: worst on the coarse
// mesh, where the 64 neutrinos of one coarse cell share all 8 nodes (1.5 of
// 2.0 ms).  A warp therefore takes 32 PER consecutive particles; when the box
// of their fine nodes holds at most kBoxCells nodes it bins the corners in
// shared memory and adds each touched node to the mesh once, else (random
// order, sparse species, a box that straddles the end of a mesh row) it adds
// the corners directly.  Coarse corners are summed over the runs of lanes in
// the same coarse cell.  The box is per warp, not per block: no block
// barriers, and 256 neutrinos span 4 compression cells (17 x 5 x 5 nodes)
// where a block's 2,048 would straddle a mesh row half of the time.
// 256^3 mesh, 16.8M cell-ordered neutrinos: float32 2004 -> 339 us, int64
// 1932 -> 443 us, three weights (float atomics on shared memory, which bound
// it) 1433 -> 917 us; 2.1M particles in random order on 128^3 75 -> 76 us (the
// look at the box).  A third of the float32 time is the coarse mesh's, 20 us
// the global adds of the boxes.

constexpr int kDepThreads = 256;
constexpr int kDepWarps = kDepThreads / 32;
constexpr int kBoxCells = 640;    // 40 KB per block in two 32-bit words
// Runs of equal coarse cells in a warp: one or two are summed run by run
// (warp_sum8: 27 us less than with the scan for the neutrinos above), up
// to kMaxRuns by a segmented scan (2.1M CDM particles, 4 or 5 runs: 44 us, run
// by run 61), more go to the mesh one by one.
constexpr int kMaxRuns = 8;

// Nodes touched by the particles of a warp: origin and extents (upper nodes
// included), in mesh cells without wrap.
struct WarpBox {
  int ox, oy, oz, ex, ey, ez;
  bool fits;
};
// Nodes up to which a group of `count` particles is binned: clearing and
// flushing the box has to cost less than the 8 adds per particle that it saves
// (64 CDM particles over 33 x 5 x 5 nodes: 76 us binned, 44 us direct).
__device__ __forceinline__ int box_cap(int count) { return 4 * count < kBoxCells ? 4 * count : kBoxCells; }

// Box of the particles first .. first + count - 1 (count > 0), the same on every lane.
// FINITE: a group with a coordinate that is no number has none, because its corner
// terms are no numbers either, which integer bins cannot hold and the mesh has to
// show (float bins can).
template <bool FINITE>
__device__ __forceinline__ WarpBox warp_box(const float* x, int64_t first, int count, int nf, int cap) {
  int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
  float odd = 0.f;   // 0 x summed over the coordinates: 0, or NaN
  // the first 32 particles, then (unless their box is too large already: a
  // random order is found out after 1 / PER of the work) the others
  for (int part = 0; part < 2; ++part) {
    const int from = part ? 32 : 0, to = part ? count : (count < 32 ? count : 32);
#pragma unroll 4
    for (int k = from + (threadIdx.x & 31); k < to; k += 32) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float xd = x[3 * (first + k) + d];
        if (FINITE) odd = __fmaf_rn(xd, 0.f, odd);
        int i0 = (int)floorf(xd);
        if (i0 >= nf) i0 -= nf;
        if (i0 < 0) i0 += nf;
        lo[d] = min(lo[d], i0);
        hi[d] = max(hi[d], i0);
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      lo[d] = __reduce_min_sync(0xffffffffu, lo[d]);
      hi[d] = __reduce_max_sync(0xffffffffu, hi[d]);
    }
    if ((float)(hi[0] - lo[0] + 2) * (float)(hi[1] - lo[1] + 2) * (float)(hi[2] - lo[2] + 2) > (float)cap) break;
  }
  WarpBox b{lo[0], lo[1], lo[2], 0, 0, 0, false};
  if (FINITE && __any_sync(0xffffffffu, odd != 0.f)) return b;
  // extents are checked one by one, so that no product overflows
  const long long e0 = (long long)hi[0] - lo[0] + 2, e1 = (long long)hi[1] - lo[1] + 2,
                  e2 = (long long)hi[2] - lo[2] + 2;
  if (e0 >= 2 && e1 >= 2 && e2 >= 2 && e0 <= cap && e1 <= cap && e2 <= cap && e0 * e1 * e2 <= cap) {
    b.ex = (int)e0;
    b.ey = (int)e1;
    b.ez = (int)e2;
    b.fits = true;
  }
  return b;
}

// Shared-memory bins of one warp's mass deposit: two 32-bit words per node,
// t = 2^16 hi + lo, added with native integer atomics (float32 atomics on
// shared memory take 402 us in place of 339 for the neutrinos above).  int64: the
// term itself (the caller bounds the mass so that neither word overflows).
// float32: the term in units of 2^-16 / scale, scale a power of two such that
// the mass of a whole group stays below 2^30 / scale: at most 2^-37 of the
// particle mass, so the bins add no error of their own (one 32-bit word in
// units of 2^-22 of the mass raised the acceleration error of the sparse
// species from 1.0e-6 to 2.5e-6).
template <typename Acc> struct Bins;
template <> struct Bins<float> {
  static __device__ __forceinline__ void add(uint32_t* s, int i, float v, float scale) {
    // |v scale| <= 2^22: adding 1.5 2^23 rounds to an integer in the low bits
    const float a = __fmul_rn(v, scale), magic = 12582912.0f;
    const float r = __fadd_rn(a, magic);
    const float lo = __fmaf_rn(__fsub_rn(a, __fsub_rn(r, magic)), 65536.0f, magic);
    atomicAdd(reinterpret_cast<int*>(s) + kBoxCells + i, __float_as_int(r) - 0x4B400000);
    atomicAdd(reinterpret_cast<int*>(s) + i, __float_as_int(lo) - 0x4B400000);
  }
  static __device__ __forceinline__ float get(const uint32_t* s, int i, float inv) {
    const float lo = __int2float_rn((int)s[i]), hi = __int2float_rn((int)s[kBoxCells + i]);
    return __fmul_rn(__fmaf_rn(lo, 1.0f / 65536.0f, hi), inv);
  }
};
template <> struct Bins<long long> {
  static __device__ __forceinline__ void add(uint32_t* s, int i, long long v, float) {
    atomicAdd(s + i, (uint32_t)(v & 0xffff));
    atomicAdd(s + kBoxCells + i, (uint32_t)(int32_t)(v >> 16));
  }
  static __device__ __forceinline__ long long get(const uint32_t* s, int i, float) {
    return ((long long)(int32_t)s[kBoxCells + i] << 16) + (long long)s[i];
  }
};
// Bins of per-particle weights (any float values): float32 sums.
struct FloatBins {
  static __device__ __forceinline__ float get(const uint32_t* s, int i, float) { return __uint_as_float(s[i]); }
};

__device__ __forceinline__ void mesh_add(float* a, float v) { atomicAdd(a, v); }
__device__ __forceinline__ void mesh_add(long long* a, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(a), (unsigned long long)v);
}

// The 8 corner terms of a particle at mesh position p (mesh units), with the
// lower node i0 and the wrapped upper node i1: float32 m w_x w_y w_z, or the
// conservative integer split of M.
__device__ __forceinline__ void corner_terms(const float p[3], int n, float m, long long, int i0[3], int i1[3],
                                             float out[8]) {
  float w0[3], w1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) cic_axis(p[d], n, i0[d], i1[d], w0[d], w1[d]);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const float w = __fmul_rn(__fmul_rn(dx ? w1[0] : w0[0], dy ? w1[1] : w0[1]), dz ? w1[2] : w0[2]);
    out[c] = __fmul_rn(m, w);
  }
}
__device__ __forceinline__ void corner_terms(const float p[3], int n, float, long long M, int i0[3], int i1[3],
                                             long long out[8]) {
  long long a1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) fixed_axis(p[d], n, i0[d], i1[d], a1[d]);
  fixed_corners(M, a1, out);
}
template <typename Acc>
__device__ __forceinline__ void add_corners(Acc* rho, int n, const int i0[3], const int i1[3], const Acc t[8]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int gx = c & 1 ? i1[0] : i0[0], gy = (c >> 1) & 1 ? i1[1] : i0[1], gz = c >> 2 ? i1[2] : i0[2];
    mesh_add(&rho[((int64_t)gz * n + gy) * n + gx], t[c]);
  }
}

// Adds the touched nodes of a warp's box to the periodic mesh rho[n^3].
template <class B, typename Acc>
__device__ __forceinline__ void flush_box(const uint32_t* s, const WarpBox& b, Acc* rho, int n, float inv) {
  const int lane = threadIdx.x & 31;
  const int rows = b.ey * b.ez;
  int ly = 0, gz = b.oz;
  for (int r = 0; r < rows; ++r) {
    int gy = b.oy + ly;
    if (gy >= n) gy -= n;
    Acc* row = rho + ((int64_t)gz * n + gy) * n;
    for (int lx = lane; lx < b.ex; lx += 32) {
      const Acc v = B::get(s, r * b.ex + lx, inv);
      int gx = b.ox + lx;
      if (gx >= n) gx -= n;
      if (v != (Acc)0) mesh_add(row + gx, v);
    }
    if (++ly == b.ey) {
      ly = 0;
      if (++gz >= n) gz -= n;
    }
  }
}

// Local index of a box node, and the corner c relative to the lower one.
__device__ __forceinline__ int box_at(const WarpBox& b, const int i0[3]) {
  return ((i0[2] - b.oz) * b.ey + (i0[1] - b.oy)) * b.ex + (i0[0] - b.ox);
}
__device__ __forceinline__ int box_corner(const WarpBox& b, int c) {
  return ((c >> 2) * b.ey + ((c >> 1) & 1)) * b.ex + (c & 1);
}

// Sums of 8 values over the warp's lanes with `mine`; lane l returns the sum of
// value l >> 2.  Each of the first three exchanges halves the values a lane
// still carries (4 + 2 + 1 shuffles, then 2 of the last value) where a scan of
// all 8 values takes 40.
template <typename Acc>
__device__ __forceinline__ Acc warp_sum8(const Acc t[8], bool mine) {
  const int lane = threadIdx.x & 31;
  Acc a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const Acc lo = mine ? t[i] : (Acc)0, hi = mine ? t[i + 4] : (Acc)0;
    a[i] = (lane & 16 ? hi : lo) + __shfl_xor_sync(0xffffffffu, lane & 16 ? lo : hi, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
    b[i] = (lane & 8 ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 8 ? a[i] : a[i + 2], 8);
  c = (lane & 4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

// The positions are read again for each of the three uses (box, fine, coarse;
// a warp's 3 KB stay in L1) rather than kept: kept, they cost 126 registers.
// scale = 0 switches the bins off (a mass that does not fit them).
template <typename Acc, int PER>
__global__ void __launch_bounds__(kDepThreads) k_deposit(const float* x, int64_t n, float m, long long M,
                                                         float scale, Geo g, Acc* rho_c, Acc* rho_f) {
  __shared__ uint32_t bins[kDepWarps][2 * kBoxCells];
  const int lane = threadIdx.x & 31;
  uint32_t* s = bins[threadIdx.x >> 5];
  constexpr int kGroup = 32 * PER;
  const int64_t groups = (n + kGroup - 1) / kGroup;
  const int64_t warps = (int64_t)gridDim.x * kDepWarps;
  for (int64_t gr = (int64_t)blockIdx.x * kDepWarps + (threadIdx.x >> 5); gr < groups; gr += warps) {
    const int64_t first = gr * kGroup;
    const int count = n - first < kGroup ? (int)(n - first) : kGroup;
    WarpBox b = warp_box<true>(x, first, count, g.nf, box_cap(count));
    b.fits = b.fits && scale != 0.f;
    if (b.fits) {
      const int vol = b.ex * b.ey * b.ez;
      for (int i = lane; i < vol; i += 32) {
        s[i] = 0u;
        s[kBoxCells + i] = 0u;
      }
      __syncwarp();
    }
    for (int k = lane; k < count; k += 32) {
      const float* xp = x + 3 * (first + k);
      const float p[3] = {xp[0], xp[1], xp[2]};
      int i0[3], i1[3];
      Acc t[8];
      corner_terms(p, g.nf, m, M, i0, i1, t);
      if (b.fits) {
        const int at = box_at(b, i0);
#pragma unroll
        for (int c = 0; c < 8; ++c) Bins<Acc>::add(s, at + box_corner(b, c), t[c], scale);
      } else {
        add_corners(rho_f, g.nf, i0, i1, t);
      }
    }
    if (b.fits) {
      __syncwarp();
      flush_box<Bins<Acc>>(s, b, rho_f, g.nf, 1.0f / scale);
      __syncwarp();
    }
    if (rho_c) {
      const float sc = 1.0f / (float)g.rc;
      for (int k0 = 0; k0 < count; k0 += 32) {      // whole warps: run_reduce shuffles
        const bool live = k0 + lane < count;
        const float* xp = x + 3 * (first + k0 + lane);
        float u[3] = {0.f, 0.f, 0.f};
        if (live) {
#pragma unroll
          for (int d = 0; d < 3; ++d) u[d] = __fmul_rn(xp[d], sc);
        }
        int i0[3], i1[3];
        Acc t[8];
        corner_terms(u, g.nc, m, M, i0, i1, t);
        const unsigned key = live ? (unsigned)((i0[2] * g.nc + i0[1]) * g.nc + i0[0]) : 0xffffffffu;
        const unsigned prev = __shfl_up_sync(0xffffffffu, key, 1);
        unsigned heads = __ballot_sync(0xffffffffu, live && (lane == 0 || prev != key));
        const int runs = __popc(heads);
        if (runs > 2) {
          bool put = live;
          if (runs <= kMaxRuns) {
            if (!live) {
#pragma unroll
              for (int c = 0; c < 8; ++c) t[c] = (Acc)0;
            }
            put = run_reduce<8, Acc>(key, t) && put;
          }
          if (put) add_corners(rho_c, g.nc, i0, i1, t);
          continue;
        }
        while (heads) {                             // the same on every lane
          const int lead = __ffs(heads) - 1;
          heads &= heads - 1;
          const bool mine = key == __shfl_sync(0xffffffffu, key, lead) && lane >= lead &&
                            (heads == 0 || lane < __ffs(heads) - 1);
          const Acc sum = warp_sum8(t, mine);
          const int c = lane >> 2;                  // the corner this lane's sum belongs to
          int at[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            at[d] = __shfl_sync(0xffffffffu, i0[d], lead) + ((c >> d) & 1);
            if (at[d] >= g.nc) at[d] -= g.nc;
          }
          if ((lane & 3) == 0) mesh_add(&rho_c[((int64_t)at[2] * g.nc + at[1]) * g.nc + at[0]], sum);
        }
      }
    }
  }
}

// Periodic CIC deposit of nw per-particle weights (w[p nw + c], c < nw <= 4)
// onto nw fine meshes out[c][nf^3] (float32, the mesh convention of the
// deposit above): number and momentum densities for the power spectra of
// the compression study.  One component of the warp's box at a time.
template <int PER>
__global__ void __launch_bounds__(kDepThreads) k_deposit_weights(const float* x, int64_t n, const float* w, int nw,
                                                                 Geo g, float* out) {
  __shared__ uint32_t bins[kDepWarps][kBoxCells];
  const int64_t nf3 = (int64_t)g.nf * g.nf * g.nf;
  const int lane = threadIdx.x & 31;
  uint32_t* s = bins[threadIdx.x >> 5];
  constexpr int kGroup = 32 * PER;
  const int64_t groups = (n + kGroup - 1) / kGroup;
  const int64_t warps = (int64_t)gridDim.x * kDepWarps;
  for (int64_t gr = (int64_t)blockIdx.x * kDepWarps + (threadIdx.x >> 5); gr < groups; gr += warps) {
    const int64_t first = gr * kGroup;
    const int count = n - first < kGroup ? (int)(n - first) : kGroup;
    const WarpBox b = warp_box<false>(x, first, count, g.nf, box_cap(count));
    if (!b.fits) {
      for (int k = lane; k < count; k += 32) {
        const float* xp = x + 3 * (first + k);
        const float p[3] = {xp[0], xp[1], xp[2]};
        int i0[3], i1[3];
        float t[8];
        corner_terms(p, g.nf, 1.0f, 0, i0, i1, t);
        float q4[4] = {0.f, 0.f, 0.f, 0.f};
        for (int q = 0; q < nw; ++q) q4[q] = w[(first + k) * nw + q];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int gx = c & 1 ? i1[0] : i0[0], gy = (c >> 1) & 1 ? i1[1] : i0[1], gz = c >> 2 ? i1[2] : i0[2];
          float* node = out + ((int64_t)gz * g.nf + gy) * g.nf + gx;
          for (int q = 0; q < nw; ++q) atomicAdd(node + q * nf3, __fmul_rn(q4[q], t[c]));
        }
      }
      continue;
    }
    for (int q = 0; q < nw; ++q) {
      float* rho = out + q * nf3;
      const int vol = b.ex * b.ey * b.ez;
      for (int i = lane; i < vol; i += 32) s[i] = 0u;
      __syncwarp();
      for (int k = lane; k < count; k += 32) {
        const float* xp = x + 3 * (first + k);
        const float p[3] = {xp[0], xp[1], xp[2]};
        int i0[3], i1[3];
        float t[8];
        corner_terms(p, g.nf, w[(first + k) * nw + q], 0, i0, i1, t);
        const int at = box_at(b, i0);
#pragma unroll
        for (int c = 0; c < 8; ++c) atomicAdd(reinterpret_cast<float*>(s) + at + box_corner(b, c), t[c]);
      }
      __syncwarp();
      flush_box<FloatBins>(s, b, rho, g.nf, 1.f);
      __syncwarp();
    }
  }
}

// ---- force interpolation, kick and drift of float particles -----------------
//
// Bound by the gathers: 24 loads of single values per particle from the fine
// mesh, each warp load touching 10 to 32 lines.  Where the particles are at
// least half as many as the nodes the mesh is first rewritten with its three
// components next to each other (k_interleave, a streaming pass), and a corner
// is one 16-byte load.  2.1M particles in random order on 128^3, kick + drift
// 132 -> 78 us (gather alone 150 -> 69); 16.8M on 256^3 in random order 2764 ->
// 1939 us, in cell order 507 us either way.  (Gathering cell-ordered groups from
// boxes in shared memory: 447 us, but 4861 in random order, for want of L1.)
__global__ void k_interleave(const float* acc, int64_t n3, float4* out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = make_float4(__ldg(acc + i), __ldg(acc + n3 + i), __ldg(acc + 2 * n3 + i), 0.f);
}

// KICK: kick and drift x, v in place; else the interpolated acceleration goes to out.
template <bool KICK>
__global__ void k_interpolate(float* x, float* v, int64_t n, Geo g, const float* acc_c, const float* acc_f,
                              const float4* acc4, float ck, float cd, float* out) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    float xx[3] = {x[3 * p], x[3 * p + 1], x[3 * p + 2]};
    float a[3];
    accel_at(g, acc_c, acc_f, acc4, xx[0], xx[1], xx[2], a);
    if (KICK) {
      float vv[3] = {v[3 * p], v[3 * p + 1], v[3 * p + 2]};
      kick_drift(xx, vv, a, ck, cd, (float)g.nf);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        x[3 * p + d] = xx[d];
        v[3 * p + d] = vv[d];
      }
    } else {
#pragma unroll
      for (int d = 0; d < 3; ++d) out[3 * p + d] = a[d];
    }
  }
}

// ------------------------------------------------------------ launchers --

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 32) b = 152 * 32;
  return (int)(b < 1 ? 1 : b);
}

// Particles per lane of the deposits: 8 (256 consecutive particles share a
// box) from 2.5M particles, where every resident warp gets two groups; below
// that 2, so that the groups spread evenly (2.1M particles in random order on
// 128^3: 80 us with 8, 76 us with 2).
constexpr int64_t kDepWide = (int64_t)152 * 32 * 512;

template <typename Acc>
static cudaError_t deposit_launch(const float* x, int64_t n, float m, long long M, float scale, const Geo& g, Acc* rho_c,
                                  Acc* rho_f, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (n >= kDepWide) k_deposit<Acc, 8><<<grid_for(n, kDepThreads * 8), kDepThreads, 0, st>>>(x, n, m, M, scale, g, rho_c, rho_f);
  else k_deposit<Acc, 2><<<grid_for(n, kDepThreads * 2), kDepThreads, 0, st>>>(x, n, m, M, scale, g, rho_c, rho_f);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_deposit(const float* x, int64_t n, float m, const Geo& g, float* rho_c, float* rho_f, cudaStream_t st) {
  // a group of 256 particles stays below 2^30 units: unit <= 2^-21 |m|, at least 2^-120
  float scale = 0.f;
  const float am = fabsf(m);
  if (am > 0.f && am < 1e30f) {
    int e = 0;
    frexpf(am, &e);                       // am < 2^e
    scale = ldexpf(1.f, 22 - e < 120 ? 22 - e : 120);
  }
  return deposit_launch<float>(x, n, m, 0, scale, g, rho_c, rho_f, st);
}

cudaError_t launch_deposit_fixed(const float* x, int64_t n, long long M, const Geo& g, long long* rho_c,
                                 long long* rho_f, cudaStream_t st) {
  // 256 particles of a warp, corner terms of at most |M| + 1: the upper words
  // sum to at most 256 (|M| / 2^16 + 1) < 2^31 for |M| < 2^38
  const float scale = M > -(1ll << 38) && M < (1ll << 38) ? 1.f : 0.f;
  return deposit_launch<long long>(x, n, 0.f, M, scale, g, rho_c, rho_f, st);
}

cudaError_t launch_deposit_weights(const float* x, int64_t n, const float* w, int nw, const Geo& g, float* out,
                                  cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (n >= kDepWide) k_deposit_weights<8><<<grid_for(n, kDepThreads * 8), kDepThreads, 0, st>>>(x, n, w, nw, g, out);
  else k_deposit_weights<2><<<grid_for(n, kDepThreads * 2), kDepThreads, 0, st>>>(x, n, w, nw, g, out);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_decompress(const PCodes& in, const int64_t* off, const Geo& g, float* x, float* v, cudaStream_t st) {
  if (in.n == 0) return cudaSuccess;
  k_decompress<<<grid_for(in.n, kDecChunk), kDecThreads, 0, st>>>(in, off, g, x, v);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_interleave(const float* acc, int64_t n3, float4* out, cudaStream_t st) {
  k_interleave<<<grid_for(n3, 256), 256, 0, st>>>(acc, n3, out);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_interpolate(const float* x, int64_t n, const Geo& g, const float* acc_c, const float* acc_f,
                               const float4* acc4, float* a, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_interpolate<false><<<grid_for(n, 256), 256, 0, st>>>(const_cast<float*>(x), nullptr, n, g, acc_c, acc_f, acc4, 0.f,
                                                         0.f, a);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_kick_drift(float* x, float* v, int64_t n, const Geo& g, const float* acc_c, const float* acc_f,
                              const float4* acc4, float ck, float cd, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_interpolate<true><<<grid_for(n, 256), 256, 0, st>>>(x, v, n, g, acc_c, acc_f, acc4, ck, cd, nullptr);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pm
