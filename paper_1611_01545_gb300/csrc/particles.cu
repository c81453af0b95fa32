// Particle-side kernels of the PM step:
//   * compress of one species (Sec. 2.4; decompress and the kernels over
//     float particles are in plain.cu);
//   * the fused decode + deposit that reads the codes directly (binned in
//     shared memory per block of compression cells; the other fused pass,
//     interpolate + kick + drift + recompress, is in kick.cu).
#include <cuda_runtime.h>
#include <stdint.h>

#include "blocks.cuh"
#include "cic.cuh"
#include "particles.cuh"

namespace pm {

// ------------------------------------------------ recompress passes ------

// Warp-aggregated count / rank of a cell key; key 0xffffffff = inactive lane.
__device__ __forceinline__ void count_cell(uint32_t* counts, uint32_t key) {
  unsigned peers = __match_any_sync(0xffffffffu, key);
  int leader = __ffs(peers) - 1;
  if (key != 0xffffffffu && (threadIdx.x & 31) == leader) atomicAdd(counts + key, (unsigned)__popc(peers));
}
__device__ __forceinline__ uint32_t take_rank(uint32_t* counts, uint32_t key) {
  unsigned peers = __match_any_sync(0xffffffffu, key);
  int lane = threadIdx.x & 31;
  int leader = __ffs(peers) - 1;
  unsigned old = 0;
  if (key != 0xffffffffu && lane == leader) old = atomicSub(counts + key, (unsigned)__popc(peers));
  old = __shfl_sync(0xffffffffu, old, leader);
  unsigned below = __popc(peers & ((1u << lane) - 1u));
  return old - (unsigned)__popc(peers) + below;
}

__device__ __forceinline__ void write_codes(PCodesOut o, int64_t dst, const float x[3], const float v[3], float inv_r,
                                            int ncmp, float s, bool vzero) {
  const int half = o.vel16 ? 32768 : 128;
  int q[3], qv[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    int c;
    encode_pos(x[d], inv_r, ncmp, c, q[d]);
    qv[d] = encode_vel(v[d], s, half, vzero);
  }
  o.pos[dst] = (uint32_t)q[0] | ((uint32_t)q[1] << 8) | ((uint32_t)q[2] << 16);
  store_vel(o.vel, o.vel16, dst, qv);
}

__device__ __forceinline__ uint32_t cell_key(const float x[3], float inv_r, int ncmp) {
  int c[3], q;
#pragma unroll
  for (int d = 0; d < 3; ++d) encode_pos(x[d], inv_r, ncmp, c[d], q);
  return (uint32_t)(c[0] + ncmp * (c[1] + ncmp * c[2]));
}

// pm_compress passes over float input.  MODE 0: count cells (+ v_max); MODE 1: scatter codes.
template <int MODE>
__global__ void k_compress_pass(const float* x, const float* v, int64_t n, Geo g, uint32_t* counts,
                                uint32_t* vmax_bits, const float* vmax_in, const int64_t* off, PCodesOut o,
                                int* status) {
  const float inv_r = 1.0f / (float)g.rcmp;
  const float nf = (float)g.nf;
  float vm = 0.f, s = 0.f;
  bool vzero = false;
  if (MODE == 1) {
    vm = *o.vmax;
    vzero = !(vm > 0.f);
    s = vzero ? 0.f : __fdiv_rn(o.vel16 ? 32768.0f : 128.0f, vm);
  }
  float local_max = 0.f;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nround = ((n + stride - 1) / stride) * stride;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nround; p += stride) {
    uint32_t key = 0xffffffffu;
    float xx[3], vv[3];
    if (p < n) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        xx[d] = x[3 * p + d];
        vv[d] = v[3 * p + d];
        local_max = fmaxf(local_max, fabsf(vv[d]));
      }
      bool ok = xx[0] >= 0.f && xx[0] < nf && xx[1] >= 0.f && xx[1] < nf && xx[2] >= 0.f && xx[2] < nf;
      if (ok) key = cell_key(xx, inv_r, g.ncmp);
      else if (MODE == 0) atomicOr(status, ST_RANGE);
    }
    if (MODE == 0) {
      count_cell(counts, key);
    } else {
      uint32_t r = take_rank(counts, key);
      if (key != 0xffffffffu) {
        int64_t dst = off[key] + r;
        if (dst < n && r < 0x80000000u) write_codes(o, dst, xx, vv, inv_r, g.ncmp, s, vzero);
        else atomicOr(status, ST_CORRUPT);
      }
    }
  }
  if (MODE == 0 && vmax_in == nullptr) block_vmax(local_max, vmax_bits);
}

// --------------------------------------------- fused passes over codes ----

__device__ __forceinline__ void smem_acc(long long* a, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(a), (unsigned long long)v);
}
__device__ __forceinline__ void smem_acc(float* a, float v) { atomicAdd(a, v); }
__device__ __forceinline__ void global_add(float* a, float v) { atomicAdd(a, v); }
__device__ __forceinline__ void global_add(long long* a, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(a), (unsigned long long)v);
}

// Mass of each CIC corner: float mode m w_x w_y w_z in float32; fixed mode
// the conservative integer split of the fixed-point deposit (2^-32 units).
__device__ __forceinline__ void corner_masses(float m, long long, const float w1[3], float out[8]) {
  float w0[3] = {__fsub_rn(1.f, w1[0]), __fsub_rn(1.f, w1[1]), __fsub_rn(1.f, w1[2])};
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    float w = __fmul_rn(__fmul_rn(dx ? w1[0] : w0[0], dy ? w1[1] : w0[1]), dz ? w1[2] : w0[2]);
    out[c] = __fmul_rn(m, w);
  }
}
__device__ __forceinline__ void corner_masses(float, long long M, const float w1[3], long long out[8]) {
  long long a1[3] = {(long long)__fmul_rn(w1[0], 1048576.0f), (long long)__fmul_rn(w1[1], 1048576.0f),
                     (long long)__fmul_rn(w1[2], 1048576.0f)};
  fixed_corners(M, a1, out);
}

// Decode + deposit of both species for one cell block, binned in shared memory
// (32-bit fixed point with a per-block power-of-two scale, converted to
// float32 before the flush; or int64 in units of 2^-32 mass for the
// fixed-point mode) and flushed once per cell.  smem: row offsets (2 species), fine region
// (RX r + 1)(RY r + 1)(RZ r + 1), coarse region (RX + 1)(RY + 1)(RZ + 1).
// Threads per CTA of the deposit.
#ifndef PM_DEPOSIT_THREADS
#define PM_DEPOSIT_THREADS 256
#endif

// Register budget of the deposit: resident CTAs per SM it is compiled for
// (6: 40 registers; measured 0.391 -> 0.347 ms against the compiler's own
// allocation on the 256^3 workload; the int64 mode keeps 4).  0 keeps the
// compiler's allocation.
#ifndef PM_DEPOSIT_MINB
#define PM_DEPOSIT_MINB 6
#endif
#if PM_DEPOSIT_MINB > 0
#define PM_DEPOSIT_BOUNDS __launch_bounds__(PM_DEPOSIT_THREADS, sizeof(Acc) == 4 ? PM_DEPOSIT_MINB : 4)
#else
#define PM_DEPOSIT_BOUNDS
#endif
template <typename Acc>
__global__ void PM_DEPOSIT_BOUNDS k_deposit_codes(PCodes c0, PCodes c1, const int64_t* off0, const int64_t* off1, Geo g, Blk bk,
                                float m0, float m1, long long M0, long long M1, Acc* rho_c, Acc* rho_f) {
  extern __shared__ __align__(16) unsigned char smraw[];
  for_each_block(bk, [&](const int bid) {
    const int r = g.rcmp;
    const int fx = bk.RX * r + 1, fy = bk.RY * r + 1, fz = bk.RZ * r + 1;
    const int cx = bk.RX + 1, cy = bk.RY + 1, cz = bk.RZ + 1;
    const int nrow = bk.RY * bk.RZ;
    int64_t* roff = reinterpret_cast<int64_t*>(smraw);
    Acc* sf = reinterpret_cast<Acc*>(roff + 2 * nrow * (bk.RX + 1));
    Acc* sc = sf + fx * fy * fz;
    // Coarse density: the int64 mode deposits each particle's 8 coarse corners
    // (exact, order independent); the float mode restricts the block's fine
    // tile onto the coarse cells it touches when it flushes (CIC restriction
    // is exact and linear, so the blocks' partial sums add up to it).
    const bool dep_coarse = g.two && rho_c != nullptr && sizeof(Acc) == 8;
    const bool restr = g.two && rho_c != nullptr && sizeof(Acc) == 4;
    const int nsf = fx * fy * fz, nsc = dep_coarse ? cx * cy * cz : 0;
    for (int i = threadIdx.x; i < nsf + nsc; i += blockDim.x) sf[i] = (Acc)0;
    const CellBlock cb = block_of(bk, bid);
    load_row_offsets(off0, g, bk, cb, roff);
    load_row_offsets(off1, g, bk, cb, roff + nrow * (bk.RX + 1));
    __syncthreads();
    // Float mode: the block bins its corner masses in 32-bit fixed point
    // (integer shared-memory atomics, several times the rate of float ones,
    // and independent of the order of the adds) with a power-of-two scale S.
    // A fine node receives mass only from particles of the (at most 8)
    // compression cells around it, so 8 x the block's heaviest compression
    // cell bounds every node's total; S = 2^floor(log2(2^31 / bound)) keeps
    // the scaled total below 2^31, and the corner roundings below 2^31 more.
    float S = 1.f;
    if constexpr (sizeof(Acc) == 4) {
      float cm = 0.f;
      const int nrx = bk.RX + 1, ncells = nrow * bk.RX;
      for (int i = threadIdx.x; i < ncells; i += blockDim.x) {
        const int row = i / bk.RX, k = i - row * bk.RX;
        const int64_t* r0 = roff + row * nrx + k;
        const int64_t* r1 = r0 + nrow * nrx;
        const int64_t a0 = r0[0] < c0.n ? r0[0] : c0.n, b0 = r0[1] < c0.n ? r0[1] : c0.n;
        const int64_t a1 = r1[0] < c1.n ? r1[0] : c1.n, b1 = r1[1] < c1.n ? r1[1] : c1.n;
        const float w = __fadd_ru(__fmul_ru((float)(b0 - a0), m0), __fmul_ru((float)(b1 - a1), m1));
        cm = fmaxf(cm, w);
      }
      cm = block_max_all(cm);
      if (cm > 0.f) {
        const float x = fminf(__fdiv_rd(268435456.0f, cm), 1.329228e36f);   // 2^31 / (8 cm), at most 2^120
        S = __uint_as_float(__float_as_uint(x) & 0xff800000u);
      }
    }
    const float pscale = (float)r / 256.0f;
    const int bxf = cb.ix0 * r, byf = cb.iy0 * r, bzf = cb.iz0 * r;
    for (int s = 0; s < 2; ++s) {
      const PCodes& cs = s ? c1 : c0;
      // float mode: the species mass times the block's power-of-two scale
      // (exact), so a corner's fixed-point value is rint(m S w)
      const float m = sizeof(Acc) == 4 ? __fmul_rn(s ? m1 : m0, S) : (s ? m1 : m0);
      const long long M = s ? M1 : M0;
      const int64_t* ro_s = roff + s * nrow * (bk.RX + 1);
      for (int row = 0; row < nrow; ++row) {
        const int64_t* ro = ro_s + row * (bk.RX + 1);
        const int iy = cb.iy0 + row % bk.RY, iz = cb.iz0 + row / bk.RY;
        // A corrupt stream (flagged by the scan) may claim more particles than
        // exist; never read past the caller's n records.
        const int64_t p0 = ro[0] < cs.n ? ro[0] : cs.n;
        const int64_t p1 = ro[bk.RX] < cs.n ? ro[bk.RX] : cs.n;
        const int64_t rounds = (p1 - p0 + blockDim.x - 1) / blockDim.x;
        for (int64_t it = 0; it < rounds; ++it) {
          const int64_t p = p0 + it * blockDim.x + threadIdx.x;
          const bool live = p < p1;
          int ixl = 0;
          float px = 0.f, py = 0.f, pz = 0.f;
          if (live) {
            ixl = row_cell(ro, bk.RX, p);
            int q[3];
            unpack_pos(cs.pos[p], q);
            if (dep_coarse) {
              px = decode_pos(cb.ix0 + ixl, q[0], pscale);
              py = decode_pos(iy, q[1], pscale);
              pz = decode_pos(iz, q[2], pscale);
            }
            // fine CIC in local region coordinates (no wrap inside the block).
            // Decoded positions are exact dyadics, x = c r + (2q + 1) r / 512,
            // so the fine cell and the weight come from the codes in integer
            // arithmetic (the same values as floor(x) and x - floor(x)).
            int num[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) num[d] = (2 * q[d] + 1) * r;
            const int lx = ixl * r + (num[0] >> 9), ly = (iy - cb.iy0) * r + (num[1] >> 9),
                      lz = (iz - cb.iz0) * r + (num[2] >> 9);
            float w1[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) w1[d] = __fmul_rn(__int2float_rn(num[d] & 511), 1.0f / 512.0f);
            Acc t8[8];
            corner_masses(m, M, w1, t8);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
              const int idx = ((lz + dz) * fy + (ly + dy)) * fx + (lx + dx);
              if constexpr (sizeof(Acc) == 4)
                atomicAdd(reinterpret_cast<unsigned int*>(sf) + idx, __float2uint_rn((float)t8[c]));
              else
                smem_acc(&sf[idx], t8[c]);
            }
          }
          if (dep_coarse) {
            // Coarse cell == compression cell (coarse_ratio == cmp_ratio), so every
            // particle of a run shares its 8 coarse corners: sum the run in
            // registers and let its last lane do 8 shared-memory adds.
            Acc cv[8];
            if (live) {
              const float sc_inv = 1.0f / (float)g.rc;
              float ux = __fmul_rn(px, sc_inv), uy = __fmul_rn(py, sc_inv), uz = __fmul_rn(pz, sc_inv);
              float v1[3] = {__fsub_rn(ux, floorf(ux)), __fsub_rn(uy, floorf(uy)), __fsub_rn(uz, floorf(uz))};
              corner_masses(m, M, v1, cv);
            } else {
#pragma unroll
              for (int c = 0; c < 8; ++c) cv[c] = (Acc)0;
            }
            const unsigned key = live ? (unsigned)ixl : 0xffffffffu;
            if (run_reduce<8, Acc>(key, cv) && live) {
              const int kx = ixl, ky = row % bk.RY, kz = row / bk.RY;
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
                smem_acc(&sc[((kz + dz) * cy + (ky + dy)) * cx + (kx + dx)], cv[c]);
              }
            }
          }
        }
      }
    }
    __syncthreads();
    if constexpr (sizeof(Acc) == 4) {
      // fixed point -> float32 (S is a power of two: the scaling is exact)
      const float inv_s = 1.0f / S;
      const unsigned int* si = reinterpret_cast<const unsigned int*>(sf);
      for (int i = threadIdx.x; i < nsf; i += blockDim.x) sf[i] = __fmul_rn(__uint2float_rn(si[i]), inv_s);
      __syncthreads();
    }
    const int nf = g.nf;
    // flush: one warp per region row (z, y), lanes along x
    for (int line = threadIdx.x >> 5; line < fy * fz; line += blockDim.x >> 5) {
      const int lz = line / fy, ly = line - lz * fy;
      int gy = byf + ly, gz = bzf + lz;
      if (gy >= nf) gy -= nf;
      if (gz >= nf) gz -= nf;
      Acc* grow = rho_f + ((int64_t)gz * nf + gy) * nf;
      const Acc* srow = sf + line * fx;
      for (int lx = threadIdx.x & 31; lx < fx; lx += 32) {
        const Acc val = srow[lx];
        if (val == (Acc)0) continue;
        int gx = bxf + lx;
        if (gx >= nf) gx -= nf;
        global_add(grow + gx, val);
      }
    }
    const int nc = g.nc;
    for (int i = threadIdx.x; i < nsc; i += blockDim.x) {
      Acc val = sc[i];
      if (val == (Acc)0) continue;
      int lx = i % cx, ly = (i / cx) % cy, lz = i / (cx * cy);
      int gx = cb.ix0 + lx, gy = cb.iy0 + ly, gz = cb.iz0 + lz;
      if (gx >= nc) gx -= nc;
      if (gy >= nc) gy -= nc;
      if (gz >= nc) gz -= nc;
      global_add(&rho_c[((int64_t)gz * nc + gy) * nc + gx], val);
    }
    if (restr) {
      // rho_c(C) += sum_k w(kx) w(ky) w(kz) tile(r C + k), w(k) = 1 - |k| / r, over the
      // tile's part; coarse cells C = block cell + (0 .. RX, 0 .. RY, 0 .. RZ); separable.
      const float* tile = reinterpret_cast<const float*>(sf);
      float* T1 = reinterpret_cast<float*>(sc) + cx * cy * cz;   // [fz][fy][cx]
      float* T2 = T1 + fz * fy * cx;                             // [fz][cy][cx]
      const float inv = 1.0f / (float)r;
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
      for (int line = warp; line < fz * fy; line += nwarp) {
        const float* row = tile + line * fx;
        for (int q = lane; q < cx; q += 32) {
          float t = 0.f;
          for (int k = 1 - r; k < r; ++k) {
            const int j = r * q + k;
            if (j >= 0 && j < fx) t = fmaf(1.0f - (float)(k < 0 ? -k : k) * inv, row[j], t);
          }
          T1[line * cx + q] = t;
        }
      }
      __syncthreads();
      for (int line = warp; line < fz * cy; line += nwarp) {
        const int lz = line / cy, qy = line - lz * cy;
        for (int q = lane; q < cx; q += 32) {
          float t = 0.f;
          for (int k = 1 - r; k < r; ++k) {
            const int j = r * qy + k;
            if (j >= 0 && j < fy) t = fmaf(1.0f - (float)(k < 0 ? -k : k) * inv, T1[(lz * fy + j) * cx + q], t);
          }
          T2[line * cx + q] = t;
        }
      }
      __syncthreads();
      for (int line = warp; line < cz * cy; line += nwarp) {
        const int qz = line / cy, qy = line - qz * cy;
        int gy = cb.iy0 + qy, gz = cb.iz0 + qz;
        if (gy >= nc) gy -= nc;
        if (gz >= nc) gz -= nc;
        float* crow = reinterpret_cast<float*>(rho_c) + ((int64_t)gz * nc + gy) * nc;
        for (int q = lane; q < cx; q += 32) {
          float t = 0.f;
          for (int k = 1 - r; k < r; ++k) {
            const int j = r * qz + k;
            if (j >= 0 && j < fz) t = fmaf(1.0f - (float)(k < 0 ? -k : k) * inv, T2[(j * cy + qy) * cx + q], t);
          }
          int gx = cb.ix0 + q;
          if (gx >= nc) gx -= nc;
          if (t != 0.f) atomicAdd(crow + gx, t);
        }
      }
    }
  });
}

// ---- deposit of the shapes in use -------------------------------------------
//
// The float deposit for blocks of RX_MAX x RY x RZ compression cells of 4 fine
// cells or shorter in x (the shapes of the defaults and of tuned programs); other
// shapes, ratios and the int64 mode take the kernel above.  Issue bound (74% of
// issue slots), a third of it spent on the block's 1.3 nodes per particle
// rather than on the particles, so:
//   * strides are constants, offsets and indices 32-bit and relative to the
//     cell row, the fine node comes from the code's upper 2 bits and the
//     weight (2 q + 1) / 128 from its lower 6: weights are kept in units of
//     1 / 128, exact in float32, and the scaled mass takes the powers of two;
//   * one walk over the bins converts, adds four nodes at a time to the mesh
//     (16-byte reductions), and forms the x restriction of the coarse density
//     from the same four values and the left neighbour's carry.
// 256^3 workload 0.178 -> 0.118 ms (blocks of 32 x 2 x 1; with its launch 0.192 ->
// 0.130, 64 x 1 x 1 0.125, 32 x 2 x 2 0.177: 5 instead of 6 CTAs per SM and spills),
// 768^3 (5.1e8 particles) 4.56 -> 2.98 ms (3.07 with planes 4 banks apart), clustered 512^3 in its default shape
// 1.71 -> 0.89 ms.
template <int RX_MAX, int RY, int RZ> struct DepShape {
  static constexpr int row = 4 * RX_MAX + 4;          // words per bin row (4 RX + 1 used), whole 16-byte words
  static constexpr int fy = 4 * RY + 1, fz = 4 * RZ + 1, rows = fy * fz;
  // planes start 16 banks apart modulo 32, rows 4: the 4^3 lower nodes of a cell's particles, which the
  // lanes of a warp add to, lie at most 2 deep in a bank
  static constexpr int plane = row * fy + ((16 - row * fy) & 31);
  static constexpr int cx = RX_MAX + 1, cy = RY + 1, cz = RZ + 1;
  static constexpr int lists = RY * RZ;                // cell rows
  // bins, x-restricted rows, xy-restricted rows, relative offsets of both species
  static constexpr size_t smem = 4 * ((size_t)plane * fz + rows * cx + fz * cy * cx + 2 * lists * RX_MAX);
};
// Compile-time tunables: resident CTAs per SM of the deposit.
#ifndef PM_DEPOSIT_ROWS_MINB
#define PM_DEPOSIT_ROWS_MINB 6
#endif

// Weight of the coarse tent at distance k fine cells (ratio 4).
__device__ __forceinline__ float tent4(int k) { return 1.0f - 0.25f * (float)(k < 0 ? -k : k); }

template <int RX_MAX, int RY, int RZ>
__global__ void __launch_bounds__(PM_DEPOSIT_THREADS, PM_DEPOSIT_ROWS_MINB)
    k_deposit_rows(PCodes c0, PCodes c1, const int64_t* off0, const int64_t* off1, Geo g, Blk bk, float m0, float m1,
                   float* rho_c, float* rho_f) {
  using D = DepShape<RX_MAX, RY, RZ>;
  constexpr int T = PM_DEPOSIT_THREADS;
  constexpr uint32_t kSeg = 1u << 30;   // particles of a cell row handled with one set of 32-bit offsets
  extern __shared__ __align__(16) unsigned char smraw[];
  uint32_t* bins = reinterpret_cast<uint32_t*>(smraw);
  float* T1 = reinterpret_cast<float*>(bins + D::plane * D::fz);   // [fz][fy][cx]
  float* T2 = T1 + D::rows * D::cx;                                 // [fz][cy][cx]
  uint32_t* rel = reinterpret_cast<uint32_t*>(T2 + D::fz * D::cy * D::cx);   // [species][list][RX_MAX]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for_each_block(bk, [&](const int bid) {
    const int RX = bk.RX, cx = RX + 1;
    const CellBlock cb = block_of(bk, bid);
    for (int i = threadIdx.x; i < D::plane * D::fz / 4; i += T) reinterpret_cast<uint4*>(bins)[i] = make_uint4(0, 0, 0, 0);
    // Offsets of the block's cell rows and the mass of its heaviest cell: 8
    // times that bounds every node's total (a node receives mass only from the
    // at most 8 compression cells around it), so with the power of two S =
    // 2^floor(log2(2^31 / bound)) the scaled totals stay below 2^31, and the
    // corner roundings below 2^31 more.
    float cm = 0.f;
    for (int i = threadIdx.x; i < D::lists * RX_MAX; i += T) {
      const int l = i / RX_MAX, j = i - l * RX_MAX;
      uint32_t r0 = kSeg, r1 = kSeg;
      if (j < RX) {
        const int64_t c = cb.ix0 + (int64_t)g.ncmp * (cb.iy0 + l % RY + (int64_t)g.ncmp * (cb.iz0 + l / RY));
        const int64_t a0 = off0[c + j], a1 = off1[c + j];
        const int64_t d0 = a0 - off0[c], d1 = a1 - off1[c];
        r0 = d0 < kSeg ? (uint32_t)d0 : kSeg;
        r1 = d1 < kSeg ? (uint32_t)d1 : kSeg;
        const int64_t b0 = off0[c + j + 1], b1 = off1[c + j + 1];
        const int64_t n0 = (b0 < c0.n ? b0 : c0.n) - (a0 < c0.n ? a0 : c0.n);
        const int64_t n1 = (b1 < c1.n ? b1 : c1.n) - (a1 < c1.n ? a1 : c1.n);
        cm = fmaxf(cm, __fadd_ru(__fmul_ru((float)n0, m0), __fmul_ru((float)n1, m1)));
      }
      rel[i] = r0;
      rel[D::lists * RX_MAX + i] = r1;
    }
    cm = block_max_all(cm);   // (its barriers also order the bins and offsets)
    float S = 1.f;
    if (cm > 0.f) {
      const float x = fminf(__fdiv_rd(268435456.0f, cm), 1.329228e36f);   // 2^31 / (8 cm), at most 2^120
      S = __uint_as_float(__float_as_uint(x) & 0xff800000u);
    }
    for (int s = 0; s < 2; ++s) {
      const int64_t n = s ? c1.n : c0.n;
      // corner value m S w_x w_y w_z with weights in units of 1 / 128
      const float m = __fmul_rn(__fmul_rn(s ? m1 : m0, S), 1.0f / 2097152.0f);
      for (int l = 0; l < D::lists; ++l) {
        const int64_t* off = (s ? off1 : off0) + cb.ix0 +
                             (int64_t)g.ncmp * (cb.iy0 + l % RY + (int64_t)g.ncmp * (cb.iz0 + l / RY));
        uint32_t* ro = rel + (s * D::lists + l) * RX_MAX;
        uint32_t* lbins = bins + (l / RY) * 4 * D::plane + (l % RY) * 4 * D::row;
        // a corrupt stream (flagged by the scan) may claim more particles than
        // exist; never read past the caller's n records
        const int64_t o0 = off[0], o1 = off[RX];
        const int64_t p0 = o0 < n ? o0 : n, p1 = o1 < n ? o1 : n;
        for (int64_t seg = p0; seg < p1; seg += kSeg) {
          if (seg > p0) {   // a row of more than 2^30 particles: offsets of its next part
            __syncthreads();
            for (int j = threadIdx.x; j < RX; j += T) {
              const int64_t d = off[j] - seg;
              ro[j] = d <= 0 ? 0u : (d < kSeg ? (uint32_t)d : kSeg);
            }
            __syncthreads();
          }
          const uint32_t count = p1 - seg < kSeg ? (uint32_t)(p1 - seg) : kSeg;
          const uint32_t* pos = (s ? c1.pos : c0.pos) + seg;
          uint32_t next = threadIdx.x < count ? pos[threadIdx.x] : 0u;
          for (uint32_t i = threadIdx.x; i < count; i += T) {
            const uint32_t pw = next;
            if (i + T < count) next = pos[i + T];
            // the last cell whose offset is at most i (entries past the row hold 2^30)
            int k = 0;
#pragma unroll
            for (int d = RX_MAX / 2; d > 0; d >>= 1)
              if (ro[k + d] <= i) k += d;
            const uint32_t hi = (pw >> 6) & 0x030303u, lo = ((pw & 0x3f3f3fu) << 1) | 0x010101u;
            uint32_t* b = lbins + 4 * k + (hi & 3u) + D::row * ((hi >> 8) & 3u) + D::plane * (hi >> 16);
            const float wx1 = __uint2float_rn(lo & 0xffu), wy1 = __uint2float_rn((lo >> 8) & 0xffu),
                        wz1 = __uint2float_rn(lo >> 16);
            const float wx0 = 128.0f - wx1, wy0 = 128.0f - wy1;
            const float mz1 = __fmul_rn(m, wz1), mz0 = __fmul_rn(m, 128.0f - wz1);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float wxy = __fmul_rn(c & 1 ? wx1 : wx0, (c >> 1) & 1 ? wy1 : wy0);   // exact
              atomicAdd(b + (c & 1) + D::row * ((c >> 1) & 1) + D::plane * (c >> 2),
                        __float2uint_rn(__fmul_rn(wxy, c >> 2 ? mz1 : mz0)));
            }
          }
        }
      }
    }
    __syncthreads();
    // One warp per bin row: fixed point -> float32 (S is a power of two: exact),
    // four nodes per lane, to the mesh; the restriction along x on the way,
    // R[q] = sum_k w(k) row[4 q + k].
    const float inv_s = 1.0f / S;
    const int nf = g.nf, bxf = 4 * cb.ix0;
    for (int line = warp; line < D::rows; line += T / 32) {
      const int lz = line / D::fy, ly = line - lz * D::fy;
      int gy = 4 * cb.iy0 + ly, gz = 4 * cb.iz0 + lz;
      if (gy >= nf) gy -= nf;
      if (gz >= nf) gz -= nf;
      float* grow = rho_f + ((int64_t)gz * nf + gy) * nf;
      const uint32_t* row = bins + lz * D::plane + ly * D::row;
      float carry = 0.f;                                  // what the cells left of lane 0 give its coarse cell
      for (int q0 = 0; q0 < RX; q0 += 32) {
        const int q = q0 + lane;
        const bool in = q < RX;
        const uint4 u = in ? reinterpret_cast<const uint4*>(row)[q] : make_uint4(0, 0, 0, 0);
        float4 v;
        v.x = __fmul_rn(__uint2float_rn(u.x), inv_s);
        v.y = __fmul_rn(__uint2float_rn(u.y), inv_s);
        v.z = __fmul_rn(__uint2float_rn(u.z), inv_s);
        v.w = __fmul_rn(__uint2float_rn(u.w), inv_s);
        if ((u.x | u.y | u.z | u.w) != 0u) atomicAdd(reinterpret_cast<float4*>(grow + bxf) + q, v);
        const float up = fmaf(0.75f, v.w, fmaf(0.5f, v.z, 0.25f * v.y));          // for the coarse cell to the right
        const float own = fmaf(0.25f, v.w, fmaf(0.5f, v.z, fmaf(0.75f, v.y, v.x)));
        float left = __shfl_up_sync(0xffffffffu, up, 1);
        if (lane == 0) left = carry;
        if (in) T1[line * D::cx + q] = own + left;
        carry = __shfl_sync(0xffffffffu, up, RX - q0 < 32 ? RX - 1 - q0 : 31);
      }
      if (lane == 0) {                                    // the upper halo node
        const float v = __fmul_rn(__uint2float_rn(row[4 * RX]), inv_s);
        const int gx = bxf + 4 * RX == nf ? 0 : bxf + 4 * RX;
        if (v != 0.f) atomicAdd(grow + gx, v);
        T1[line * D::cx + RX] = v + carry;
      }
    }
    if (!rho_c) return;
    __syncthreads();
    for (int i = threadIdx.x; i < D::fz * D::cy * D::cx; i += T) {
      const int q = i % D::cx, qy = i / D::cx % D::cy, lz = i / (D::cx * D::cy);
      if (q >= cx) continue;
      float t = 0.f;
#pragma unroll
      for (int k = -3; k <= 3; ++k) {
        const int j = 4 * qy + k;
        if (j >= 0 && j < D::fy) t = fmaf(tent4(k), T1[(lz * D::fy + j) * D::cx + q], t);
      }
      T2[i] = t;
    }
    __syncthreads();
    const int nc = g.nc;
    for (int i = threadIdx.x; i < D::cz * D::cy * D::cx; i += T) {
      const int q = i % D::cx, qy = i / D::cx % D::cy, qz = i / (D::cx * D::cy);
      if (q >= cx) continue;
      float t = 0.f;
#pragma unroll
      for (int k = -3; k <= 3; ++k) {
        const int j = 4 * qz + k;
        if (j >= 0 && j < D::fz) t = fmaf(tent4(k), T2[(j * D::cy + qy) * D::cx + q], t);
      }
      int gx = cb.ix0 + q, gy = cb.iy0 + qy, gz = cb.iz0 + qz;
      if (gx >= nc) gx -= nc;
      if (gy >= nc) gy -= nc;
      if (gz >= nc) gz -= nc;
      if (t != 0.f) atomicAdd(rho_c + ((int64_t)gz * nc + gy) * nc + gx, t);
    }
  });
}

template <int RX_MAX, int RY, int RZ>
static void launch_rows(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1, const Geo& g,
                        const Blk& bk, float m0, float m1, float* rho_c, float* rho_f, cudaStream_t st) {
  const auto k = k_deposit_rows<RX_MAX, RY, RZ>;
  constexpr size_t smem = DepShape<RX_MAX, RY, RZ>::smem;
  allow_smem(k, smem);
  k<<<block_grid(k, bk, PM_DEPOSIT_THREADS, smem), PM_DEPOSIT_THREADS, smem, st>>>(c0, c1, off0, off1, g, bk, m0, m1,
                                                                                   g.two ? rho_c : nullptr, rho_f);
}

// ------------------------------------------------------------ launchers --

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 32) b = 152 * 32;
  return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_compress(const float* x, const float* v, int64_t n, const Geo& g, uint32_t* counts,
                            uint32_t* vmax_bits, const float* vmax_in, int64_t* off, pm_codes_t& out, bool vel16,
                            void* scan_state, int* status, cudaStream_t st) {
  PCodesOut o{reinterpret_cast<uint32_t*>(out.pos), out.vel, out.vmax, vel16};
  cudaMemsetAsync(vmax_bits, 0, sizeof(uint32_t), st);
  int grid = grid_for(n > 0 ? n : 1, 256);
  k_compress_pass<0><<<grid, 256, 0, st>>>(x, v, n, g, counts, vmax_bits, vmax_in, off, o, status);
  const uint32_t* vsrc = vmax_in ? reinterpret_cast<const uint32_t*>(vmax_in) : vmax_bits;
  cudaError_t e = scan_counts(counts, g.ncell, n, off, out, vsrc, scan_state, status, st);
  if (e != cudaSuccess) return e;
  k_compress_pass<1><<<grid, 256, 0, st>>>(x, v, n, g, counts, vmax_bits, vmax_in, off, o, status);
  note_launches(2);
  return cudaGetLastError();
}

size_t deposit_codes_smem(const Geo& g, const Blk& bk, bool fixed) {
  size_t nrow = (size_t)bk.RY * bk.RZ;
  size_t fine = (size_t)(bk.RX * g.rcmp + 1) * (bk.RY * g.rcmp + 1) * (bk.RZ * g.rcmp + 1);
  size_t coarse = g.two ? (size_t)(bk.RX + 1) * (bk.RY + 1) * (bk.RZ + 1) : 0;
  // float two-level: room for the restriction's x and y partial sums
  size_t restr = (g.two && !fixed) ? ((size_t)(bk.RZ * g.rcmp + 1) * ((bk.RY * g.rcmp + 1) + (bk.RY + 1)) *
                                      (bk.RX + 1)) : 0;
  return 2 * nrow * (bk.RX + 1) * sizeof(int64_t) + (fine + coarse) * (fixed ? 8 : 4) + restr * 4;
}

cudaError_t launch_deposit_codes(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1,
                                 const Geo& g, const Blk& bk, float m0, float m1, long long M0, long long M1,
                                 void* rho_c, void* rho_f, bool fixed, cudaStream_t st) {
  const size_t smem = deposit_codes_smem(g, bk, fixed);
  // the row kernel adds 16-byte words to the mesh: its base must be aligned (its rows are, nf = 4 n_cmp)
  const bool rows = !fixed && g.rcmp == 4 && (!g.two || g.rc == 4) && (reinterpret_cast<uintptr_t>(rho_f) & 15) == 0;
  float* rc = static_cast<float*>(rho_c);
  float* rf = static_cast<float*>(rho_f);
  if (rows && bk.RX <= 64 && bk.RY == 1 && bk.RZ == 1) {
    launch_rows<64, 1, 1>(c0, c1, off0, off1, g, bk, m0, m1, rc, rf, st);
  } else if (rows && bk.RX <= 32 && bk.RY == 2 && bk.RZ == 1) {
    launch_rows<32, 2, 1>(c0, c1, off0, off1, g, bk, m0, m1, rc, rf, st);
  } else if (fixed) {
    const auto k = k_deposit_codes<long long>;
    allow_smem(k, smem);
    k<<<block_grid(k, bk, PM_DEPOSIT_THREADS, smem), PM_DEPOSIT_THREADS, smem, st>>>(
        c0, c1, off0, off1, g, bk, m0, m1, M0, M1, static_cast<long long*>(rho_c), static_cast<long long*>(rho_f));
  } else {
    const auto k = k_deposit_codes<float>;
    allow_smem(k, smem);
    k<<<block_grid(k, bk, PM_DEPOSIT_THREADS, smem), PM_DEPOSIT_THREADS, smem, st>>>(c0, c1, off0, off1, g, bk, m0, m1,
                                                                                     M0, M1, rc, rf);
  }
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pm
