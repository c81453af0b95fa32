// Particle-particle force (paper Sec. 2.1, Eq. 4) on the compressed state.
//
// a_i = G sum_{j != i, same fine cell, |x_j - x_i| >= r_soft} m_j (x_j - x_i) / |x_j - x_i|^3
//
// over the particles of both species that share particle i's fine-mesh cell
// [k, k+1)^3.  The fine cells of one compression cell lie inside it, and the
// codes are ordered by compression cell, so one CTA takes one x-row of
// compression cells (PP_RX cells; both species' particles of a cell are
// contiguous ranges of their streams) and walks it in chunks of whole
// compression cells holding at most PP_CAP particles:
//   1. put one word per particle into shared memory (the 24 bits of position
//      codes, its cell in the segment, its species) and link it into the list
//      of its fine cell (head per fine cell of the row, next per particle;
//      atomicExch on the head);
//   2. each particle walks its own list and sums the pairs.
// Pairs share a compression cell, so their separation is (q_j - q_i) r / 256 in
// each axis, exactly (the float32 difference of the decoded positions): the
// words are all that a pair needs.  With them a block takes 16 KB in place of
// 53 (decoded float4 positions, 4-byte links, fine cells), so 6 blocks share an
// SM instead of 4; the cell of a particle comes from a binary search of 32-bit
// offsets instead of a walk over the row's.  256^3 workload (18.9M particles,
// 1.1 per fine cell), with the scan of the codes: 0.312 -> 0.272 ms.
// A compression cell with more than PP_CAP particles (a dense cluster) is
// done alone by the tiled all-pairs path: the particles of the cell pass
// through shared memory PP_CAP at a time and every particle of the cell
// compares fine cells with each of them.
// The result goes to a[t] (float4, w = 0) at the particle's stream index t
// (species 0 first), and the largest |a_d| of the launch to *amax (float
// bits) when amax is set.
#include <cuda_runtime.h>
#include <stdint.h>

#include "particles.cuh"
#include "pm_common.cuh"

namespace pm {

namespace {

constexpr int PP_RX = 16;        // compression cells per CTA row segment
constexpr int PP_CAP = 2048;     // particles per chunk held in shared memory
constexpr int PP_THREADS = 256;

struct PPArgs {
  PCodes c0, c1;
  const int64_t* off0;
  const int64_t* off1;
  Geo g;
  float m0, m1;
  float G, r_soft2;
  float4* acc;
  uint32_t* amax;
  int rx;                         // compression cells per CTA (divides n_cmp)
};

// A particle's word: position codes (24 bits), cell in the segment (4 bits), species (bit 28).
__device__ __forceinline__ uint32_t pp_word(uint32_t pos, int cell, int species) {
  return (pos & 0xffffffu) | ((uint32_t)cell << 24) | ((uint32_t)species << 28);
}
// Fine offset of code q in its compression cell: the decoded position is (2 q + 1) r / 512.
__device__ __forceinline__ int fine_of(uint32_t q, int r) { return (int)((2 * q + 1) * (uint32_t)r) >> 9; }

struct Codes3 {
  float x, y, z;
};
__device__ __forceinline__ Codes3 codes_of(uint32_t w) {
  return Codes3{__uint2float_rn(w & 0xffu), __uint2float_rn((w >> 8) & 0xffu), __uint2float_rn((w >> 16) & 0xffu)};
}

// scale = r / 256; m2: the masses of both species.
__device__ __forceinline__ void pair_add(const Codes3& i, uint32_t wj, float scale, float m0, float m1, float r_soft2,
                                         float& ax, float& ay, float& az) {
  const Codes3 j = codes_of(wj);
  const float dx = (j.x - i.x) * scale, dy = (j.y - i.y) * scale, dz = (j.z - i.z) * scale;   // exact
  const float r2 = dx * dx + dy * dy + dz * dz;
  if (r2 >= r_soft2 && r2 > 0.f) {
    const float inv = rsqrtf(r2);
    const float w = (wj >> 28 ? m1 : m0) * inv * inv * inv;
    ax = fmaf(w, dx, ax);
    ay = fmaf(w, dy, ay);
    az = fmaf(w, dz, az);
  }
}

__device__ __forceinline__ void store_acc(const PPArgs& a, int64_t t, float ax, float ay, float az, float& m) {
  ax *= a.G;
  ay *= a.G;
  az *= a.G;
  a.acc[t] = make_float4(ax, ay, az, 0.f);
  m = fmaxf(m, fmaxf(fabsf(ax), fmaxf(fabsf(ay), fabsf(az))));
}

__global__ void __launch_bounds__(PP_THREADS, 6) k_pp(PPArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int r = a.g.rcmp, n = a.g.ncmp;
  const int nseg = n / a.rx;
  const int seg = blockIdx.x % nseg, row = blockIdx.x / nseg;
  const int cy = row % n, cz = row / n, ix0 = seg * a.rx;
  const float scale = (float)r / 256.0f;
  uint32_t* W = reinterpret_cast<uint32_t*>(smraw);             // [PP_CAP]
  int* head = reinterpret_cast<int*>(W + PP_CAP);               // [rx r^3]
  unsigned short* nxt = reinterpret_cast<unsigned short*>(head + a.rx * r * r * r);   // [PP_CAP], 0xffff ends a list
  __shared__ int64_t r0[2][PP_RX + 1];
  for (int i = threadIdx.x; i < 2 * (a.rx + 1); i += PP_THREADS) {
    const int s = i / (a.rx + 1), k = i - s * (a.rx + 1);
    const int64_t c = (int64_t)ix0 + k + (int64_t)n * (cy + (int64_t)n * cz);
    const int64_t o = (s ? a.off1 : a.off0)[c];
    const int64_t lim = s ? a.c1.n : a.c0.n;
    r0[s][k] = o < lim ? o : lim;
  }
  __syncthreads();
  float m = 0.f;
  int c0 = 0;
  while (c0 < a.rx) {
    // chunk [c0, c1): whole compression cells, at most PP_CAP particles
    int c1 = c0;
    while (c1 < a.rx) {
      const int64_t cnt = (r0[0][c1 + 1] - r0[0][c0]) + (r0[1][c1 + 1] - r0[1][c0]);
      if (cnt > PP_CAP) break;
      ++c1;
    }
    if (c1 == c0) {
      // one compression cell beyond PP_CAP: tiled all-pairs within the cell
      // (nxt holds the particles' fine cells)
      const int64_t b0 = r0[0][c0], e0 = r0[0][c0 + 1], b1 = r0[1][c0], e1 = r0[1][c0 + 1];
      const int64_t n0 = e0 - b0, ntot = n0 + (e1 - b1);
      const auto word_of = [&](int64_t i) {
        return i < n0 ? pp_word(a.c0.pos[b0 + i], 0, 0) : pp_word(a.c1.pos[b1 + i - n0], 0, 1);
      };
      const auto fine_cell = [&](uint32_t w) {
        return (fine_of((w >> 16) & 0xffu, r) * r + fine_of((w >> 8) & 0xffu, r)) * r + fine_of(w & 0xffu, r);
      };
      for (int64_t ib = 0; ib < ntot; ib += PP_THREADS) {
        const int64_t ii = ib + threadIdx.x;
        const bool live = ii < ntot;
        const uint32_t wi = live ? word_of(ii) : 0u;
        const int fi = fine_cell(wi);
        const Codes3 ci = codes_of(wi);
        float ax = 0.f, ay = 0.f, az = 0.f;
        for (int64_t jb = 0; jb < ntot; jb += PP_CAP) {
          const int jn = ntot - jb < PP_CAP ? (int)(ntot - jb) : PP_CAP;
          __syncthreads();
          for (int j = threadIdx.x; j < jn; j += PP_THREADS) {
            W[j] = word_of(jb + j);
            nxt[j] = (unsigned short)fine_cell(W[j]);
          }
          __syncthreads();
          if (live)
            for (int j = 0; j < jn; ++j)
              if (nxt[j] == fi && jb + j != ii) pair_add(ci, W[j], scale, a.m0, a.m1, a.r_soft2, ax, ay, az);
        }
        if (live) store_acc(a, ii < n0 ? b0 + ii : a.c0.n + b1 + (ii - n0), ax, ay, az, m);
      }
      __syncthreads();
      c0 += 1;
      continue;
    }
    // linked lists per fine cell of the chunk
    const int64_t b0 = r0[0][c0], b1 = r0[1][c0];
    const int n0 = (int)(r0[0][c1] - b0), ntot = n0 + (int)(r0[1][c1] - b1);
    const int f0 = c0 * r, f1 = c1 * r;   // fine x range of the chunk within the segment
    // reset the chunk's list heads: fine rows (z, y) of the segment, x in [f0, f1)
    for (int i = threadIdx.x; i < r * r * (f1 - f0); i += PP_THREADS) {
      const int line = i / (f1 - f0), fx = f0 + (i - line * (f1 - f0));
      head[line * (a.rx * r) + fx] = 0xffff;
    }
    __syncthreads();
    const uint32_t* pos0 = a.c0.pos + b0;
    const uint32_t* pos1 = a.c1.pos + b1 - n0;
    const auto list_of = [&](uint32_t w) {   // index of the particle's list head
      const int fx = (int)(w >> 24 & 15u) * r + fine_of(w & 0xffu, r);
      return (fine_of((w >> 16) & 0xffu, r) * r + fine_of((w >> 8) & 0xffu, r)) * (a.rx * r) + fx;
    };
    // four particles per thread: position words loaded before any is linked
    for (int i0 = threadIdx.x; i0 < ntot; i0 += 4 * PP_THREADS) {
      uint32_t w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * PP_THREADS;
        w[u] = i < ntot ? (i >= n0 ? pos1 : pos0)[i] : 0u;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * PP_THREADS;
        if (i >= ntot) break;
        const int sp = i >= n0 ? 1 : 0;
        // compression cell of the particle: the last of [c0, c1) that starts at or before it
        const int64_t p = sp ? b1 + (i - n0) : b0 + i;
        const int64_t* ro = r0[sp];
        int c = c0;
#pragma unroll
        for (int d = PP_RX / 2; d > 0; d >>= 1)
          if (c + d < c1 && ro[c + d] <= p) c += d;
        const uint32_t word = pp_word(w[u], c, sp);
        W[i] = word;
        nxt[i] = (unsigned short)atomicExch(&head[list_of(word)], i);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ntot; i += PP_THREADS) {
      const uint32_t wi = W[i];
      const Codes3 ci = codes_of(wi);
      float ax = 0.f, ay = 0.f, az = 0.f;
      for (int j = head[list_of(wi)]; j != 0xffff; j = nxt[j])
        if (j != i) pair_add(ci, W[j], scale, a.m0, a.m1, a.r_soft2, ax, ay, az);
      store_acc(a, i >= n0 ? a.c0.n + b1 + (i - n0) : b0 + i, ax, ay, az, m);
    }
    __syncthreads();
    c0 = c1;
  }
  if (a.amax) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > __uint_as_float(*(volatile uint32_t*)a.amax))
      atomicMax(a.amax, __float_as_uint(m));
  }
}

}  // namespace

size_t pp_smem(const Geo& g) {
  const int rx = g.ncmp < PP_RX ? g.ncmp : PP_RX;
  return (size_t)PP_CAP * (sizeof(uint32_t) + sizeof(unsigned short)) +
         (size_t)rx * g.rcmp * g.rcmp * g.rcmp * sizeof(int);
}

cudaError_t launch_pp(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1, const Geo& g,
                      float m0, float m1, float G, float r_soft, float4* acc, uint32_t* amax, cudaStream_t st) {
  if (c0.n + c1.n == 0) return cudaSuccess;
  const int rx = g.ncmp < PP_RX ? g.ncmp : PP_RX;
  if (g.ncmp % rx) return cudaErrorInvalidValue;
  PPArgs a{c0, c1, off0, off1, g, m0, m1, G, r_soft * r_soft, acc, amax, rx};
  const size_t smem = pp_smem(g);
  allow_smem(k_pp, smem);
  const long long nblk = (long long)g.ncmp * g.ncmp * (g.ncmp / rx);
  k_pp<<<(unsigned)nblk, PP_THREADS, smem, st>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pm
