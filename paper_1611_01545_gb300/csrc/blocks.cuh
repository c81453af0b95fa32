// Cell blocks of the fused passes (deposit, kick): block order, persistent
// draws, row offsets, the new-cell window and block maxima.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "particles.cuh"

namespace pm {

// Block of compression cells handled by one CTA: x cells [bx*RX, +RX), rows y [by*RY, +RY), z [bz*RZ, +RZ).
struct CellBlock {
  int ix0, iy0, iz0;
};
// Blocks are handed out x fastest, then in bricks of bk.brick x bk.brick
// (y, z) block rows (the host picks bricks for large meshes, see
// block_brick), so that the blocks running at the same time cover a compact
// region: the partial writes that neighbouring blocks make to the same
// cells (new-cell ranges of the recompressed codes, fine density halos)
// then meet in L2 before the lines are evicted.
__device__ __forceinline__ CellBlock block_of(const Blk& bk, int bid) {
  const int nbx = bk.nbx, nby = bk.nby;
  const int bx = bid % nbx, r = bid / nbx;
  int by, bz;
  const int B = bk.brick;
  if (B > 1) {
    const int in = r % (B * B), brick = r / (B * B);
    const int nyb = nby / B;
    by = (brick % nyb) * B + in % B;
    bz = (brick / nyb) * B + in / B;
  } else {
    by = r % nby;
    bz = r / nby;
  }
  return CellBlock{bx * bk.RX, by * bk.RY, bz * bk.RZ};
}

// Runs body(bid) for the cell blocks of this CTA: its own block (one CTA per
// cell block), or, when bk.work is set (persistent launch), blocks drawn one
// at a time from the device counter *bk.work until all are taken, so that
// CTAs that drew light blocks take more of them.  body must use __syncthreads
// uniformly; the barrier before each draw keeps the next block's shared-memory
// set-up from overlapping the previous block's flush.
template <class F>
__device__ __forceinline__ void for_each_block(const Blk& bk, F&& body) {
  if (!bk.work) {
    body((int)blockIdx.x);
    return;
  }
  __shared__ int s_bid;
  const int nblk = bk.nbx * bk.nby * bk.nbz;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_bid = atomicAdd(bk.work, 1);
    __syncthreads();
    const int bid = s_bid;
    if (bid >= nblk) break;
    body(bid);
  }
}

// Loads the CSR offsets of the block's rows into smem: roff[r*(RX+1) + i], r = row (y fastest).
__device__ __forceinline__ void load_row_offsets(const int64_t* off, const Geo& g, const Blk& bk, CellBlock cb,
                                                 int64_t* roff) {
  const int nrow = bk.RY * bk.RZ;
  for (int i = threadIdx.x; i < nrow * (bk.RX + 1); i += blockDim.x) {
    int r = i / (bk.RX + 1), k = i - r * (bk.RX + 1);
    int iy = cb.iy0 + r % bk.RY, iz = cb.iz0 + r / bk.RY;
    int64_t c = (int64_t)cb.ix0 + k + (int64_t)g.ncmp * (iy + (int64_t)g.ncmp * iz);
    roff[i] = off[c];
  }
}

// Index (0..RX-1) of the cell of stream index p within a row's offsets ro[0..RX].
__device__ __forceinline__ int row_cell(const int64_t* ro, int RX, int64_t p) {
  int lo = 0, hi = RX - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (ro[mid] <= p) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// 4-byte global -> shared copy that does not stall the issuing thread
// (cp.async); async_copies_wait() waits for all of the thread's copies.
__device__ __forceinline__ void copy_async4(float* smem_dst, const float* gmem_src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void async_copies_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Block maximum of values m >= 0, returned to every thread.  Every thread of
// the block must call it.
__device__ __forceinline__ float block_max_all(float m) {
  __shared__ float red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __syncthreads();   // red may still be read by a previous call
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  float r = 0.f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmaxf(r, red[w]);
  return r;
}

// Block maximum of m into *vmax_bits (float bits of a value >= 0): one atomic
// per block, and none when the block's maximum does not exceed the current
// value.  Every thread of the block must call it.
__device__ __forceinline__ void block_vmax(float m, uint32_t* vmax_bits) {
  __shared__ float red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __syncthreads();   // red may still be read by a previous call
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
    if (m > 0.f && m > __uint_as_float(*(volatile uint32_t*)vmax_bits)) atomicMax(vmax_bits, __float_as_uint(m));
  }
}

// Grid of a cell-block launch: one CTA per block, or (bk.work set) as many
// CTAs as fit on the device at once, capped by the block count.
template <class K>
static int block_grid(K kernel, const Blk& bk, int threads, size_t smem) {
  const int nblk = bk.nbx * bk.nby * bk.nbz;
  if (!bk.work) return nblk;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  const long long resident = (long long)(per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
  return (int)(resident < nblk ? resident : nblk);
}

}  // namespace pm
