// The fused interpolate + kick + drift + recompress passes of the step (paper
// Sec. 2.3 force readback, Sec. 2.4 codec): count pass and scatter.
#include <cuda_runtime.h>
#include <stdint.h>

#include "blocks.cuh"
#include "cic.cuh"
#include "particles.cuh"

namespace pm {

// Bound on |v'_d| = |v_d + c_k a_d(x)| before the kick: decoded |v_d| < v_max
// (bin centres) and a CIC-interpolated component never exceeds the largest
// mesh value, so v_max' = v_max + |c_k| (max|a_coarse| + max|a_fine|); every
// operation rounds up, so the float result is not below the exact bound.
__global__ void k_vmax_bound(const float* vin0, const float* vin1, const uint32_t* amax, float ck, float* vout0,
                             float* vout1) {
  const float a = __fadd_ru(__fadd_ru(__uint_as_float(amax[0]), __uint_as_float(amax[1])), __uint_as_float(amax[2]));
  const float ka = __fmul_ru(fabsf(ck), a);
  *vout0 = __fadd_ru(*vin0, ka);
  *vout1 = __fadd_ru(*vin1, ka);
}

// The same CIC gather when the lower corner's local index (lx, ly, lz) and the
// upper weights w1 are already known; same weights and order as gather().
__device__ __forceinline__ void gather_idx(const float* S, int fx, int fy, int fz, int lx, int ly, int lz,
                                           const float w1[3], float a[3]) {
  const float w0[3] = {__fsub_rn(1.0f, w1[0]), __fsub_rn(1.0f, w1[1]), __fsub_rn(1.0f, w1[2])};
  const int plane = fx * fy * fz;
  const float* base = S + (lz * fy + ly) * fx + lx;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const float w = __fmul_rn(__fmul_rn(dx ? w1[0] : w0[0], dy ? w1[1] : w0[1]), dz ? w1[2] : w0[2]);
    const float* q = base + (dz * fy + dy) * fx + dx;
    s0 = __fmaf_rn(w, q[0], s0);
    s1 = __fmaf_rn(w, q[plane], s1);
    s2 = __fmaf_rn(w, q[2 * plane], s2);
  }
  a[0] = s0;
  a[1] = s1;
  a[2] = s2;
}

// Strides of a staged force region (fx x fy x fz nodes, 3 components) in
// shared memory: rows padded to 4 and planes to 16 banks modulo 32, so that
// the nodes around the particles of one compression cell, which the lanes of
// a warp gather at the same time, fall in different banks.
struct RegionStrides {
  int row, plane, comp;
};
#ifndef PM_IKD_PAD
#define PM_IKD_PAD 1
#endif
__host__ __device__ __forceinline__ RegionStrides region_strides(int fx, int fy, int fz) {
  RegionStrides st;
  st.row = PM_IKD_PAD ? fx + ((4 - fx) & 31) : fx;
  const int p0 = st.row * fy;
  st.plane = PM_IKD_PAD ? p0 + ((16 - p0) & 31) : p0;
  st.comp = st.plane * fz;
  return st;
}

// gather_idx on a region with the strides above; same weights and order.
__device__ __forceinline__ void gather_strided(const float* S, RegionStrides st, int lx, int ly, int lz,
                                               const float w1[3], float a[3]) {
  const float w0[3] = {__fsub_rn(1.0f, w1[0]), __fsub_rn(1.0f, w1[1]), __fsub_rn(1.0f, w1[2])};
  const float* base = S + lz * st.plane + ly * st.row + lx;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const float w = __fmul_rn(__fmul_rn(dx ? w1[0] : w0[0], dy ? w1[1] : w0[1]), dz ? w1[2] : w0[2]);
    const float* q = base + dz * st.plane + dy * st.row + dx;
    s0 = __fmaf_rn(w, q[0], s0);
    s1 = __fmaf_rn(w, q[st.comp], s1);
    s2 = __fmaf_rn(w, q[2 * st.comp], s2);
  }
  a[0] = s0;
  a[1] = s1;
  a[2] = s2;
}

// Window of destination compression cells owned by a cell block's histogram:
// the block widened by D cells on each side (clamped to the mesh), periodic.
struct Win {
  int ox, oy, oz, wx, wy, wz;
};
__device__ __forceinline__ Win window_of(const Geo& g, const Blk& bk, CellBlock cb) {
  Win w;
  const int n = g.ncmp, D = bk.D;
  w.wx = bk.wx;
  w.wy = bk.wy;
  w.wz = bk.wz;
  w.ox = w.wx == n ? 0 : cb.ix0 - D;
  w.oy = w.wy == n ? 0 : cb.iy0 - D;
  w.oz = w.wz == n ? 0 : cb.iz0 - D;
  return w;
}
// Window slot of the compression cell with coordinates (cx, cy, cz), or -1.
// The offset from the window's origin lies in (-n, n + D]; of l, l + n and
// l - n the one in [0, n) is the smallest as an unsigned number.
__device__ __forceinline__ unsigned window_offset(int c, int o, unsigned n) {
  const unsigned l = (unsigned)(c - o);
  return min(min(l, l + n), l - n);
}
__device__ __forceinline__ int window_slot_xyz(const Win& w, int n, int cx, int cy, int cz) {
  const unsigned lx = window_offset(cx, w.ox, n), ly = window_offset(cy, w.oy, n), lz = window_offset(cz, w.oz, n);
  const bool in = lx < (unsigned)w.wx && ly < (unsigned)w.wy && lz < (unsigned)w.wz;
  return in ? (int)((lz * w.wy + ly) * w.wx + lx) : -1;
}

// Per-particle scratch record of the two recompress passes (stream index t
// of ntot particles, both species).  Exact v_max' mode: one 16-byte record
// {new position word, v'_x, v'_y, v'_z as float bits}.  Bound mode (codes
// final in the count pass): 8-bit codes as one 8-byte record {position
// word, velocity word}; 16-bit codes as a 4-byte position word and, in a
// second array after the first (16-byte aligned), an 8-byte velocity word.
__device__ __forceinline__ unsigned long long* coded_vel16(uint4* tpv, int64_t ntot) {
  return reinterpret_cast<unsigned long long*>(reinterpret_cast<unsigned char*>(tpv) + ((4 * ntot + 15) & ~15ll));
}
__device__ __forceinline__ uint4 load_record(const uint4* tpv, int64_t t, int coded, bool vel16, int64_t ntot) {
  if (!coded) return tpv[t];
  if (!vel16) {
    const uint2 r = reinterpret_cast<const uint2*>(tpv)[t];
    return make_uint4(r.x, r.y, 0u, 0u);
  }
  const uint32_t pw = reinterpret_cast<const uint32_t*>(tpv)[t];
  const unsigned long long v = coded_vel16(const_cast<uint4*>(tpv), ntot)[t];
  return make_uint4(pw, (uint32_t)v, (uint32_t)(v >> 32), 0u);
}

// Cell index of window row r = lz wy + ly at x = 0 (add window_x for the column).
__device__ __forceinline__ uint32_t window_row(const Geo& g, const Win& w, int r) {
  const int n = g.ncmp;
  const int lz = r / w.wy, ly = r - lz * w.wy;
  int cy = w.oy + ly, cz = w.oz + lz;
  if (cy < 0) cy += n; else if (cy >= n) cy -= n;
  if (cz < 0) cz += n; else if (cz >= n) cz -= n;
  return (uint32_t)(n * (cy + n * cz));
}
__device__ __forceinline__ uint32_t window_x(const Geo& g, const Win& w, int lx) {
  int cx = w.ox + lx;
  if (cx < 0) cx += g.ncmp; else if (cx >= g.ncmp) cx -= g.ncmp;
  return (uint32_t)cx;
}

// ---- interpolate + kick + drift + recompress -------------------------------
//
// Two passes over cell blocks.  The count pass decodes every particle, gathers
// its force, kicks and drifts it, and writes a 16-byte record (below) and a
// 4-byte key; the new-cell counts of the block are histogrammed in shared
// memory over the block's window and added to the global counts once per
// window cell.  Both adds return what they found: a particle's rank within its
// block's share of the cell (shared memory) and the start of that share within
// the cell (global memory, kept per block and window cell in `start`).  So the
// scatter knows every destination, newoff[cell] + start + rank, without
// counting again: no histogram, no cursors, no atomics but for far movers
// (256^3 workload, 8-bit codes: 0.266 ms when it counted again, 0.247 now;
// 768^3, 5.1e8 particles with 16-bit codes: 8.4 ms both, 4.5 of them its
// scattered stores).
//
// Key of a particle in its block's window: the top bit, then the window slot,
// then its rank in the low kb bits.  A far mover (outside the window, or with
// a rank that does not fit) has its new cell as the key; far movers of a cell
// are counted apart and placed behind the cell's window movers by a cursor.
constexpr uint32_t kInWindow = 0x80000000u;

// Arguments of the count pass.
struct KickArgs {
  PCodes c0, c1;
  const int64_t* off0;
  const int64_t* off1;
  Geo g;
  Blk bk;
  const float* acc_c;
  const float* acc_f;
  float ck, cd;
  RecompressTables t;
  uint32_t* vmax_bits;
  uint32_t* tkey;
  uint4* tpv;
  const float* vq0;       // v_max' known before the pass (bound mode): quantise here, the scatter copies codes
  const float* vq1;
  const float4* app;      // particle-particle term (Eq. 4), precomputed per particle
  int coarse;             // gather the coarse force separately (0: the fine mesh carries it)
};

// Rank of the calling lane among the block's particles of its window slot:
// what atomicAdd(hist + slot, 1) returns.  A shared-memory atomic whose lanes
// share an address and return their values is serialised lane by lane, and the
// stream is cell ordered: cold particles stay in their cell, and consecutive
// lanes have the same slot.  Where half of the lanes continue their
// neighbour's run, the first lane of each run takes the run's ranks with one
// atomic; hot particles, which scatter, take them one by one.  All 32 lanes
// must call it; lanes without a slot pass has = false and a slot of their own
// (~0u - lane).
__device__ __forceinline__ uint32_t slot_rank(uint32_t* hist, uint32_t slot, bool has) {
  const int lane = (int)(threadIdx.x & 31);
  const uint32_t prev = __shfl_up_sync(0xffffffffu, slot, 1);
  const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || prev != slot);
  if (__popc(heads) > 16) return has ? atomicAdd(hist + slot, 1u) : 0u;
  const uint32_t upto = 0xffffffffu >> (31 - lane);   // lanes 0 .. lane
  const int first = 31 - __clz(heads & upto);         // head of this lane's run
  const uint32_t later = heads & ~upto;
  const int end = later ? __ffs(later) - 1 : 32;       // head of the next run
  uint32_t old = 0;
  if (lane == first && has) old = atomicAdd(hist + slot, (uint32_t)(end - lane));
  old = __shfl_sync(0xffffffffu, old, first);
  return old + (uint32_t)(lane - first);
}

// One species' part of the pass, as every particle of it needs it.
struct Kicked {
  Win win;
  int n, kb;
  float to_code;          // 256 / r: position codes per fine cell
  float ck, cd, nf;
  uint32_t* hist;         // shared memory, this species' window
  uint32_t* far;
  bool coded, qzero;
  float qs;
  int half;
};

// Kick, drift and recode one particle whose gathered acceleration is a, and
// store its key and record: tk and rec point at the particle's own.  All lanes
// of the warp call it (slot_rank); live: the lane has a particle.
// Positions are recoded in one conversion: x 256 / r is exact (a power of two
// times x) and below 2^24, so its integer part holds the cell (upper bits) and
// the in-cell code (low byte), the same as floor(x / r) and floor(256 frac).
template <bool V16>
__device__ __forceinline__ void kick_and_store(const Kicked& k, bool live, float x[3], float v[3], const float a[3],
                                               uint32_t* tk, uint4* tpv, unsigned long long* vel16, int64_t t,
                                               float& local_max) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    v[d] = __fmaf_rn(k.ck, a[d], v[d]);
    x[d] = wrap_near(__fmaf_rn(k.cd, v[d], x[d]), k.nf);
  }
  if (!(x[0] >= 0.f && x[0] < k.nf && x[1] >= 0.f && x[1] < k.nf && x[2] >= 0.f && x[2] < k.nf)) {
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] = wrap_far(x[d], k.nf);
  }
  int code[3], cell[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    code[d] = (int)__fmul_rn(x[d], k.to_code);
    cell[d] = code[d] >> 8;
  }
  const int slot = window_slot_xyz(k.win, k.n, cell[0], cell[1], cell[2]);
  const bool inw = live && slot >= 0;
  const uint32_t rank = slot_rank(k.hist, inw ? (uint32_t)slot : ~0u - (threadIdx.x & 31), inw);
  if (!live) return;
  uint32_t key;
  if (inw && (rank >> k.kb) == 0) {
    key = kInWindow | ((uint32_t)slot << k.kb) | rank;
  } else {
    key = (uint32_t)(cell[0] + k.n * (cell[1] + k.n * cell[2]));
    atomicAdd(k.far + key, 1u);
  }
  *tk = key;
  const uint32_t pw = __byte_perm(__byte_perm(code[0], code[1], 0x0040), code[2], 0x0410) & 0xffffffu;
  if (k.coded) {
    int c3[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) c3[d] = encode_vel(v[d], k.qs, k.half, k.qzero);
    if (V16) {
      reinterpret_cast<uint32_t*>(tpv)[t] = pw;
      vel16[t] = (unsigned long long)((uint32_t)c3[0] | ((uint32_t)c3[1] << 16)) | ((unsigned long long)c3[2] << 32);
    } else {
      reinterpret_cast<uint2*>(tpv)[t] = make_uint2(pw, (uint32_t)c3[0] | ((uint32_t)c3[1] << 8) | ((uint32_t)c3[2] << 16));
    }
  } else {
    tpv[t] = make_uint4(pw, __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]));
    local_max = fmaxf(local_max, fmaxf(fabsf(v[0]), fmaxf(fabsf(v[1]), fabsf(v[2]))));
  }
}

// Species part of a block: window, histogram and quantiser.
__device__ __forceinline__ Kicked kicked_of(const KickArgs& k, const Win& win, int s, uint32_t* hist, int W,
                                            bool vel16) {
  Kicked q;
  q.win = win;
  q.n = k.g.ncmp;
  q.kb = k.t.kb;
  q.to_code = 256.0f / (float)k.g.rcmp;
  q.ck = k.ck;
  q.cd = k.cd;
  q.nf = (float)k.g.nf;
  q.hist = hist + s * W;
  q.far = s ? k.t.far1 : k.t.far0;
  const float* vq = s ? k.vq1 : k.vq0;
  q.coded = vq != nullptr;
  const float vqm = q.coded ? *vq : 0.f;
  q.half = vel16 ? 32768 : 128;
  q.qzero = !(vqm > 0.f);
  q.qs = (q.coded && !q.qzero) ? __fdiv_rn((float)q.half, vqm) : 0.f;
  return q;
}

// Adds a block's window counts to the global ones and notes where its share
// of each cell starts.  All atomics of a thread are issued before any result
// is used.
__device__ __forceinline__ void flush_window(const KickArgs& k, const Win& win, const uint32_t* hist, int W, int bid) {
  constexpr int J = 4;
  uint32_t* start = k.t.start + (size_t)bid * 2 * W;
  for (int i0 = threadIdx.x; i0 < 2 * W; i0 += J * blockDim.x) {
    uint32_t at[J];
    bool some[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int i = i0 + j * blockDim.x;
      uint32_t m = i < 2 * W ? hist[i] : 0u;
      m = m < (1u << k.t.kb) ? m : (1u << k.t.kb);   // ranks beyond went to the far movers
      some[j] = m != 0u;
      if (some[j]) {
        const int sp = i >= W ? 1 : 0, r = i - sp * W;
        const int row = r / win.wx, lx = r - row * win.wx;
        at[j] = atomicAdd((sp ? k.t.counts1 : k.t.counts0) + window_row(k.g, win, row) + window_x(k.g, win, lx), m);
      }
    }
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (some[j]) start[i0 + j * blockDim.x] = at[j];
  }
}

// The force region of a cell block, rows of 4-byte copies: any shape.
__device__ __forceinline__ void stage_region(const float* acc, const Geo& g, RegionStrides st, int fx, int fy, int fz,
                                             int bxf, int byf, int bzf, float* sf) {
  const int nf = g.nf;
  const int64_t nf3 = (int64_t)nf * nf * nf;
  const int lines = 3 * fz * fy;
  for (int li = threadIdx.x >> 5; li < lines; li += blockDim.x >> 5) {
    const int comp = li / (fz * fy), rem = li - comp * fz * fy;
    const int lz = rem / fy, ly = rem - lz * fy;
    int gz = bzf + lz, gy = byf + ly;
    if (gz >= nf) gz -= nf;
    if (gy >= nf) gy -= nf;
    const float* src = acc + comp * nf3 + ((int64_t)gz * nf + gy) * nf;
    float* dst = sf + comp * st.comp + lz * st.plane + ly * st.row;
    for (int lx = threadIdx.x & 31; lx < fx; lx += 32) {
      int gx = bxf + lx;
      if (gx >= nf) gx -= nf;
      copy_async4(dst + lx, src + gx);   // all of a thread's copies in flight at once
    }
  }
}
// The coarse force around a cell block ((RX + 1)(RY + 1)(RZ + 1) nodes).
__device__ __forceinline__ void stage_coarse(const float* acc, const Geo& g, const Blk& bk, CellBlock cb, float* sc) {
  const int nc = g.nc, cx = bk.RX + 1, cy = bk.RY + 1, cz = bk.RZ + 1;
  const int64_t nc3 = (int64_t)nc * nc * nc;
  for (int i = threadIdx.x; i < 3 * cx * cy * cz; i += blockDim.x) {
    const int comp = i / (cx * cy * cz), rem = i - comp * cx * cy * cz;
    const int lz = rem / (cx * cy), rem2 = rem - lz * cx * cy;
    const int ly = rem2 / cx, lx = rem2 - ly * cx;
    int gx = cb.ix0 + lx, gy = cb.iy0 + ly, gz = cb.iz0 + lz;
    if (gx >= nc) gx -= nc;
    if (gy >= nc) gy -= nc;
    if (gz >= nc) gz -= nc;
    sc[i] = __ldg(acc + comp * nc3 + ((int64_t)gz * nc + gy) * nc + gx);
  }
}

// Threads per CTA of the count pass and of the scatter, and the resident CTAs
// per SM they are compiled for (sets their register budget).
constexpr int kKickThreads = 512, kKickMinBlocks = 2;   // any shape
// (scatter at 768^3: 4 CTAs per SM 8.02 ms, 5 8.25, 6 8.92, 8 with one particle per thread at a time 8.56)
constexpr int kScatterThreads = 256, kScatterMinBlocks = 4;

// Count pass, any block shape.
template <bool V16>
__global__ void __launch_bounds__(kKickThreads, kKickMinBlocks) k_kick_count(KickArgs k) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const Geo& g = k.g;
  const Blk& bk = k.bk;
  const bool two_c = g.two && k.coarse != 0;
  for_each_block(bk, [&](const int bid) {
    const int r = g.rcmp;
    const int nrow = bk.RY * bk.RZ;
    const int fx = bk.RX * r + 1, fy = bk.RY * r + 1, fz = bk.RZ * r + 1;
    const int cx = bk.RX + 1, cy = bk.RY + 1, cz = bk.RZ + 1;
    const CellBlock cb = block_of(bk, bid);
    const Win win = window_of(g, bk, cb);
    const int W = win.wx * win.wy * win.wz;
    int64_t* roff = reinterpret_cast<int64_t*>(smraw);
    uint32_t* hist = reinterpret_cast<uint32_t*>(roff + 2 * nrow * (bk.RX + 1));
    float* sf = reinterpret_cast<float*>(hist + 2 * W);
    const RegionStrides fst = region_strides(fx, fy, fz);
    float* sc = sf + 3 * fst.comp;
    load_row_offsets(k.off0, g, bk, cb, roff);
    load_row_offsets(k.off1, g, bk, cb, roff + nrow * (bk.RX + 1));
    for (int i = threadIdx.x; i < 2 * W; i += blockDim.x) hist[i] = 0;
    stage_region(k.acc_f, g, fst, fx, fy, fz, cb.ix0 * r, cb.iy0 * r, cb.iz0 * r, sf);
    if (two_c) stage_coarse(k.acc_c, g, bk, cb, sc);
    async_copies_wait();
    __syncthreads();
    const float pscale = (float)r / 256.0f;
    for (int s = 0; s < 2; ++s) {
      const PCodes& in = s ? k.c1 : k.c0;
      const int64_t toff = s ? k.c0.n : 0;
      const Kicked q = kicked_of(k, win, s, hist, W, V16);
      unsigned long long* vel16 = coded_vel16(k.tpv, k.c0.n + k.c1.n);
      const float step = __fmul_rn(*in.vmax, 1.0f / (float)q.half);
      float local_max = 0.f;
      const int64_t* ro_s = roff + s * nrow * (bk.RX + 1);
      for (int row = 0; row < nrow; ++row) {
        const int64_t* ro = ro_s + row * (bk.RX + 1);
        const int ky = row % bk.RY, kz = row / bk.RY;
        // a corrupt stream (flagged by the scan) may claim more particles than
        // exist; never read past the caller's n records
        const int64_t p0 = ro[0] < in.n ? ro[0] : in.n;
        const int64_t p1 = ro[bk.RX] < in.n ? ro[bk.RX] : in.n;
        for (int64_t pb = p0; pb < p1; pb += blockDim.x) {
          const int64_t p = pb + threadIdx.x;
          const bool live = p < p1;
          float x[3] = {0.f, 0.f, 0.f}, v[3] = {0.f, 0.f, 0.f}, a[3] = {0.f, 0.f, 0.f};
          if (live) {
            const int ixl = row_cell(ro, bk.RX, p);
            int qp[3], qv[3];
            unpack_pos(in.pos[p], qp);
            load_vel(in.vel, V16, p, qv);
            x[0] = decode_pos(cb.ix0 + ixl, qp[0], pscale);
            x[1] = decode_pos(cb.iy0 + ky, qp[1], pscale);
            x[2] = decode_pos(cb.iz0 + kz, qp[2], pscale);
#pragma unroll
            for (int d = 0; d < 3; ++d) v[d] = decode_vel(qv[d], q.half, step);
            // Decoded positions are exact dyadics, so the CIC cell and weight come
            // from the codes in integer arithmetic: x = c r + (2q + 1) r / 512.
            int num[3];
            float w1[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              num[d] = (2 * qp[d] + 1) * r;
              w1[d] = __fmul_rn(__int2float_rn(num[d] & 511), 1.0f / 512.0f);
            }
            gather_strided(sf, fst, ixl * r + (num[0] >> 9), ky * r + (num[1] >> 9), kz * r + (num[2] >> 9), w1, a);
            if (two_c) {
              // coarse cell == compression cell: corner (ixl, ky, kz), weight (2q + 1) / 512
              float b[3], u1[3];
#pragma unroll
              for (int d = 0; d < 3; ++d) u1[d] = __fmul_rn(__int2float_rn(2 * qp[d] + 1), 1.0f / 512.0f);
              gather_idx(sc, cx, cy, cz, ixl, ky, kz, u1, b);
#pragma unroll
              for (int d = 0; d < 3; ++d) a[d] = __fadd_rn(b[d], a[d]);
            }
            if (k.app) {
              const float4 q4 = k.app[toff + p];
              a[0] = __fadd_rn(a[0], q4.x);
              a[1] = __fadd_rn(a[1], q4.y);
              a[2] = __fadd_rn(a[2], q4.z);
            }
          }
          kick_and_store<V16>(q, live, x, v, a, k.tkey + toff + p, k.tpv, vel16, toff + p, local_max);
        }
      }
      if (!q.coded) block_vmax(local_max, k.vmax_bits + s);
    }
    __syncthreads();
    flush_window(k, win, hist, W, bid);
  });
}

// Count pass for blocks of one row of at most kRowCells compression cells of 4
// fine cells (the shapes that the defaults and the autotuner pick).  Issue
// bound, so what a particle costs in instructions is what counts: the strides
// of the staged region are constants whatever the row's length, offsets and
// indices are 32-bit and relative to the row, codes are taken apart without
// 64-bit shifts, and the next particle's codes are loaded while this one is
// worked on.  256^3 workload, 8-bit codes: 0.380 ms before, 0.311 now (with the
// ranks); 768^3, 5.1e8 particles: 9.93 -> 8.31 ms.
// CELLS: the longest row, 64, or 32 where a dense set's rows are dealt out in
// pieces (kick_blocks): with 5 CTAs of 256 threads per SM the staging, the
// particles and the flush of different blocks overlap better than with 2 of 512
// over 64 cells (0.307 -> 0.296 ms; 768^3 8.13 -> 7.71; 64 cells with 640 threads
// 8.37, 32 cells with 320 threads and 4 CTAs 8.23, 16 cells with 128 and 10 CTAs
// 8.60).  Windows of half-width 2 and sparse sets keep 64 cells: their blocks do
// more per window cell than per particle (clustered 512^3 with half-width 2:
// scatter 1.46 ms with 64 cells, 1.72 with 32).
// STAGED: the block's force region is copied to shared memory (41 or 80 KB).  That costs 300 values per cell, 24 are needed per particle: below
// kStageFrom particles per cell the forces are gathered from the mesh directly
// (192^3 mesh with 2.8 particles per cell: 0.114 ms staged, 0.042 direct).
constexpr int kStageFrom = 12;
constexpr int kDirectThreads = 128, kDirectMinBlocks = 8;
template <int CELLS> struct RowRegion {
  static constexpr int row = 4 * CELLS + 4;                     // 4 banks modulo 32, whole 16-byte words
  static constexpr int plane = 5 * row + 28;                    // 16 banks modulo 32
  static constexpr int comp = 5 * plane;
  static_assert(row % 32 == 4 && plane % 32 == 16 && comp % 4 == 0, "bank layout, 16-byte rows");
};

__device__ __forceinline__ void copy_async16(float* smem_dst, const float* gmem_src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}

// The force at lower node (base) and upper weights w1; same weights and order as gather().
template <class R>
__device__ __forceinline__ void gather_row_region(const float* base, const float w1[3], float a[3]) {
  const float w0[3] = {__fsub_rn(1.0f, w1[0]), __fsub_rn(1.0f, w1[1]), __fsub_rn(1.0f, w1[2])};
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const float w = __fmul_rn(__fmul_rn(dx ? w1[0] : w0[0], dy ? w1[1] : w0[1]), dz ? w1[2] : w0[2]);
    const float* q = base + dz * R::plane + dy * R::row + dx;
    s0 = __fmaf_rn(w, q[0], s0);
    s1 = __fmaf_rn(w, q[R::comp], s1);
    s2 = __fmaf_rn(w, q[2 * R::comp], s2);
  }
  a[0] = s0;
  a[1] = s1;
  a[2] = s2;
}

template <bool STAGED, int CELLS> struct RowForm {
  static constexpr int threads = !STAGED ? kDirectThreads : (CELLS == 32 ? 256 : kKickThreads);
  static constexpr int min_blocks = !STAGED ? kDirectMinBlocks : (CELLS == 32 ? 5 : kKickMinBlocks);
};
template <bool V16, bool STAGED, int CELLS>
__global__ void __launch_bounds__(RowForm<STAGED, CELLS>::threads, RowForm<STAGED, CELLS>::min_blocks)
    k_kick_count_row(KickArgs k) {
  using R = RowRegion<CELLS>;
  constexpr int kRowCells = CELLS;
  extern __shared__ __align__(16) unsigned char smraw[];
  const Geo& g = k.g;
  const Blk& bk = k.bk;
  const bool two_c = g.two && k.coarse != 0;
  constexpr uint32_t kSeg = 1u << 30;   // particles of a row handled with one set of 32-bit offsets
  constexpr int kThreads = RowForm<STAGED, CELLS>::threads;
  for_each_block(bk, [&](const int bid) {
    const int RX = bk.RX;
    const CellBlock cb = block_of(bk, bid);
    const Win win = window_of(g, bk, cb);
    const int W = win.wx * win.wy * win.wz;
    float* sf = reinterpret_cast<float*>(smraw);                               // staged region, then the coarse one
    float* sc = sf + (STAGED ? 3 * R::comp : 0);
    uint32_t* rel = reinterpret_cast<uint32_t*>(sc + (two_c ? 12 * (kRowCells + 1) : 0));   // [2][kRowCells]
    uint32_t* hist = rel + 2 * kRowCells;
    const int64_t c0 = cb.ix0 + (int64_t)g.ncmp * (cb.iy0 + (int64_t)g.ncmp * cb.iz0);
    for (int i = threadIdx.x; i < 2 * kRowCells; i += kThreads) {
      const int s = i / kRowCells, j = i % kRowCells;
      const int64_t* off = (s ? k.off1 : k.off0) + c0;
      const int64_t d = j < RX ? off[j] - off[0] : kSeg;
      rel[i] = d < kSeg ? (uint32_t)d : kSeg;
    }
    for (int i = threadIdx.x; i < 2 * W; i += kThreads) hist[i] = 0;
    const int bxf = cb.ix0 * 4, byf = cb.iy0 * 4, bzf = cb.iz0 * 4;
    if (STAGED) {
      // row starts are 16-byte aligned on both sides (nf and ix0 4 are multiples of 4)
      const int nf = g.nf;
      const int64_t nf3 = (int64_t)nf * nf * nf;
      for (int li = threadIdx.x >> 5; li < 75; li += kThreads / 32) {
        const int comp = li / 25, rem = li - comp * 25;
        const int lz = rem / 5, ly = rem - lz * 5;
        int gz = bzf + lz, gy = byf + ly;
        if (gz >= nf) gz -= nf;
        if (gy >= nf) gy -= nf;
        const float* src = k.acc_f + comp * nf3 + ((int64_t)gz * nf + gy) * nf;
        float* dst = sf + comp * R::comp + lz * R::plane + ly * R::row;
        for (int j = threadIdx.x & 31; j <= RX; j += 32) {
          if (j < RX) copy_async16(dst + 4 * j, src + bxf + 4 * j);
          else copy_async4(dst + 4 * j, src + (bxf + 4 * j == nf ? 0 : bxf + 4 * j));
        }
      }
      if (two_c) stage_coarse(k.acc_c, g, bk, cb, sc);
      async_copies_wait();
    }
    __syncthreads();
    for (int s = 0; s < 2; ++s) {
      const PCodes& in = s ? k.c1 : k.c0;
      const int64_t toff = s ? k.c0.n : 0;
      const Kicked q = kicked_of(k, win, s, hist, W, V16);
      unsigned long long* vel16 = coded_vel16(k.tpv, k.c0.n + k.c1.n);
      const float step = __fmul_rn(*in.vmax, 1.0f / (float)q.half);
      const float vmid = (float)q.half - 0.5f;
      float local_max = 0.f;
      const int64_t* off = (s ? k.off1 : k.off0) + c0;
      const uint32_t* ro = rel + s * kRowCells;
      // a corrupt stream (flagged by the scan) may claim more particles than
      // exist; never read past the caller's n records
      const int64_t o0 = off[0], o1 = off[RX];
      const int64_t p0 = o0 < in.n ? o0 : in.n, p1 = o1 < in.n ? o1 : in.n;
      for (int64_t seg = p0; seg < p1; seg += kSeg) {
        if (seg > p0) {   // a row of more than 2^30 particles: offsets of its next part
          __syncthreads();
          for (int j = threadIdx.x; j < RX; j += kThreads) {
            const int64_t d = off[j] - seg;
            rel[s * kRowCells + j] = d <= 0 ? 0u : (d < kSeg ? (uint32_t)d : kSeg);
          }
          __syncthreads();
        }
        const uint32_t m = p1 - seg < kSeg ? (uint32_t)(p1 - seg) : kSeg;
        const uint32_t* pos = in.pos + seg;
        const uint2* vel_w = reinterpret_cast<const uint2*>(in.vel) + (V16 ? seg : 0);
        const uint32_t* vel_b = reinterpret_cast<const uint32_t*>(in.vel) + (V16 ? 0 : seg);
        uint32_t pw = 0;
        uint2 vw = make_uint2(0, 0);
        if (threadIdx.x < m) {
          pw = pos[threadIdx.x];
          if (V16) vw = vel_w[threadIdx.x];
          else vw.x = vel_b[threadIdx.x];
        }
        for (uint32_t b = 0; b < m; b += kThreads) {
          const uint32_t i = b + threadIdx.x;
          const bool live = i < m;
          const uint32_t cpw = pw;
          const uint2 cvw = vw;
          if (i + kThreads < m) {
            pw = __ldcs(pos + i + kThreads);   // read once
            if (V16) vw = __ldcs(vel_w + i + kThreads);
            else vw.x = __ldcs(vel_b + i + kThreads);
          }
          // the last cell whose offset is at most i (entries past the row hold 2^30)
          int ixl = 0;
#pragma unroll
          for (int d = kRowCells / 2; d > 0; d >>= 1)
            if (ro[ixl + d] <= i) ixl += d;
          // fine cell in the compression cell (2 bits) and weight (2 q + 1) / 128 of each axis
          const uint32_t hi = (cpw >> 6) & 0x030303u, lo = ((cpw & 0x3f3f3fu) << 1) | 0x010101u;
          const int nx = 4 * ixl + (int)(hi & 3u), ny = (int)((hi >> 8) & 3u), nz = (int)(hi >> 16);
          const float w1[3] = {__fmul_rn(__uint2float_rn(lo & 0xffu), 1.0f / 128.0f),
                               __fmul_rn(__uint2float_rn((lo >> 8) & 0xffu), 1.0f / 128.0f),
                               __fmul_rn(__uint2float_rn(lo >> 16), 1.0f / 128.0f)};
          // node + weight: the decoded position, exactly
          float x[3] = {__fadd_rn(__int2float_rn(bxf + nx), w1[0]), __fadd_rn(__int2float_rn(byf + ny), w1[1]),
                        __fadd_rn(__int2float_rn(bzf + nz), w1[2])};
          uint32_t u[3];
          if (V16) {
            u[0] = cvw.x & 0xffffu;
            u[1] = cvw.x >> 16;
            u[2] = cvw.y & 0xffffu;
          } else {
            u[0] = cvw.x & 0xffu;
            u[1] = (cvw.x >> 8) & 0xffu;
            u[2] = (cvw.x >> 16) & 0xffu;
          }
          float v[3], a[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) v[d] = __fmul_rn(__fsub_rn(__uint2float_rn(u[d]), vmid), step);
          if (STAGED) {
            gather_row_region<R>(sf + nz * R::plane + ny * R::row + nx, w1, a);
            if (two_c && live) {
              // coarse cell == compression cell: corner (ixl, 0, 0), weight (2q + 1) / 512
              float b3[3], u1[3];
#pragma unroll
              for (int d = 0; d < 3; ++d)
                u1[d] = __fmul_rn(__int2float_rn((int)(2 * ((cpw >> (8 * d)) & 0xffu) + 1)), 1.0f / 512.0f);
              gather_idx(sc, RX + 1, 2, 2, ixl, 0, 0, u1, b3);
#pragma unroll
              for (int d = 0; d < 3; ++d) a[d] = __fadd_rn(b3[d], a[d]);
            }
          } else {
            a[0] = a[1] = a[2] = 0.f;
            if (live) {
              gather(k.acc_f, g.nf, x[0], x[1], x[2], a);
              if (two_c) {
                float b3[3];
                gather(k.acc_c, g.nc, __fmul_rn(x[0], 0.25f), __fmul_rn(x[1], 0.25f), __fmul_rn(x[2], 0.25f), b3);
#pragma unroll
                for (int d = 0; d < 3; ++d) a[d] = __fadd_rn(b3[d], a[d]);
              }
            }
          }
          if (k.app && live) {
            const float4 q4 = k.app[toff + seg + i];
            a[0] = __fadd_rn(a[0], q4.x);
            a[1] = __fadd_rn(a[1], q4.y);
            a[2] = __fadd_rn(a[2], q4.z);
          }
          const int64_t t = toff + seg + i;
          kick_and_store<V16>(q, live, x, v, a, k.tkey + t, k.tpv, vel16, t, local_max);
        }
      }
      if (!q.coded) block_vmax(local_max, k.vmax_bits + s);
    }
    __syncthreads();
    flush_window(k, win, hist, W, bid);
  });
}

// Arguments of the scatter.
struct ScatterArgs {
  int64_t n0, n1;
  const int64_t* off0;
  const int64_t* off1;
  Geo g;
  Blk bk;
  RecompressTables t;
  const int64_t* newoff0;
  const int64_t* newoff1;
  PCodesOut o0, o1;
  const uint32_t* tkey;
  const uint4* tpv;
  int coded;
  int* status;
};

// Scatter: places every particle of a cell block in its new cell, newoff[cell]
// + start + rank from the count pass (far movers behind the cell's window
// movers, by a cursor), quantising the velocity with the new v_max.  Bound by
// its scattered stores: a cell's hot neutrinos land in some 27 cells, so a
// warp's stores touch about 23 sectors per array.
template <bool V16>
__global__ void __launch_bounds__(kScatterThreads, kScatterMinBlocks) k_kick_scatter(ScatterArgs k) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const Geo& g = k.g;
  const Blk& bk = k.bk;
  for_each_block(bk, [&](const int bid) {
    const CellBlock cb = block_of(bk, bid);
    const Win win = window_of(g, bk, cb);
    const int W = win.wx * win.wy * win.wz;
    int64_t* base = reinterpret_cast<int64_t*>(smraw);     // [2 W] first index of the block's share of a window cell
    const uint32_t* start = k.t.start + (size_t)bid * 2 * W;
    for (int i = threadIdx.x; i < 2 * W; i += blockDim.x) {
      const int sp = i >= W ? 1 : 0, r = i - sp * W;
      const int row = r / win.wx, lx = r - row * win.wx;
      base[i] = (sp ? k.newoff1 : k.newoff0)[window_row(g, win, row) + window_x(g, win, lx)] + (int64_t)start[i];
    }
    __syncthreads();
    const uint32_t rank_mask = (1u << k.t.kb) - 1u;
    for (int s = 0; s < 2; ++s) {
      const int64_t n = s ? k.n1 : k.n0;
      const int64_t toff = s ? k.n0 : 0;
      const PCodesOut& o = s ? k.o1 : k.o0;
      const int64_t* base_s = base + s * W;
      const int half = V16 ? 32768 : 128;
      const float vm = *o.vmax;
      const bool vzero = !(vm > 0.f);
      const float sv = vzero ? 0.f : __fdiv_rn((float)half, vm);
      for (int row = 0; row < bk.RY * bk.RZ; ++row) {
        const int iy = cb.iy0 + row % bk.RY, iz = cb.iz0 + row / bk.RY;
        const int64_t* off = (s ? k.off1 : k.off0) + cb.ix0 + (int64_t)g.ncmp * (iy + (int64_t)g.ncmp * iz);
        const int64_t o0 = off[0], o1 = off[bk.RX];
        const int64_t p0 = o0 < n ? o0 : n, p1 = o1 < n ? o1 : n;
        // several particles per thread loaded before any is placed
        constexpr int U = 2;
        for (int64_t pb = p0 + threadIdx.x; pb < p1; pb += U * kScatterThreads) {
          uint32_t tk[U];
          uint4 pv[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int64_t p = pb + u * kScatterThreads;
            if (p < p1) {
              tk[u] = k.tkey[toff + p];
              pv[u] = load_record(k.tpv, toff + p, k.coded, V16, k.n0 + k.n1);
            }
          }
          // far movers' cursors and offsets: all in flight before any is used
          uint32_t top[U], ahead[U];
          int64_t at[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (pb + u * kScatterThreads < p1 && !(tk[u] & kInWindow)) {
              top[u] = atomicSub((s ? k.t.far1 : k.t.far0) + tk[u], 1u);
              ahead[u] = (s ? k.t.counts1 : k.t.counts0)[tk[u]];
              at[u] = (s ? k.newoff1 : k.newoff0)[tk[u]];
            }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            if (pb + u * kScatterThreads >= p1) continue;
            const int64_t dst = tk[u] & kInWindow
                                    ? base_s[(tk[u] & ~kInWindow) >> k.t.kb] + (int64_t)(tk[u] & rank_mask)
                                    : at[u] + (int64_t)ahead[u] + (int64_t)top[u] - 1;
            if (dst < 0 || dst >= n) {
              atomicOr(k.status, ST_CORRUPT);
              continue;
            }
            o.pos[dst] = pv[u].x;
            if (k.coded) {
              if (V16)
                reinterpret_cast<unsigned long long*>(o.vel)[dst] =
                    (unsigned long long)pv[u].y | ((unsigned long long)pv[u].z << 32);
              else
                reinterpret_cast<uint32_t*>(o.vel)[dst] = pv[u].y;
              continue;
            }
            int qv[3];
            qv[0] = encode_vel(__uint_as_float(pv[u].y), sv, half, vzero);
            qv[1] = encode_vel(__uint_as_float(pv[u].z), sv, half, vzero);
            qv[2] = encode_vel(__uint_as_float(pv[u].w), sv, half, vzero);
            store_vel(o.vel, V16, dst, qv);
          }
        }
      }
    }
  });
}

// ------------------------------------------------------------ launchers --

// Brick order of the cell blocks (block_of): edge in block rows, and the
// number of (y, z) block rows from which it is used.  Measured on the
// 1536^3 workload (147,456 kick-block rows): scatter 90.1 -> 70.5 ms; on
// the 256^3 workload (4,096 rows, whose new codes fit in L2 anyway) it made
// the scatter 4% slower, so smaller grids keep the row order.
#ifndef PM_BLOCK_BRICK
#define PM_BLOCK_BRICK 16
#endif
#ifndef PM_BRICK_MIN_ROWS
#define PM_BRICK_MIN_ROWS 32768
#endif

size_t kick_count_smem(const Geo& g, const Blk& bk) {
  size_t nrow = (size_t)bk.RY * bk.RZ;
  size_t coarse = g.two ? (size_t)(bk.RX + 1) * (bk.RY + 1) * (bk.RZ + 1) : 0;
  const RegionStrides st = region_strides(bk.RX * g.rcmp + 1, bk.RY * g.rcmp + 1, bk.RZ * g.rcmp + 1);
  return 2 * nrow * (bk.RX + 1) * sizeof(int64_t) + 2 * (size_t)window_cells(g, bk) * 4 +
         3 * ((size_t)st.comp + coarse) * sizeof(float);
}

// Shared memory per block that a shape may need to be accepted (pm_set_tuning), in
// terms of the general kernels: offsets, and 12 bytes per window cell and species for
// the scatter.  The scatter takes less, 8 bytes per window cell, and the row form of
// the count pass at most 127 KB.
size_t kick_scatter_smem(const Geo& g, const Blk& bk) {
  size_t nrow = (size_t)bk.RY * bk.RZ;
  return 2 * nrow * (bk.RX + 1) * sizeof(int64_t) + 2 * (size_t)window_cells(g, bk) * (8 + 4);
}

int block_brick(const Blk& bk) {
  const int B = PM_BLOCK_BRICK;
  return (B > 1 && bk.nby % B == 0 && bk.nbz % B == 0 && (int64_t)bk.nby * bk.nbz >= PM_BRICK_MIN_ROWS) ? B : 1;
}

// Edge of the window along an axis on which the block has R cells.
static int window_edge(const Geo& g, const Blk& bk, int R) {
  if (bk.D < 0) return 0;
  return R + 2 * bk.D < g.ncmp ? R + 2 * bk.D : g.ncmp;
}
static void set_window(const Geo& g, Blk& bk) {
  bk.wx = window_edge(g, bk, bk.RX);
  bk.wy = window_edge(g, bk, bk.RY);
  bk.wz = window_edge(g, bk, bk.RZ);
}
int window_cells(const Geo& g, const Blk& bk) {
  return window_edge(g, bk, bk.RX) * window_edge(g, bk, bk.RY) * window_edge(g, bk, bk.RZ);
}


// The blocks that the passes take for an asked shape: single rows of more than
// kKickRowCells cells are cut in halves for dense sets and windows of half-width 1.
Blk kick_blocks(const Geo& g, Blk bk, int64_t particles) {
  if (g.rcmp == 4 && bk.RY == 1 && bk.RZ == 1 && bk.D == 1 && particles >= (int64_t)kStageFrom * g.ncell)
    while (bk.RX > kKickRowCells && bk.RX % 2 == 0) {
      bk.RX /= 2;
      bk.nbx *= 2;
    }
  return bk;
}

// Start tables: 8 bytes per block and window cell.
size_t table_bytes(const Geo& g, const Blk& bk) {
  return (size_t)bk.nbx * bk.nby * bk.nbz * 2 * (size_t)window_cells(g, bk) * 4;
}

// Rank bits of a key: what the top bit and the window slot leave.
static int rank_bits(const Geo& g, const Blk& bk) {
  int slot = 0;
  while ((1 << slot) < window_cells(g, bk)) ++slot;
  return 31 - slot;
}

template <bool V16>
static cudaError_t kick_count(const KickArgs& k, int64_t particles, cudaStream_t st) {
  const Blk& bk = k.bk;
  const bool row = bk.RY == 1 && bk.RZ == 1 && bk.RX <= 64 && k.g.rcmp == 4;
  const bool halves = row && bk.RX <= kKickRowCells && bk.D == 1;
  const bool staged = particles >= (int64_t)kStageFrom * k.g.ncell;
  size_t smem;
  int threads = kKickThreads;
  void (*f)(KickArgs);
  if (row) {
    const int cells = staged && halves ? 32 : 64;
    if (!staged) f = k_kick_count_row<V16, false, 64>;
    else if (halves) f = k_kick_count_row<V16, true, 32>;
    else f = k_kick_count_row<V16, true, 64>;
    threads = !staged ? kDirectThreads : (halves ? RowForm<true, 32>::threads : kKickThreads);
    smem = 4 * ((staged ? 3 * (size_t)(halves ? RowRegion<32>::comp : RowRegion<64>::comp) : 0) +
                (k.g.two && k.coarse ? 12 * (cells + 1) : 0) + 2 * cells + 2 * (size_t)window_cells(k.g, bk));
  } else {
    f = k_kick_count<V16>;
    smem = kick_count_smem(k.g, bk);
  }
  allow_smem(f, smem);
  f<<<block_grid(f, bk, threads, smem), threads, smem, st>>>(k);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_kick_count(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1,
                              const Geo& g, const Blk& bk, const float* acc_c, const float* acc_f, float ck, float cd,
                              const RecompressTables& t, uint32_t* vmax_bits, uint32_t* tkey, uint4* tpv,
                              const float* vq0, const float* vq1, const float4* app, bool coarse, cudaStream_t st) {
  KickArgs k{c0, c1, off0, off1, g, bk, acc_c, acc_f, ck, cd, t, vmax_bits, tkey, tpv, vq0, vq1, app, coarse ? 1 : 0};
  k.t.kb = rank_bits(g, bk);
  set_window(g, k.bk);
  return c0.vel16 ? kick_count<true>(k, c0.n + c1.n, st) : kick_count<false>(k, c0.n + c1.n, st);
}

cudaError_t launch_kick_scatter(int64_t n0, int64_t n1, const int64_t* off0, const int64_t* off1, const Geo& g,
                                const Blk& bk, const RecompressTables& t, const int64_t* newoff0,
                                const int64_t* newoff1, const PCodesOut& o0, const PCodesOut& o1, const uint32_t* tkey,
                                const uint4* tpv, bool coded, int* status, cudaStream_t st) {
  ScatterArgs k{n0, n1, off0, off1, g, bk, t, newoff0, newoff1, o0, o1, tkey, tpv, coded ? 1 : 0, status};
  k.t.kb = rank_bits(g, bk);
  set_window(g, k.bk);
  const size_t smem = 2 * (size_t)window_cells(g, bk) * sizeof(int64_t);
  const auto f = o0.vel16 ? k_kick_scatter<true> : k_kick_scatter<false>;
  allow_smem(f, smem);
  f<<<block_grid(f, bk, kScatterThreads, smem), kScatterThreads, smem, st>>>(k);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_vmax_bound(const float* vin0, const float* vin1, const uint32_t* amax, float ck, float* vout0,
                              float* vout1, cudaStream_t st) {
  k_vmax_bound<<<1, 1, 0, st>>>(vin0, vin1, amax, ck, vout0, vout1);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pm
