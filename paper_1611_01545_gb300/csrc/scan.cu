// Cell-count scans of the cell-ordered codec (Sec. 2.4): count byte with the
// 255 escape -> CSR offsets, and cell counts -> offsets, count bytes and the
// ordered escape list.  One launch per scan, for one or two species.
//
// What bounds it: latency.  The counts of a 64^3 compression mesh are 0.5 MB,
// and the three-launch form (tile sums, scan of the sums, tile prefixes, with
// two more launches for the escape checks and the total) spent 30 us per scan
// on launches and on reading the counts twice, half of a small mesh's step.
// Here a tile of 2,048 cells is read once; its prefix over the earlier tiles
// comes from decoupled look-back (Merrill and Garland 2016): each tile
// publishes its own sum, then walks back over the published sums, a warp's 32
// at a time, until it meets a tile whose whole prefix is known.  Tiles are
// numbered by a ticket drawn when their block starts, so every tile waited for
// is already running.  Tickets count on from launch to launch and published sums
// carry their launch's number: a launch relies on nothing that an earlier one has
// to clear, and launches that overlap on one state, which callers must not let
// happen, spoil no later one.  Per scan of two species this saves 14 to 16 us on 64^3
// cells and 20 us on 16^3 (two steps and a deposit on a 64^3 mesh: 272 -> 171
// us, with the step's memsets folded in).
#include <cuda_runtime.h>
#include <stdint.h>

#include "particles.cuh"

namespace pm {

namespace {

struct V2 {
  long long a;   // particles
  int b;         // cells that need an escape entry
};
__device__ __forceinline__ V2 v2add(V2 x, V2 y) { return V2{x.a + y.a, x.b + y.b}; }

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ V2 warp_incl(V2 v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    long long a = __shfl_up_sync(0xffffffffu, v.a, o);
    int b = __shfl_up_sync(0xffffffffu, v.b, o);
    if (lane >= o) { v.a += a; v.b += b; }
  }
  return v;
}

// Exclusive block scan of one V2 per thread; returns the exclusive prefix and the block total.
__device__ __forceinline__ V2 block_excl(V2 v, V2* total) {
  constexpr int NW = SCAN_THREADS / 32;
  __shared__ V2 warp_sums[NW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const V2 inc = warp_incl(v);
  if (lane == 31) warp_sums[wid] = inc;
  __syncthreads();
  V2 before{inc.a - v.a, inc.b - v.b}, all{0, 0};
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    if (w < wid) before = v2add(before, warp_sums[w]);
    all = v2add(all, warp_sums[w]);
  }
  *total = all;
  return before;
}

// A tile's published sum in two 64-bit words, particles and cells with an escape
// entry, each under a head that says what it is: the launch's number in the top 28
// bits, then a bit for a whole prefix (else the tile's own sum).  A pair whose heads
// agree belongs together.  Below the head fit 3.4e10, more particles than a device
// can hold; a corrupt stream that claims more saturates and fails the check of the
// total.
constexpr int kHeadShift = 35;
constexpr unsigned long long kValueMask = (1ull << kHeadShift) - 1;
constexpr unsigned kLaunchMask = (1u << 28) - 1;

struct alignas(16) TileSum {
  unsigned long long a, b;
};
__device__ __forceinline__ TileSum tile_sum(V2 v, unsigned launch, bool whole) {
  const unsigned long long head = ((unsigned long long)launch << 1 | (whole ? 1u : 0u)) << kHeadShift;
  const unsigned long long a = (unsigned long long)v.a < kValueMask ? (unsigned long long)v.a : kValueMask;
  return TileSum{head | a, head | (unsigned)v.b};
}
__device__ __forceinline__ V2 value_of(const TileSum& t) {
  return V2{(long long)(t.a & kValueMask), (int)(t.b & kValueMask)};
}

// Device state of one species' scan, zeroed once before its first launch.  Every
// launch on it draws as many tickets as it has tiles, the same number each time.
struct ScanState {
  unsigned long long ticket, pad;
  __device__ TileSum* tiles() { return reinterpret_cast<TileSum*>(this + 1); }
};
static_assert(sizeof(ScanState) == 16, "one 16-byte header");

__device__ __forceinline__ TileSum load_sum(const TileSum* p) {
  TileSum t;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(t.a), "=l"(t.b) : "l"(p) : "memory");
  return t;
}
__device__ __forceinline__ void store_sum(TileSum* p, TileSum t) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(t.a), "l"(t.b) : "memory");
}

// Prefix of tile `tile` over the earlier tiles of launch number `launch`, by the
// first warp.  A wait is given up after `limit` cycles, or at once where a later
// launch has overwritten what it waits for (status ST_TIMEOUT).
constexpr long long kWaitLimit = 2000000000LL;   // about a second
__device__ __forceinline__ V2 look_back(const TileSum* tiles, int tile, unsigned launch, long long limit, int* status) {
  const int lane = threadIdx.x & 31;
  V2 sum{0, 0};
  for (int last = tile - 1; last >= 0; last -= 32) {
    const int i = last - lane;
    TileSum w = i >= 0 ? load_sum(tiles + i) : tile_sum(V2{0, 0}, launch, true);
    const auto waiting = [&] { return (unsigned)(w.a >> (kHeadShift + 1)) != launch || ((w.a ^ w.b) >> kHeadShift) != 0; };
    if (__any_sync(0xffffffffu, waiting())) {
      const long long t0 = clock64();
      while (__any_sync(0xffffffffu, waiting())) {
        if (i >= 0) w = load_sum(tiles + i);
        const unsigned ahead = ((unsigned)(w.a >> (kHeadShift + 1)) - launch) & kLaunchMask;
        const bool later = ahead != 0 && ahead <= kLaunchMask / 2;
        if (__any_sync(0xffffffffu, later || clock64() - t0 > limit)) {
          if (lane == 0) atomicOr(status, ST_TIMEOUT);
          return sum;
        }
      }
    }
    const unsigned known = __ballot_sync(0xffffffffu, (w.a >> kHeadShift & 1u) != 0);
    const int upto = known ? __ffs(known) - 1 : 31;   // nearest tile whose whole prefix is known
    V2 v = lane <= upto ? value_of(w) : V2{0, 0};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v.a += __shfl_xor_sync(0xffffffffu, v.a, o);
      v.b += __shfl_xor_sync(0xffffffffu, v.b, o);
    }
    sum = v2add(sum, v);
    if (known) break;
  }
  return sum;
}

// Counts of compression cells from the count bytes and the escape list.
struct CodesCount {
  const uint8_t* cnt;
  const uint32_t* esc;
  const uint32_t* n_esc;
  int64_t esc_cap;
  const float* vmax;
  int* status;
  __device__ V2 of(unsigned k, int64_t c) const {
    if (k != 255u) return V2{(long long)k, 0};
    long long ne = (long long)*n_esc;
    if (ne > esc_cap) ne = esc_cap;
    long long lo = 0, hi = ne - 1;
    while (lo <= hi) {
      long long mid = (lo + hi) >> 1;
      long long cm = esc[2 * mid];
      if (cm == c) return V2{(long long)esc[2 * mid + 1], 1};
      if (cm < c) lo = mid + 1; else hi = mid - 1;
    }
    atomicOr(status, ST_CORRUPT);
    return V2{0, 1};
  }
  // counts of cells c .. c + 7 below n
  __device__ void load(int64_t c, int64_t n, V2 (&v)[SCAN_ITEMS]) const {
    if (c + SCAN_ITEMS <= n && (reinterpret_cast<uintptr_t>(cnt) & 7) == 0) {
      const unsigned long long w = *reinterpret_cast<const unsigned long long*>(cnt + c);
#pragma unroll
      for (int k = 0; k < SCAN_ITEMS; ++k) v[k] = of((unsigned)(w >> (8 * k)) & 255u, c + k);
    } else {
#pragma unroll
      for (int k = 0; k < SCAN_ITEMS; ++k) v[k] = c + k < n ? of(cnt[c + k], c + k) : V2{0, 0};
    }
  }
  // Every escape entry must name a cell whose byte is 255, hold >= 255 and
  // ascend; v_max must be finite and >= 0.  Entries are dealt to the tiles.
  __device__ void validate(int tile, int tiles, int64_t ncell) const {
    long long ne = *n_esc;
    if (tile == 0 && threadIdx.x == 0) {
      const float vm = *vmax;
      if (!(vm >= 0.f) || isinf(vm)) atomicOr(status, ST_CORRUPT);
      if (ne > esc_cap) atomicOr(status, ST_CORRUPT);
    }
    if (ne > esc_cap) ne = esc_cap;
    for (long long i = (long long)tile * SCAN_THREADS + threadIdx.x; i < ne; i += (long long)tiles * SCAN_THREADS) {
      const uint32_t c = esc[2 * i], k = esc[2 * i + 1];
      const bool bad = (int64_t)c >= ncell || k < 255u || cnt[c] != 255u || (i > 0 && esc[2 * (i - 1)] >= c);
      if (bad) atomicOr(status, ST_CORRUPT);
    }
  }
};

// Counts of the recompressed cells (library memory, 16-byte aligned).
struct U32Count {
  const uint32_t* cnt;
  const uint32_t* far;   // counted apart, or null
  static __device__ V2 of(uint32_t k) { return V2{(long long)k, k >= 255u ? 1 : 0}; }
  __device__ void load(int64_t c, int64_t n, V2 (&v)[SCAN_ITEMS]) const {
    if (c + SCAN_ITEMS <= n) {
      uint4 p = reinterpret_cast<const uint4*>(cnt + c)[0], q = reinterpret_cast<const uint4*>(cnt + c)[1];
      if (far) {
        const uint4 a = reinterpret_cast<const uint4*>(far + c)[0], b = reinterpret_cast<const uint4*>(far + c)[1];
        p = make_uint4(p.x + a.x, p.y + a.y, p.z + a.z, p.w + a.w);
        q = make_uint4(q.x + b.x, q.y + b.y, q.z + b.z, q.w + b.w);
      }
      v[0] = of(p.x); v[1] = of(p.y); v[2] = of(p.z); v[3] = of(p.w);
      v[4] = of(q.x); v[5] = of(q.y); v[6] = of(q.z); v[7] = of(q.w);
    } else {
#pragma unroll
      for (int k = 0; k < SCAN_ITEMS; ++k) v[k] = c + k < n ? of(cnt[c + k] + (far ? far[c + k] : 0u)) : V2{0, 0};
    }
  }
  __device__ void validate(int, int, int64_t) const {}
};

__device__ __forceinline__ void put_offsets(int64_t* off, int64_t c, int64_t n, V2 ex, const V2 (&v)[SCAN_ITEMS]) {
  int64_t o[SCAN_ITEMS];
  o[0] = ex.a;
#pragma unroll
  for (int k = 1; k < SCAN_ITEMS; ++k) o[k] = o[k - 1] + v[k - 1].a;
  if (c + SCAN_ITEMS <= n) {
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k += 2) *reinterpret_cast<longlong2*>(off + c + k) = make_longlong2(o[k], o[k + 1]);
  } else {
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k)
      if (c + k < n) off[c + k] = o[k];
  }
}

// Decompress offsets: off[c] = sum_{c' < c} count(c').  A step also clears its
// new-cell counts here, in place of a memset of its own.
struct PutOffsets {
  int64_t* off;
  uint32_t* clear;
  uint32_t* clear2;
  __device__ void operator()(int64_t c, int64_t n, V2 ex, const V2 (&v)[SCAN_ITEMS]) const {
    put_offsets(off, c, n, ex, v);
    put_zeros(clear, c, n);
    put_zeros(clear2, c, n);
  }
  static __device__ __forceinline__ void put_zeros(uint32_t* a, int64_t c, int64_t n) {
    if (!a) return;
    if (c + SCAN_ITEMS <= n) {
      reinterpret_cast<uint4*>(a + c)[0] = make_uint4(0, 0, 0, 0);
      reinterpret_cast<uint4*>(a + c)[1] = make_uint4(0, 0, 0, 0);
    } else {
      for (int k = 0; k < SCAN_ITEMS; ++k)
        if (c + k < n) a[c + k] = 0;
    }
  }
};

// Compress outputs: CSR offsets, count bytes, ordered escape list.
struct PutCodes {
  int64_t* off;
  uint8_t* cnt;
  uint32_t* esc;
  int64_t esc_cap;
  int* status;
  __device__ void operator()(int64_t c, int64_t n, V2 ex, const V2 (&v)[SCAN_ITEMS]) const {
    put_offsets(off, c, n, ex, v);
    unsigned long long w = 0;
    int at = ex.b;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      w |= (unsigned long long)(v[k].a >= 255 ? 255 : v[k].a) << (8 * k);
      if (v[k].b) {
        if ((int64_t)at < esc_cap) {
          esc[2 * (int64_t)at] = (uint32_t)(c + k);
          esc[2 * (int64_t)at + 1] = (uint32_t)v[k].a;
        } else {
          atomicOr(status, ST_OVERFLOW);
        }
        ++at;
      }
    }
    if (c + SCAN_ITEMS <= n && (reinterpret_cast<uintptr_t>(cnt) & 7) == 0) {
      *reinterpret_cast<unsigned long long*>(cnt + c) = w;
    } else {
#pragma unroll
      for (int k = 0; k < SCAN_ITEMS; ++k)
        if (c + k < n) cnt[c + k] = (uint8_t)(w >> (8 * k));
    }
  }
};

// What the tiles of one species do beside the prefixes: the last one writes
// off[n] = total, checks it and sets n_esc if asked; the first copies v_max
// (float bits) and clears `words` 32-bit words, if asked.
struct FinishArgs {
  int64_t expect;
  int64_t* off;
  uint32_t* n_esc_out;
  int64_t esc_cap;
  const uint32_t* vmax_bits;
  float* vmax_out;
  uint32_t* clear;
  int words;
  uint4* mesh;           // and a mesh of mesh_words 16-byte words, a slice per tile and species
  int64_t mesh_words;
};

template <class T> struct Pair { T v[2]; };

template <class Get, class Put>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan(Pair<Get> gets, Pair<Put> puts, Pair<FinishArgs> fin,
                                                     int64_t n, int tiles, unsigned char* state, size_t stride,
                                                     long long limit, int* status) {
  const Get& get = gets.v[blockIdx.y];
  const FinishArgs& f = fin.v[blockIdx.y];
  ScanState* st = reinterpret_cast<ScanState*>(state + blockIdx.y * stride);
  __shared__ int s_tile;
  __shared__ unsigned s_launch;
  __shared__ V2 s_prefix;
  if (threadIdx.x == 0) {
    const unsigned long long t = atomicAdd(&st->ticket, 1ull), l = t / (unsigned)tiles;
    s_tile = (int)(t - l * (unsigned)tiles);
    s_launch = (unsigned)(l + 1) & kLaunchMask;   // (zeroed words are no launch's)
  }
  __syncthreads();
  const int tile = s_tile;
  const unsigned launch = s_launch;
  const int64_t c = (int64_t)tile * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  V2 v[SCAN_ITEMS];
  get.load(c, n, v);
  V2 own{0, 0}, total;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) own = v2add(own, v[k]);
  V2 ex = block_excl(own, &total);
  TileSum* sums = st->tiles();
  if (threadIdx.x < 32) {
    V2 before{0, 0};
    if (tile > 0) {
      if (threadIdx.x == 0) store_sum(sums + tile, tile_sum(total, launch, false));
      before = look_back(sums, tile, launch, limit, status);
    }
    if (threadIdx.x == 0) {
      store_sum(sums + tile, tile_sum(v2add(before, total), launch, true));
      s_prefix = before;
    }
  }
  get.validate(tile, tiles, n);
  if (tile == 0) {
    if (threadIdx.x == 0 && f.vmax_out) *f.vmax_out = __uint_as_float(*f.vmax_bits);
    for (int i = threadIdx.x; i < f.words; i += SCAN_THREADS) f.clear[i] = 0u;
  }
  if (f.mesh) {
    const int64_t slices = (int64_t)tiles * gridDim.y;
    const int64_t per = (f.mesh_words + slices - 1) / slices;
    const int64_t from = ((int64_t)blockIdx.y * tiles + tile) * per;
    const int64_t to = from + per < f.mesh_words ? from + per : f.mesh_words;
    for (int64_t i = from + threadIdx.x; i < to; i += SCAN_THREADS) f.mesh[i] = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  const V2 prefix = s_prefix;
  ex = v2add(ex, prefix);
  puts.v[blockIdx.y](c, n, ex, v);
  if (threadIdx.x == 0 && tile == tiles - 1) {
    const V2 t = v2add(prefix, total);
    f.off[n] = t.a;
    if (t.a != f.expect) atomicOr(status, ST_CORRUPT);
    if (f.n_esc_out) *f.n_esc_out = (uint32_t)(t.b < f.esc_cap ? t.b : f.esc_cap);
  }
}

int scan_tiles(int64_t n) { return (int)((n + SCAN_TILE - 1) / SCAN_TILE); }

// nsp (1 or 2) species in one launch.
cudaError_t scan_codes_n(const pm_codes_t* in, int nsp, int64_t ncell, int64_t* const* off, void* state, int* status,
                         const ScanClear* clear, cudaStream_t st) {
  Pair<CodesCount> get{};
  Pair<PutOffsets> put{};
  Pair<FinishArgs> fin{};
  for (int s = 0; s < nsp; ++s) {
    get.v[s] = CodesCount{in[s].cnt, in[s].esc, in[s].n_esc, in[s].esc_cap, in[s].vmax, status};
    put.v[s] = PutOffsets{off[s], clear ? clear->counts[s] : nullptr, clear ? clear->far[s] : nullptr};
    fin.v[s] = FinishArgs{in[s].n, off[s], nullptr, 0, nullptr, nullptr, s == 0 && clear ? clear->small : nullptr,
                          s == 0 && clear ? clear->small_words : 0,
                          clear ? static_cast<uint4*>(clear->mesh) : nullptr, clear ? clear->mesh_words : 0};
  }
  const int tiles = scan_tiles(ncell);
  k_scan<<<dim3(tiles, nsp), SCAN_THREADS, 0, st>>>(get, put, fin, ncell, tiles, static_cast<unsigned char*>(state),
                                                    scan_state_bytes(ncell), kWaitLimit, status);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t scan_counts_n(const uint32_t* const* counts, const uint32_t* const* far, int nsp, int64_t ncell, const int64_t* expect,
                          int64_t* const* off, pm_codes_t* out, const uint32_t* const* vmax_bits, void* state,
                          int* status, cudaStream_t st) {
  Pair<U32Count> get{};
  Pair<PutCodes> put{};
  Pair<FinishArgs> fin{};
  for (int s = 0; s < nsp; ++s) {
    get.v[s] = U32Count{counts[s], far ? far[s] : nullptr};
    put.v[s] = PutCodes{off[s], out[s].cnt, out[s].esc, out[s].esc_cap, status};
    fin.v[s] = FinishArgs{expect[s], off[s], out[s].n_esc, out[s].esc_cap, vmax_bits[s],
                          vmax_bits[s] ? out[s].vmax : nullptr, nullptr, 0, nullptr, 0};
  }
  const int tiles = scan_tiles(ncell);
  k_scan<<<dim3(tiles, nsp), SCAN_THREADS, 0, st>>>(get, put, fin, ncell, tiles, static_cast<unsigned char*>(state),
                                                    scan_state_bytes(ncell), kWaitLimit, status);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// State of one species' scan; the two-species scans use twice this.  Zero it once.
size_t scan_state_bytes(int64_t ncell) { return sizeof(ScanState) + sizeof(TileSum) * (size_t)scan_tiles(ncell); }

cudaError_t scan_codes(const pm_codes_t& in, int64_t ncell, int64_t* off, void* state, int* status,
                       cudaStream_t st) {
  int64_t* offs[1] = {off};
  return scan_codes_n(&in, 1, ncell, offs, state, status, nullptr, st);
}

cudaError_t scan_codes2(const pm_codes_t in[2], int64_t ncell, int64_t* off0, int64_t* off1, void* state, int* status,
                        const ScanClear* clear, cudaStream_t st) {
  int64_t* offs[2] = {off0, off1};
  return scan_codes_n(in, 2, ncell, offs, state, status, clear, st);
}

cudaError_t scan_counts(const uint32_t* counts, int64_t ncell, int64_t expect, int64_t* off, pm_codes_t& out,
                        const uint32_t* vmax_bits, void* state, int* status, cudaStream_t st) {
  const uint32_t* c[1] = {counts};
  const uint32_t* vb[1] = {vmax_bits};
  int64_t* o[1] = {off};
  return scan_counts_n(c, nullptr, 1, ncell, &expect, o, &out, vb, state, status, st);
}

cudaError_t scan_counts2(const uint32_t* const counts[2], const uint32_t* const far[2], int64_t ncell,
                         const int64_t expect[2], int64_t* off0, int64_t* off1, pm_codes_t out[2],
                         const uint32_t* vmax_bits, void* state, int* status, cudaStream_t st) {
  const uint32_t* vb[2] = {vmax_bits, vmax_bits ? vmax_bits + 1 : nullptr};
  int64_t* o[2] = {off0, off1};
  return scan_counts_n(counts, far, 2, ncell, expect, o, out, vb, state, status, st);
}

}  // namespace pm
