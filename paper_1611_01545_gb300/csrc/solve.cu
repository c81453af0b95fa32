// Fourier-space PM solve on periodic windows (paper Sec. 2.1, Eqs. 1-3).
//
// One "problem" is an N^3 window of a periodic source mesh whose cell 0 sits
// at origin p*t - b (p = problem coordinates): the whole coarse / single mesh
// (t = N, b = 0), or one buffered fine tile (Fig. 1; N = T = t + 2b).  Three
// kernels per batch of problems:
//   A  per z plane: load the real window plane, real-to-complex along x (two
//      rows packed as one complex row), complex FFT along y -> half spectrum;
//   B  per ky: FFT along z, multiply by the precomputed kernel of each force
//      component (i K_d), inverse FFT along z, keep the output z range;
//   C  per (output z, component): inverse FFT along y, complex-to-real along
//      x (two rows packed), store the output interior into the destination
//      mesh [3][n][n][n].
// The kernel tables already contain the 1/N^3 (tiles) or 1/V (periodic)
// normalisation, so both transform directions are unnormalised.
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include "fft.cuh"
#include "pm_common.cuh"
#include "tma.cuh"

namespace pm {
using namespace pmfft;

template <int N> struct SolveCfg {
  static constexpr int NH = N / 2 + 1;
  static constexpr int NP = spec_pitch(N);   // row pitch (complex values) of the spectrum buffers
// Compile-time tunables of the 96^3 passes (the alternatives' times stand at each
// pass): threads of pass A, blocks per SM of A and C, columns, threads and blocks
// per SM of pass B.
#ifndef PM_SOLVE_THREADS
#define PM_SOLVE_THREADS 416
#endif
#ifndef PM_SOLVE_A_MINB
#define PM_SOLVE_A_MINB 3
#endif
#ifndef PM_PASSB_KT
#define PM_PASSB_KT 18
#endif
#ifndef PM_PASSB_TMA_THREADS
#define PM_PASSB_TMA_THREADS 160
#endif
#ifndef PM_PASSB_TMA_MINB
#define PM_PASSB_TMA_MINB 5
#endif
#ifndef PM_SOLVE_C_MINB
#define PM_SOLVE_C_MINB 4
#endif
};

struct SolveArgs {
  const void* src;
  int src_n;
  int nts;
  int t, b;
  int p0;
  float2* spec;
  float2* spec3;
  const float* kern;
  const float4* kern_quads;   // pass B's layout of the kernel (null above 128)
  const float2* tw;
  float* dst;
  int comp_mode;   // pass A only: blockIdx.y selects component pb of a 3-component source at origin 0
  unsigned int* amax;   // pass C: if set, atomicMax of max |output| (float bits; values are >= 0)
  const float* pc;      // pass C: if set, add this coarse force [3][pnc^3] trilinearly prolongated to the fine nodes
  int pnc, prc;         // its edge and the fine cells per coarse cell (a power of two dividing t)
  int* status;          // library status word: ST_TIMEOUT when a bounded copy wait gives up
};

__device__ __forceinline__ int pmod(int a, int n) {
  int r = a % n;
  return r < 0 ? r + n : r;
}

__device__ __forceinline__ void problem_origin(const SolveArgs& a, int p, int& ox, int& oy, int& oz) {
  int px = p % a.nts, py = (p / a.nts) % a.nts, pz = p / (a.nts * a.nts);
  ox = px * a.t - a.b;
  oy = py * a.t - a.b;
  oz = pz * a.t - a.b;
}

// Row loops below give each warp whole rows and each lane strided columns, so
// row indices are computed once per row and no division is needed.
// Global -> shared copies that do not stall the issuing thread (cp.async);
// async_wait() waits for all of the thread's copies (a barrier must follow).
__device__ __forceinline__ void async_copy4(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)),
               "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void async_copy8(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)),
               "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

#define PM_ROWS(row, nrows) for (int row = threadIdx.x >> 5; row < (nrows); row += (blockDim.x >> 5))
#define PM_COLS(col, ncols) for (int col = threadIdx.x & 31; col < (ncols); col += 32)

template <bool FIXED>
__device__ __forceinline__ float src_value(const void* src, int64_t idx) {
  if (FIXED) return (float)((double)static_cast<const long long*>(src)[idx] * 2.3283064365386963e-10);  // 2^-32
  return __ldg(static_cast<const float*>(src) + idx);
}

__device__ __forceinline__ int wrap1(int g, int n) { return g < 0 ? g + n : (g >= n ? g - n : g); }

// Pass B works on one ky row and one chunk of KC kx columns (KC = ceil(NH/2),
// i.e. two chunks, up to N = 128): forward z FFT, the three
// kernel products i K_d F written side by side, then one batched inverse z
// FFT over all 3 KC columns, so a block needs only a few barriers.
// Large meshes (N > 128) take 16 columns per block, so their z columns fit.
template <int N> struct PassB {
  static constexpr int NH = N / 2 + 1;
  static constexpr int KC = N > 128 ? 16 : (NH + 1) / 2;
  static constexpr int nchunk = (NH + KC - 1) / KC;
#ifndef PM_PASSB_THREADS
#define PM_PASSB_THREADS 512
#endif
  static constexpr int threads = N > 128 ? 256 : ((N >= 96) ? PM_PASSB_THREADS : 256);
  // twiddles + [z][3 KC]: the forward transform runs in the first KC columns
  static constexpr size_t smem = sizeof(float2) * (N + 3 * (size_t)N * KC);
};

template <int N>
__device__ __forceinline__ void solve_b_body(const SolveArgs& a) {
  constexpr int NH = PassB<N>::NH, KC = PassB<N>::KC, NP = SolveCfg<N>::NP;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  // [z][3 KC]: component d of the products in columns d KC .. d KC + KC - 1; the
  // density spectrum F is transformed in the columns of component 0 and each
  // thread overwrites its element with the three products (in place for d = 0)
  float2* G = sm + N;
  float2* F = G;
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = a.tw[i];
  const int ys = blockIdx.x;      // ky in slot order
  const int half = blockIdx.y;    // which chunk of the kx columns
  const int pb = blockIdx.z;
  const int kx0 = half * KC;
  const int ncol = (NH - kx0) < KC ? (NH - kx0) : KC;
  const float2* in = a.spec + (size_t)pb * N * N * NP + (size_t)ys * NP + kx0;
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
    const int z = i / KC, c = i - z * KC;
    if (c < ncol) async_copy8(F + z * 3 * KC + c, in + (size_t)z * N * NP + c);
    else F[z * 3 * KC + c] = make_float2(0.f, 0.f);
  }
  async_wait();
  __syncthreads();
  fft_fwd<N, KC, 1, 3 * KC>(F, tw);
  const float* K = a.kern + (size_t)ys * NH + kx0;
  const size_t kstride = (size_t)N * N * NH;
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
    const int zs = i / KC, c = i - zs * KC;
    float2* g = G + zs * 3 * KC + c;
    const float2 f = g[0];
    if (c < ncol) {
      const float* Kz = K + (size_t)zs * N * NH + c;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float k = __ldg(Kz + d * kstride);
        g[d * KC] = make_float2(-f.y * k, f.x * k);   // i K f
      }
    } else {
#pragma unroll
      for (int d = 0; d < 3; ++d) g[d * KC] = make_float2(0.f, 0.f);
    }
  }
  __syncthreads();
  fft_inv<N, 3 * KC, 1, 3 * KC>(G, tw);
  for (int d = 0; d < 3; ++d) {
    float2* out = a.spec3 + ((size_t)pb * 3 + d) * a.t * N * NP + (size_t)ys * NP + kx0;
    for (int i = threadIdx.x; i < a.t * KC; i += blockDim.x) {
      const int zo = i / KC, c = i - zo * KC;
      if (c < ncol) out[(size_t)zo * N * NP + c] = G[(zo + a.b) * 3 * KC + d * KC + c];
    }
  }
}

template <int N>
__global__ void __launch_bounds__(PassB<N>::threads) k_large_b(SolveArgs a) {
  solve_b_body<N>(a);
}

// Transpose of the solve for one periodic mesh (the adjoint of a_d = K_d * rho):
// the three component spectra (pass A with comp_mode) are z-transformed, each
// multiplied by the conjugate kernel conj(i K_d) = -i K_d and summed, and the
// sum is inverse z-transformed into component slot 0 of spec3; pass C then
// gives the scalar result.
template <int N>
__global__ void __launch_bounds__(PassB<N>::threads) k_solve_b_adj(SolveArgs a) {
  constexpr int NH = PassB<N>::NH, KC = PassB<N>::KC, NP = SolveCfg<N>::NP;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* F = sm + N;             // [z][KC]
  float2* G = F + N * KC;         // [z][KC]
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = a.tw[i];
  const int ys = blockIdx.x, half = blockIdx.y;
  const int kx0 = half * KC;
  const int ncol = (NH - kx0) < KC ? (NH - kx0) : KC;
  const size_t kstride = (size_t)N * N * NH;
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) G[i] = make_float2(0.f, 0.f);
  for (int d = 0; d < 3; ++d) {
    const float2* in = a.spec + (size_t)d * N * N * NP + (size_t)ys * NP + kx0;
    for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
      const int z = i / KC, c = i - z * KC;
      F[i] = c < ncol ? in[(size_t)z * N * NP + c] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    fft_fwd<N, KC, 1, KC>(F, tw);
    const float* K = a.kern + d * kstride + (size_t)ys * NH + kx0;
    for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
      const int zs = i / KC, c = i - zs * KC;
      if (c < ncol) {
        const float k = __ldg(K + (size_t)zs * N * NH + c);
        const float2 f = F[i];
        G[i] = make_float2(G[i].x + f.y * k, G[i].y - f.x * k);   // += -i K f
      }
    }
    __syncthreads();
  }
  fft_inv<N, KC, 1, KC>(G, tw);
  float2* out = a.spec3 + (size_t)ys * NH + kx0;   // spec3 rows have no padding
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
    const int z = i / KC, c = i - z * KC;
    if (c < ncol) out[(size_t)z * N * NH + c] = G[i];
  }
}

// ---- copies by the tensor memory accelerator ---------------------------------
//
// Where the shapes allow it, planes and pencils move between global and shared
// memory as TMA bulk copies instead of per-thread copies:
//   A  96^3 windows of float meshes on 16-cell boundaries arrive as 36 boxes of
//      16 x 16 cells (a tensor map of the source mesh; window origins are multiples
//      of 16 cells, so no box crosses the periodic boundary), from which the first
//      transform step reads; at every size the half-spectrum plane leaves as one
//      bulk store;
//   B  at 96 the z pencils of 18 kx columns arrive as one box of 36 floats x 1 x 96
//      of the spectrum (columns past kx = N / 2 read as zeros); the output rows are
//      written from registers;
//   C  at every size the plane arrives as one bulk load.
// The spectrum rows between A and B are padded to spec_pitch(96) = 50 complex values
// (400 bytes), so rows, boxes and planes start on 16-byte boundaries.

constexpr int kTmaAlign = 128;   // shared-memory alignment of every TMA destination and source
constexpr int kBox = 16;         // edge (cells) of the pass-A window boxes

__device__ __forceinline__ unsigned char* tma_align(unsigned char* p) {
  const unsigned a = tma::smem_u32(p);
  return p + ((kTmaAlign - (a & (kTmaAlign - 1))) & (kTmaAlign - 1));
}

// Bounded wait of the whole block for phase 0 of `bar`.  When it gives up
// (the copies did not complete in time) the block records ST_TIMEOUT, waits
// once more (bounded) for copies still in flight, and the caller returns.
__device__ __forceinline__ bool block_wait(uint64_t* bar, int* status) {
  int bad = tma::mbar_wait(bar, 0) ? 0 : 1;
  bad = __syncthreads_or(bad);
  if (bad) {
    if (threadIdx.x == 0 && status) atomicOr(status, ST_TIMEOUT);
    tma::mbar_wait(bar, 0);
  }
  return !bad;
}

// ---- pass A ---------------------------------------------------------------
//
// One block per z plane of a window: real-to-complex along x (two rows packed
// as one complex row), complex along y.  Bound by shared memory like pass C:
// the earlier form moved 6,860 wavefronts per 96^3 tile plane (2,670 of them
// bank conflicts) at 83% of the load/store pipe, 0.161 ms for 64 tiles.  Here
//   * the first x step takes its inputs from the staged window boxes, without
//     a repacking pass: a half warp reads consecutive cells of one row, the two
//     halves of a warp their two rows in opposite order, so that they meet in
//     different banks;
//   * the packed rows have pitch N + 1 (odd) and the second x step gives a
//     warp's lanes different rows; it leaves the spectrum in natural order
//     (its items are in registers across a barrier, slots and frequencies
//     overlap);
//   * the packed rows are taken apart inside the first y step, two rows per item.
// 3,100 wavefronts per plane: 0.124 ms; 216 tiles of 48^3: 0.094 -> 0.075 ms;
// 416 threads against 384: 0.124 and 0.125 ms.
// Sources that are not staged by TMA (int64 meshes, interleaved components,
// other sizes) are copied to the packed rows directly.
enum SourceForm { SRC_FLOAT, SRC_FIXED, SRC_INTERLEAVED, SRC_BOXES };

template <int N> struct PassA {
  static constexpr int N1 = Factor<N>::N1, N2 = Factor<N>::N2;
  static constexpr int NH = N / 2 + 1, NP = spec_pitch(N), WP = N + 1, NB = N / kBox;
  static constexpr bool in_place = N >= 128;   // P over W: 67 KB at 128, so that 2 blocks share an SM
  static constexpr int threads = N == 128 ? 544 : (N == 96 ? PM_SOLVE_THREADS : (N == 64 ? 288 : (N == 48 ? 160 : (N == 32 ? 96 : 64))));
  static constexpr int min_blocks = N == 128 ? 2 : (N == 96 ? PM_SOLVE_A_MINB : 4);
  static constexpr size_t w_vals = ((size_t)N / 2 * WP + 1) / 2 * 2;
  // P [N][NP] (first the staged boxes), twiddles, W [N/2][WP]
  static constexpr size_t smem = kTmaAlign + sizeof(float2) * ((size_t)N * NP + N + (in_place ? 0 : w_vals));
};

template <int N, int SRC>
__global__ void __launch_bounds__(PassA<N>::threads, PassA<N>::min_blocks)
    k_solve_a(SolveArgs a, const __grid_constant__ CUtensorMap src_map) {
  using A = PassA<N>;
  constexpr int N1 = A::N1, N2 = A::N2, NH = A::NH, NP = A::NP, WP = A::WP, T = A::threads;
  constexpr int NB = A::NB > 0 ? A::NB : 1;
  extern __shared__ unsigned char smraw_a[];
  __shared__ uint64_t bar;
  float2* P = reinterpret_cast<float2*>(tma_align(smraw_a));    // [y][NP]
  float2* tw = P + N * NP;
  float2* W = A::in_place ? P : tw + N;                           // [row pair][WP]
  float* S = reinterpret_cast<float*>(P);                         // box (yb, xb) at S + (yb NB + xb) 256
  const int z = blockIdx.x, pb = blockIdx.y;
  int ox, oy, oz;
  problem_origin(a, a.p0 + pb, ox, oy, oz);
  const int n = a.src_n;
  const void* src = a.src;
  if (a.comp_mode) {
    ox = oy = oz = 0;
    src = static_cast<const float*>(a.src) + (SRC == SRC_INTERLEAVED ? (size_t)pb : (size_t)pb * n * n * n);
  }
  for (int i = threadIdx.x; i < N; i += T) tw[i] = a.tw[i];
  // origins lie in (-n, n) and N <= n, so one conditional wrap suffices
  const int gz = wrap1(oz + z, n);
  if constexpr (SRC == SRC_BOXES) {
    static_assert((size_t)NB * NB * kBox * kBox <= (size_t)2 * N * NP, "staged window must fit in P");
    if (threadIdx.x == 0) {
      tma::mbar_init(&bar, 1);
      tma::fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      if (threadIdx.x == 0) tma::mbar_arrive_expect_tx(&bar, NB * NB * kBox * kBox * (unsigned)sizeof(float));
      __syncwarp();
      for (int k = threadIdx.x; k < NB * NB; k += 32) {
        const int yb = k / NB, xb = k - yb * NB;
        tma::tensor_load_3d(S + k * kBox * kBox, &src_map, wrap1(ox + kBox * xb, n), wrap1(oy + kBox * yb, n), gz,
                            &bar);
      }
    }
    if (!block_wait(&bar, a.status)) return;
    // x step 1 from the boxes: 16 lanes per row pair j, N2 of them with an item j2
    static_assert(N2 <= 16, "a half warp per row pair");
    for (int w = threadIdx.x; w < (N / 2) * 16; w += T) {
      const int j = w >> 4, j2 = w & 15;
      if (j2 < N2) {
        const int first = (threadIdx.x >> 4) & 1;   // the row this half warp reads first
        const float* s0 = S + (2 * j / kBox) * NB * kBox * kBox + (2 * j % kBox) * kBox + first * kBox;
        const int other = first ? -kBox : kBox;
        float2 v[N1];
#pragma unroll
        for (int j1 = 0; j1 < N1; ++j1) {
          const int x = N2 * j1 + j2;
          const float* q = s0 + (x / kBox) * kBox * kBox + x % kBox;
          const float p0 = q[0], p1 = q[other];
          v[j1] = first ? make_float2(p1, p0) : make_float2(p0, p1);
        }
        Dft<N1, -1>::run(v);
#pragma unroll
        for (int k1 = 1; k1 < N1; ++k1) v[k1] = cmul(v[k1], tw[j2 * k1]);
        float2* base = W + j * WP + j2;
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) base[N2 * k1] = v[k1];
      }
    }
  } else {
    constexpr int CS = SRC == SRC_INTERLEAVED ? 4 : 1;
    PM_ROWS(y, N) {
      const int64_t rowbase = ((int64_t)gz * n + wrap1(oy + y, n)) * n;
      float* w = reinterpret_cast<float*>(W + (y >> 1) * WP) + (y & 1);
      if (SRC == SRC_FIXED) {
        PM_COLS(x, N) w[2 * x] = src_value<true>(src, rowbase + wrap1(ox + x, n));
      } else {
        const float* srow = static_cast<const float*>(src) + rowbase * CS;
        PM_COLS(x, N) async_copy4(w + 2 * x, srow + wrap1(ox + x, n) * CS);
      }
    }
    if (SRC != SRC_FIXED) async_wait();
    __syncthreads();
    // x step 1: items (j2, row pair), in place
    for (int w = threadIdx.x; w < N2 * (N / 2); w += T) {
      const int j2 = w / (N / 2), j = w - j2 * (N / 2);
      float2* base = W + j * WP + j2;
      float2 v[N1];
#pragma unroll
      for (int j1 = 0; j1 < N1; ++j1) v[j1] = base[N2 * j1];
      Dft<N1, -1>::run(v);
#pragma unroll
      for (int k1 = 1; k1 < N1; ++k1) v[k1] = cmul(v[k1], tw[j2 * k1]);
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) base[N2 * k1] = v[k1];
    }
  }
  __syncthreads();
  // x step 2: items (k1, row pair), one round; slots N2 k1 + j2 -> frequencies k1 + N1 k2
  {
    static_assert(N1 * (N / 2) <= T, "one round");
    const int w = threadIdx.x;
    const bool live = w < N1 * (N / 2);
    const int k1 = w / (N / 2), j = w - k1 * (N / 2);
    float2 v[N2];
    if (live) {
#pragma unroll
      for (int j2 = 0; j2 < N2; ++j2) v[j2] = W[j * WP + N2 * k1 + j2];
      Dft<N2, -1>::run(v);
    }
    __syncthreads();
    if (live) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) W[j * WP + k1 + N1 * k2] = v[k2];
    }
  }
  __syncthreads();
  // y step 1: items (two neighbouring j2 = rows of one pair, column).  The two
  // real rows of a pair: (Z_k + conj Z_-k) / 2 and (Z_k - conj Z_-k) / (2i).
  {
    static_assert(!A::in_place || (N2 / 2) * NH <= T, "in place: one round");
    for (int w0 = 0; w0 < (N2 / 2) * NH; w0 += T) {
      const int w = w0 + threadIdx.x;
      const bool live = w < (N2 / 2) * NH;
      const int jp = live ? w / NH : 0, c = live ? w - jp * NH : 0;
      const int cm = c == 0 ? 0 : N - c;
      float2 u[N1], v[N1];
#pragma unroll
      for (int j1 = 0; j1 < N1; ++j1) {
        const float2* row = W + ((N2 / 2) * j1 + jp) * WP;
        const float2 zk = row[c], zm = row[cm];
        u[j1] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        v[j1] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
      }
      Dft<N1, -1>::run(u);
      Dft<N1, -1>::run(v);
#pragma unroll
      for (int k1 = 1; k1 < N1; ++k1) {
        u[k1] = cmul(u[k1], tw[2 * jp * k1]);
        v[k1] = cmul(v[k1], tw[(2 * jp + 1) * k1]);
      }
      if (A::in_place) __syncthreads();   // every packed row is read before P overwrites it
      if (live) {
        float2* base = P + 2 * jp * NP + c;
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
          base[N2 * k1 * NP] = u[k1];
          base[(N2 * k1 + 1) * NP] = v[k1];
        }
      }
    }
  }
  __syncthreads();
  // y step 2: items (k1, column), in place
  for (int w = threadIdx.x; w < N1 * NH; w += T) {
    const int k1 = w / NH, c = w - k1 * NH;
    float2* base = P + N2 * k1 * NP + c;
    float2 v[N2];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) v[j2] = base[j2 * NP];
    Dft<N2, -1>::run(v);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) base[k2 * NP] = v[k2];
  }
  // (the pitch's pad columns are stored too and never read)
  tma::fence_proxy_async();
  __syncthreads();
  if (threadIdx.x == 0) {
    tma::bulk_store(a.spec + ((size_t)pb * N + z) * N * NP, P, (unsigned)(N * NP * sizeof(float2)));
    tma::bulk_commit();
    tma::bulk_wait_all();
  }
}

// ---- pass B ---------------------------------------------------------------
//
// One block per ky row and KT kx columns: the forward z transform, the three
// kernel products and their inverse z transforms.  The second step of the
// forward transform, the products and the first step of each inverse transform
// run in registers per (k1, column) item; the second inverse step writes its
// output rows straight to global memory (KT consecutive complex values each),
// where it wrote all N rows to shared memory and a box store read back the
// output ones (3,140 -> 2,300 wavefronts per block of 96 x 26).  The kernel
// values lie in the order the items read them, 16 bytes per load, the first
// component's fetched before the spectrum arrives and the next one's while the
// current transform runs: 36 4-byte loads per item, each component's waited for
// in turn, kept the earlier form at 0.212 ms for 64 tiles; 0.206 now, and 0.196
// with 18 columns and 160 threads at 5 blocks per SM (18 x 224 at 4: 0.199;
// 26 x 320 at 3: 0.197).  216 tiles of 48^3 0.163 -> 0.089 ms (224 threads at 3
// blocks per SM 0.100, 13 columns with 128 threads 0.107 and 0.092 at 5 and 8).
template <int N> struct PassBR {
  static constexpr int NH = N / 2 + 1, NP = spec_pitch(N);
  // columns per block (N = 96: box rows of whole 16-byte words), and threads
  // that take each item set in few, full rounds
  static constexpr int KT = N == 128 ? 22 : (N == 96 ? PM_PASSB_KT : (N == 64 ? 17 : NH));
  static constexpr int nchunk = (NH + KT - 1) / KT;
  static constexpr int threads = N == 128 ? 192 : (N == 96 ? PM_PASSB_TMA_THREADS : (N == 16 ? 64 : 160));
  static constexpr int min_blocks = N == 128 ? 3 : (N == 96 ? PM_PASSB_TMA_MINB : (N == 48 ? 5 : 4));
  // G [3][N][KT] (component, z, column; the forward transform in component 0), twiddles
  static constexpr size_t smem = kTmaAlign + sizeof(float2) * (3 * (size_t)N * KT + N);
};

// Kernel values of one item and component: N2 / 4 words of 16 bytes, items
// next to each other (kernel_quads lays them out so).
template <int N>
__device__ __forceinline__ void load_quads(float4 (&k)[Factor<N>::N2 / 4], const float4* p) {
#pragma unroll
  for (int q = 0; q < Factor<N>::N2 / 4; ++q) k[q] = __ldg(p + q * PassBR<N>::KT * Factor<N>::N1);
}

template <int N>
__global__ void __launch_bounds__(PassBR<N>::threads, PassBR<N>::min_blocks)
    k_solve_b(SolveArgs a, const __grid_constant__ CUtensorMap spec_map) {
  using B = PassBR<N>;
  constexpr int NH = B::NH, NP = B::NP, KT = B::KT, T = B::threads;
  constexpr int N1 = Factor<N>::N1, N2 = Factor<N>::N2;
  extern __shared__ unsigned char smraw_b[];
  __shared__ uint64_t bar;
  float2* G = reinterpret_cast<float2*>(tma_align(smraw_b));   // [3][N][KT]
  float2* tw = G + 3 * N * KT;
  const int ys = blockIdx.x, kx0 = blockIdx.y * KT, pb = blockIdx.z;
  const int ncol = NH - kx0 < KT ? NH - kx0 : KT;
  // kernel values of this thread's first item and component: on their way
  // while the spectrum is loaded and its first transform step runs
  const float4* Kb = a.kern_quads + (size_t)(ys * B::nchunk + blockIdx.y) * (3 * (N2 / 4) * KT * N1);
  float4 kq[N2 / 4];
  if (threadIdx.x < KT * N1) load_quads<N>(kq, Kb + threadIdx.x);
  for (int i = threadIdx.x; i < N; i += T) tw[i] = a.tw[i];
  if constexpr (N == 96) {
    if (threadIdx.x == 0) {
      tma::mbar_init(&bar, 1);
      tma::fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      tma::mbar_arrive_expect_tx(&bar, N * KT * (unsigned)sizeof(float2));
      tma::tensor_load_3d(G, &spec_map, 2 * kx0, ys, pb * N, &bar);
    }
    if (!block_wait(&bar, a.status)) return;
  } else {
    const float2* in = a.spec + ((size_t)pb * N * N + ys) * NP + kx0;
    for (int i = threadIdx.x; i < N * KT; i += T) {
      const int z = i / KT, c = i - z * KT;
      if (c < ncol) async_copy8(G + i, in + (size_t)z * N * NP + c);
      else G[i] = make_float2(0.f, 0.f);
    }
    async_wait();
    __syncthreads();
  }
  // forward z transform, step 1: items (j2, column), in component 0
  for (int w = threadIdx.x; w < KT * N2; w += T) {
    const int j2 = w / KT, c = w - j2 * KT;
    float2* base = G + j2 * KT + c;
    float2 v[N1];
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) v[j1] = base[N2 * j1 * KT];
    Dft<N1, -1>::run(v);
#pragma unroll
    for (int k1 = 1; k1 < N1; ++k1) v[k1] = cmul(v[k1], tw[j2 * k1]);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) base[N2 * k1 * KT] = v[k1];
  }
  __syncthreads();
  // forward step 2, the products i K_d F and step 1 of each inverse
  // transform, per (k1, column) item: F(kz = k1 + N1 k2) sits at slot N2 k1 + k2
  for (int w = threadIdx.x; w < KT * N1; w += T) {
    const int k1 = w / KT, c = w - k1 * KT;
    float2 f[N2];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) f[j2] = G[(N2 * k1 + j2) * KT + c];
    Dft<N2, -1>::run(f);
    if (w >= T) load_quads<N>(kq, Kb + w);   // later rounds (the first one's are loaded already)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float2 g[N2];
#pragma unroll
      for (int q = 0; q < N2 / 4; ++q) {
        const float k[4] = {kq[q].x, kq[q].y, kq[q].z, kq[q].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) g[4 * q + e] = make_float2(-f[4 * q + e].y * k[e], f[4 * q + e].x * k[e]);   // i K f
      }
      if (d < 2) load_quads<N>(kq, Kb + (size_t)(d + 1) * (N2 / 4) * KT * N1 + w);   // in flight during this transform
      Dft<N2, 1>::run(g);
#pragma unroll
      for (int j2 = 1; j2 < N2; ++j2) g[j2] = cmul(g[j2], conjf2(tw[j2 * k1]));
      float2* gd = G + d * N * KT + N2 * k1 * KT + c;
#pragma unroll
      for (int j2 = 0; j2 < N2; ++j2) gd[j2 * KT] = g[j2];
    }
  }
  __syncthreads();
  // inverse step 2: items (component, j2, column) -> rows z = N2 j1 + j2 of the output range
  float2* out = a.spec3 + ((size_t)pb * 3 * a.t * N + ys) * NH + kx0;
  for (int w = threadIdx.x; w < 3 * KT * N2; w += T) {
    const int d = w / (KT * N2), r = w - d * KT * N2;
    const int j2 = r / KT, c = r - j2 * KT;
    const float2* base = G + d * N * KT + j2 * KT + c;
    float2 v[N1];
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) v[k1] = base[N2 * k1 * KT];
    Dft<N1, 1>::run(v);
    if (c < ncol) {
      const int z0 = j2 - a.b;
      float2* o = out + (ptrdiff_t)(d * a.t + z0) * N * NH + c;
#pragma unroll
      for (int j1 = 0; j1 < N1; ++j1) {
        const int zo = z0 + N2 * j1;
        if ((unsigned)zo < (unsigned)a.t) o[(size_t)N2 * j1 * N * NH] = v[j1];
      }
    }
  }
}

// ---- pass C ---------------------------------------------------------------
//
// One block per (output z, component): the plane's inverse y transform, the
// packed inverse x transform of the output rows, the prolongated coarse force,
// the store and the running max |a|.  What bounds it is shared memory: the
// earlier form moved 5,280 128-byte wavefronts per 96^3 tile plane, 1,650 of
// them bank conflicts, at 75% of the load/store pipe, and took 0.288 ms for 64
// tiles (0.226 without the prolongation).  Here
//   * an item of the second y step transforms two neighbouring rows at once;
//   * the x steps give a warp's lanes different row pairs (odd pitches: the x
//     step's reads of the pairs are 2 deep in a bank where rows are kept in
//     place, all else conflict free) where lanes along a row met 2 to 4 deep;
//   * the output takes a pair's two rows from one 8-byte word and the four rows
//     between two coarse rows from one x interpolation each of the coarse force
//     (fetched while the plane is on its way);
//   * for N >= 96 the rows stay in place and the x step holds its items in
//     registers across a barrier: one buffer (38 KB at 96, 67 KB at 128) instead
//     of two, so 4 blocks of 256 threads share an SM (2 of 544 at 128); smaller
//     sizes write the output rows to a second buffer, both rows of a pair in one
//     16-byte word.
// 64 tiles of 96^3 0.291 -> 0.197 ms (two buffers, 3 blocks of 384: 0.221; 5
// blocks of 256 with 48 registers: 0.199), 216 tiles of 48^3 0.182 -> 0.097 ms
// (compiled for 8 blocks per SM; for 4 0.102),
// 128^3 mesh 33 -> 21 us.  Bound by issue now (75% of the slots).  The spectrum
// rows between passes B and C are not padded: pass B's stores take 0.182 ms with
// them in place of 0.195.

// w / n for 0 <= w < 4096, n >= 1, with inv = 1 / n (w + 1/2 keeps the product
// away from whole numbers by more than its rounding).
__device__ __forceinline__ int quick_div(int w, float inv) { return (int)(((float)w + 0.5f) * inv); }

template <int N> struct PassC {
  static constexpr int N1 = Factor<N>::N1, N2 = Factor<N>::N2;
  static constexpr int NH = N / 2 + 1, NP = N / 2 + 1;   // spec3 rows have no padding
  static constexpr bool in_place = N >= 96;
  // in place the x step's items are one round: 256 threads serve 32 row pairs of
  // 96 (the buffered tiles), 384 all 48; else one round of the largest item set
  static constexpr int threads = N == 128 ? 544 : (N == 96 ? 384 : (N == 64 ? 288 : (N == 48 ? 160 : 96)));
  static constexpr int min_blocks(int t) { return N == 128 ? 2 : (N == 96 ? (t == 256 ? PM_SOLVE_C_MINB : 3) : (N == 48 ? 8 : 4)); }
  static constexpr size_t align = 128;
  // P [N][NP] (then W [pairs][N + 1]), twiddles, Y [pairs][NH] 16-byte words or, in place, room for the prolongation
  static size_t smem(int t, int b, int prc, bool prolong) {
    const size_t pairs = pair_count(t, b);
    const size_t nq = prolong ? t / prc + 1 : 0;
    return align + sizeof(float2) * ((size_t)N * NP + N) + (in_place ? 4 * nq * nq : 16 * pairs * NH);
  }
  static size_t smem_max() { return align + sizeof(float2) * ((size_t)N * NP + N) + (size_t)16 * (N / 2) * NH; }
  static bool narrow(int t, int b) { return N == 96 && pair_count(t, b) * N1 <= 256; }
  // row pairs (2 m, 2 m + 1) that hold the output rows b .. b + t - 1
  static __host__ __device__ __forceinline__ int pair_count(int t, int b) { return ((b + t - 1) >> 1) - (b >> 1) + 1; }
};

template <int N, int T = PassC<N>::threads>
__global__ void __launch_bounds__(T, PassC<N>::min_blocks(T)) k_solve_c(SolveArgs a) {
  using C = PassC<N>;
  constexpr int N1 = C::N1, N2 = C::N2, NH = C::NH, NP = C::NP, WP = N + 1;
  extern __shared__ unsigned char smraw_c[];
  __shared__ uint64_t bar;
  float2* P = reinterpret_cast<float2*>(tma_align(smraw_c));   // [y][NP]
  float2* W = P;                                                 // [pair][N + 1], once P is read
  float2* tw = P + N * NP;
  float4* Y = reinterpret_cast<float4*>(tw + N);                 // [pair][NH]: rows 2 m and 2 m + 1 at kx
  const int zo = blockIdx.x, d = blockIdx.y, pb = blockIdx.z;
  const float2* in = a.spec3 + (((size_t)pb * 3 + d) * a.t + zo) * N * NP;
  constexpr unsigned bytes = N * NP * (unsigned)sizeof(float2);
  static_assert(bytes % 16 == 0, "planes of whole 16-byte words");
  if (threadIdx.x == 0) {
    tma::mbar_init(&bar, 1);
    tma::fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    tma::mbar_arrive_expect_tx(&bar, bytes);
    tma::bulk_load(P, in, bytes, &bar);
  }
  // Prolongation of the coarse force onto this output plane: the coarse values
  // around the tile interior, interpolated in z.  Each thread fetches one while
  // the plane is on its way (meshes with more take the rest later).
  int ox, oy, oz;
  problem_origin(a, a.p0 + pb, ox, oy, oz);
  const int n = a.src_n, gz = oz + a.b + zo;
  const int nq = a.pc ? a.t / a.prc + 1 : 0, lr = a.pc ? __ffs(a.prc) - 1 : 0;
  const float inv_r = a.pc ? 1.0f / (float)a.prc : 0.f;
  const auto coarse_value = [&](int i) {
    const int qy = i / nq, qx = i - qy * nq;
    const int cz0 = gz >> lr, cz1 = cz0 + 1 == a.pnc ? 0 : cz0 + 1;
    const float wz = (float)(gz & (a.prc - 1)) * inv_r;
    int cy = ((oy + a.b) >> lr) + qy, cx = ((ox + a.b) >> lr) + qx;
    if (cy >= a.pnc) cy -= a.pnc;
    if (cx >= a.pnc) cx -= a.pnc;
    const size_t o = (size_t)cy * a.pnc + cx, plane = (size_t)a.pnc * a.pnc;
    const float* c = a.pc + (size_t)d * a.pnc * plane;
    return (1.0f - wz) * __ldg(c + cz0 * plane + o) + wz * __ldg(c + cz1 * plane + o);
  };
  float q_mine = 0.f;
  if (threadIdx.x < nq * nq) q_mine = coarse_value(threadIdx.x);
  for (int i = threadIdx.x; i < N; i += T) tw[i] = a.tw[i];
  if (!block_wait(&bar, a.status)) return;
  // inverse y transform, step 1: items (k1, column)
  for (int w = threadIdx.x; w < N1 * NH; w += T) {
    const int k1 = w / NH, c = w - k1 * NH;
    float2* base = P + N2 * k1 * NP + c;
    float2 v[N2];
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) v[k2] = base[k2 * NP];
    Dft<N2, 1>::run(v);
#pragma unroll
    for (int j2 = 1; j2 < N2; ++j2) v[j2] = cmul(v[j2], conjf2(tw[j2 * k1]));
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) base[j2 * NP] = v[j2];
  }
  __syncthreads();
  // step 2: items (two neighbouring j2, column) -> rows N2 j1 + j2 and the next
  const int m0 = a.b >> 1, np = C::pair_count(a.t, a.b);
  const float inv_np = 1.0f / (float)np;
  for (int w = threadIdx.x; w < (N2 / 2) * NH; w += T) {
    const int jp = w / NH, c = w - jp * NH;
    float2* base = P + 2 * jp * NP + c;
    float2 u[N1], v[N1];
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      u[k1] = base[N2 * k1 * NP];
      v[k1] = base[(N2 * k1 + 1) * NP];
    }
    Dft<N1, 1>::run(u);
    Dft<N1, 1>::run(v);
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) {
      if (C::in_place) {
        base[N2 * j1 * NP] = u[j1];
        base[(N2 * j1 + 1) * NP] = v[j1];
      } else {
        const int pair = (N2 / 2) * j1 + jp - m0;
        if ((unsigned)pair < (unsigned)np) Y[pair * NH + c] = make_float4(u[j1].x, u[j1].y, v[j1].x, v[j1].y);
      }
    }
  }
  __syncthreads();
  // inverse x transforms of the pairs, rows A and B packed as A + i B (A, B
  // their half spectra, extended by conjugate symmetry).  Step 1: items (k1,
  // pair), frequencies k = k1 + N1 k2.
  {
    for (int w0 = 0; w0 < np * N1; w0 += T) {   // (in place: one round)
      const int w = w0 + threadIdx.x;
      const bool live = w < np * N1;
      const int k1 = live ? quick_div(w, inv_np) : 0, j = live ? w - k1 * np : 0;
      float2 v[N2];
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) {
        const int k = k1 + N1 * k2;
        const bool low = k2 < N2 / 2 || (k2 == N2 / 2 && k1 == 0);   // k <= N / 2
        const int kk = low ? k : N - k;
        float2 A, B;
        if (C::in_place) {
          A = P[2 * (m0 + j) * NP + kk];
          B = P[(2 * (m0 + j) + 1) * NP + kk];
        } else {
          const float4 q = Y[j * NH + kk];
          A = make_float2(q.x, q.y);
          B = make_float2(q.z, q.w);
        }
        if (!low) {
          A = conjf2(A);
          B = conjf2(B);
        }
        v[k2] = make_float2(A.x - B.y, A.y + B.x);   // A + i B
      }
      Dft<N2, 1>::run(v);
#pragma unroll
      for (int j2 = 1; j2 < N2; ++j2) v[j2] = cmul(v[j2], conjf2(tw[j2 * k1]));
      if (C::in_place) __syncthreads();   // every row is read before W overwrites it
      if (live) {
        float2* base = W + j * WP + N2 * k1;
#pragma unroll
        for (int j2 = 0; j2 < N2; ++j2) base[j2] = v[j2];
      }
    }
  }
  __syncthreads();
  float* Q = reinterpret_cast<float*>(Y);   // [nq][nq]; Y is free by now
  if (threadIdx.x < nq * nq) Q[threadIdx.x] = q_mine;
  for (int i = threadIdx.x + T; i < nq * nq; i += T) Q[i] = coarse_value(i);
  // step 2: items (j2, pair), natural x = N2 j1 + j2
  for (int w = threadIdx.x; w < np * N2; w += T) {
    const int j2 = quick_div(w, inv_np), q = w - j2 * np;
    float2* base = W + q * WP + j2;
    float2 v[N1];
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) v[k1] = base[N2 * k1];
    Dft<N1, 1>::run(v);
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) base[N2 * j1] = v[j1];
  }
  __syncthreads();
  // Output cells are interior cells: origin + b + local lies inside [0, n) without wrap.
  float* dst = a.dst + (size_t)d * n * n * n + ((int64_t)gz * n + oy + a.b) * n + ox + a.b;
  float m = 0.f;
  if (a.pc && (a.b & 1) == 0) {
    // a warp takes 32 columns of the rows between two coarse rows, which share
    // their prolongation: lo at the lower coarse row, lo + f dlt between
    const int nxb = (a.t + 31) >> 5, tasks = (nq - 1) * nxb;
    const float inv_x = 1.0f / (float)nxb;
    for (int task = threadIdx.x >> 5; task < tasks; task += T / 32) {
      const int qy = quick_div(task, inv_x), xl = (task - qy * nxb) * 32 + (threadIdx.x & 31);
      if (xl >= a.t) continue;
      const float* q = Q + qy * nq + (xl >> lr);
      const float fx = (float)(xl & (a.prc - 1)) * inv_r;
      const float lo = fmaf(fx, q[1] - q[0], q[0]), dlt = fmaf(fx, q[nq + 1] - q[nq], q[nq]) - lo;
      const float2* w = W + ((qy << lr) >> 1) * WP + a.b + xl;
      float* o = dst + (int64_t)(qy << lr) * n + xl;
      float f = 0.f;
      for (int p = 0; p < a.prc; p += 2) {
        const float2 val = *w;
        m = fmaxf(m, fmaxf(fabsf(val.x), fabsf(val.y)));
        o[0] = val.x + fmaf(f, dlt, lo);
        o[n] = val.y + fmaf(f + inv_r, dlt, lo);
        f += 2.0f * inv_r;
        w += WP;
        o += 2 * (int64_t)n;
      }
    }
  } else {
    PM_ROWS(q, np) {
      const int y0 = 2 * (m0 + q) - a.b, y1 = y0 + 1;   // the pair's output rows, if inside [0, t)
      const bool in0 = y0 >= 0, in1 = y1 < a.t;
      const int q0 = y0 >> lr, q1 = y1 >> lr;
      const float f0 = (float)(y0 & (a.prc - 1)) * inv_r, f1 = (float)(y1 & (a.prc - 1)) * inv_r;
      PM_COLS(xl, a.t) {
        float2 w = W[q * WP + a.b + xl];
        if (in0) m = fmaxf(m, fabsf(w.x));
        if (in1) m = fmaxf(m, fabsf(w.y));
        if (a.pc) {
          const float fx = (float)(xl & (a.prc - 1)) * inv_r;
          const auto along_x = [&](int qy) {
            const float* q = Q + qy * nq + (xl >> lr);
            return fmaf(fx, q[1] - q[0], q[0]);
          };
          if (in0) {
            const float lo = along_x(q0), hi = along_x(q0 + 1);
            w.x += fmaf(f0, hi - lo, lo);
          }
          if (in1) {
            const float lo = along_x(q1), hi = along_x(q1 + 1);
            w.y += fmaf(f1, hi - lo, lo);
          }
        }
        if (in0) dst[(int64_t)y0 * n + xl] = w.x;
        if (in1) dst[(int64_t)y1 * n + xl] = w.y;
      }
    }
  }
  if (a.amax) {
    // warp maximum; an atomic only when it raises the running maximum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > __uint_as_float(*(volatile unsigned int*)a.amax))
      atomicMax(a.amax, __float_as_uint(m));
  }
}

// Tensor maps (encoded on the host; cuTensorMapEncodeTiled reached through
// the runtime's driver entry point, so the library links no driver library).
static PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 3-D float32 tensor: dims d0 (innermost) .. d2, byte strides s1, s2 of dims 1 and 2, box b0 x b1 x b2.
static bool map_3d(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t s1, uint64_t s2,
                   uint32_t b0, uint32_t b1, uint32_t b2) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_tiled();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) || (s1 & 15) || (s2 & 15) || (b0 * 4) % 16 || b0 > 256 ||
      b1 > 256 || b2 > 256)
    return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {s1, s2};
  cuuint32_t box[3] = {b0, b1, b2};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- Large periodic meshes (N > 128: the coarse mesh of the largest
// two-level runs).  A z plane of N^2 complex values no longer fits in shared
// memory, so passes A and C are each split into a row pass along x and a
// column pass along y, in place in the spectrum buffers:
//   AX  per (z, R rows): real-to-complex along x, two rows packed as one
//       complex row -> spec[z][y][kx] (natural order);
//   AY  per (z, KC columns): FFT along y -> spec[z][ky slot][kx], the layout
//       pass B reads;
//   B   the pass above, KC columns per block;
//   CY  per (component, z, KC columns): inverse FFT along y -> natural y;
//   CX  per (component, z, R rows): complex-to-real along x -> dst, with the
//       running max |a| when asked.
// The window is the whole mesh (one problem, origin 0).
template <int N> struct Large {
  static constexpr int NH = N / 2 + 1;
  static constexpr int R = 32;      // rows per block of the x passes
  static constexpr int KC = 16;     // columns per block of the y passes
  static constexpr int threads = 256;
  static constexpr int nchunk = (NH + KC - 1) / KC;
  static constexpr size_t smem_ax = sizeof(float2) * (N + (size_t)(R / 2) * N);
  static constexpr size_t smem_y = sizeof(float2) * (N + (size_t)N * KC);
  static constexpr size_t smem_cx = sizeof(float2) * (N + (size_t)R * NH + (size_t)(R / 2) * N);
};

template <int N, bool FIXED>
__global__ void __launch_bounds__(Large<N>::threads) k_large_ax(SolveArgs a) {
  constexpr int NH = Large<N>::NH, R = Large<N>::R;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* W = sm + N;   // R/2 packed rows of N
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = a.tw[i];
  const int y0 = blockIdx.x * R, z = blockIdx.y;
  PM_ROWS(r, R) {
    const int64_t rowbase = ((int64_t)z * N + y0 + r) * N;
    float* w = reinterpret_cast<float*>(W + (r >> 1) * N) + (r & 1);
    if (FIXED) {
      PM_COLS(x, N) w[2 * x] = src_value<FIXED>(a.src, rowbase + x);
    } else {
      const float* srow = static_cast<const float*>(a.src) + rowbase;
      PM_COLS(x, N) async_copy4(w + 2 * x, srow + x);
    }
  }
  if (!FIXED) async_wait();
  __syncthreads();
  fft_fwd<N, R / 2, N, 1>(W, tw);
  // unpack the two real rows of each packed row (as in pass A), natural kx order
  float2* out = a.spec + ((size_t)z * N + y0) * NH;
  PM_ROWS(j, R / 2) {
    const float2* Wj = W + j * N;
    float2* o0 = out + (size_t)(2 * j) * NH;
    float2* o1 = o0 + NH;
    PM_COLS(k, NH) {
      const float2 zk = Wj[slot_of<N>(k)];
      const float2 zm = Wj[slot_of<N>(k == 0 ? 0 : N - k)];
      o0[k] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
      o1[k] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
    }
  }
}

// FFT along y of KC columns of plane (blockIdx.z N + blockIdx.y) of buf
// [plane][N][NH], in place: DIR -1 natural -> slot order, +1 slot -> natural.
template <int N, int DIR>
__global__ void __launch_bounds__(Large<N>::threads) k_large_y(float2* buf, const float2* twg) {
  constexpr int NH = Large<N>::NH, KC = Large<N>::KC;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* F = sm + N;   // [y][KC]
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = twg[i];
  const int kx0 = blockIdx.x * KC;
  const int ncol = (NH - kx0) < KC ? (NH - kx0) : KC;
  float2* pl = buf + ((size_t)blockIdx.z * N + blockIdx.y) * N * NH + kx0;
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
    const int y = i / KC, c = i - y * KC;
    if (c < ncol) async_copy8(F + i, pl + (size_t)y * NH + c);
    else F[i] = make_float2(0.f, 0.f);
  }
  async_wait();
  __syncthreads();
  if (DIR < 0) fft_fwd<N, KC, 1, KC>(F, tw);
  else fft_inv<N, KC, 1, KC>(F, tw);
  for (int i = threadIdx.x; i < N * KC; i += blockDim.x) {
    const int y = i / KC, c = i - y * KC;
    if (c < ncol) pl[(size_t)y * NH + c] = F[i];
  }
}

template <int N>
__global__ void __launch_bounds__(Large<N>::threads) k_large_cx(SolveArgs a) {
  constexpr int NH = Large<N>::NH, R = Large<N>::R;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* P = sm + N;          // [R][NH], natural order
  float2* W = P + R * NH;      // R/2 packed rows of N
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = a.tw[i];
  const int y0 = blockIdx.x * R, z = blockIdx.y, d = blockIdx.z;
  const float2* in = a.spec3 + (((size_t)d * N + z) * N + y0) * NH;
  for (int i = threadIdx.x; i < R * NH; i += blockDim.x) async_copy8(P + i, in + i);
  async_wait();
  __syncthreads();
  PM_ROWS(j, R / 2) {
    const float2* Pa = P + (2 * j) * NH;
    const float2* Pb = Pa + NH;
    float2* Wj = W + j * N;
    PM_COLS(k, N) {
      float2 A, B;
      if (k <= N / 2) {
        A = Pa[k];
        B = Pb[k];
      } else {
        A = conjf2(Pa[N - k]);
        B = conjf2(Pb[N - k]);
      }
      Wj[slot_of<N>(k)] = make_float2(A.x - B.y, A.y + B.x);   // A + i B
    }
  }
  __syncthreads();
  fft_inv_rows<N, N>(W, R / 2, tw);
  float* dst = a.dst + (size_t)d * N * N * N + ((size_t)z * N + y0) * N;
  float m = 0.f;
  PM_ROWS(yl, R) {
    const float* w = reinterpret_cast<const float*>(W + (yl >> 1) * N) + (yl & 1);
    float* drow = dst + (size_t)yl * N;
    PM_COLS(x, N) {
      const float val = w[2 * x];
      m = fmaxf(m, fabsf(val));
      drow[x] = val;
    }
  }
  if (a.amax) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > __uint_as_float(*(volatile unsigned int*)a.amax))
      atomicMax(a.amax, __float_as_uint(m));
  }
}

template <int N>
static cudaError_t solve_large_n(const SolvePlan& p, const void* src, bool fixed, float* dst, cudaStream_t st,
                                 Timer* tm, unsigned int* amax) {
  using L = Large<N>;
  if (p.nts != 1 || p.b != 0 || p.t != N || p.src_n != N) return cudaErrorInvalidValue;
  static bool attr_done = false;
  if (!attr_done) {
    cudaFuncSetAttribute(k_large_ax<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_ax);
    cudaFuncSetAttribute(k_large_ax<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_ax);
    cudaFuncSetAttribute(k_large_y<N, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_y);
    cudaFuncSetAttribute(k_large_y<N, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_y);
    cudaFuncSetAttribute(k_large_b<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassB<N>::smem);
    cudaFuncSetAttribute(k_large_cx<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::smem_cx);
    attr_done = true;
  }
  SolveArgs a{src, N, 1, N, 0, 0, p.spec, p.spec3, p.kern, p.kern_quads, p.tw, dst, 0, amax, nullptr, 0, 1, p.status};
  {
    TimedScope ts(tm, "fft_a_mesh", st);
    if (fixed) k_large_ax<N, true><<<dim3(N / L::R, N), L::threads, L::smem_ax, st>>>(a);
    else k_large_ax<N, false><<<dim3(N / L::R, N), L::threads, L::smem_ax, st>>>(a);
    k_large_y<N, -1><<<dim3(L::nchunk, N, 1), L::threads, L::smem_y, st>>>(p.spec, p.tw);
  }
  {
    TimedScope ts(tm, "fft_b_mesh", st);
    k_large_b<N><<<dim3(N, PassB<N>::nchunk, 1), PassB<N>::threads, PassB<N>::smem, st>>>(a);
  }
  {
    TimedScope ts(tm, "fft_c_mesh", st);
    k_large_y<N, 1><<<dim3(L::nchunk, N, 3), L::threads, L::smem_y, st>>>(p.spec3, p.tw);
    k_large_cx<N><<<dim3(N / L::R, N, 3), L::threads, L::smem_cx, st>>>(a);
  }
  note_launches(5);
  return cudaGetLastError();
}

template <int N>
__global__ void k_tile_window(const float* src, int src_n, int nts, int t, int b, int64_t tile, float* out) {
  int px = (int)(tile % nts), py = (int)((tile / nts) % nts), pz = (int)(tile / ((int64_t)nts * nts));
  int ox = px * t - b, oy = py * t - b, oz = pz * t - b;
  int64_t total = (int64_t)N * N * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    int x = (int)(i % N), y = (int)((i / N) % N), z = (int)(i / ((int64_t)N * N));
    int gx = pmod(ox + x, src_n), gy = pmod(oy + y, src_n), gz = pmod(oz + z, src_n);
    out[i] = src[((int64_t)gz * src_n + gy) * src_n + gx];
  }
}

// Kernel table [3][z slot][y slot][NH] -> pass B's order [y slot][chunk][component]
// [quad][k1][column] of float4: quad q of item (k1, column) holds kz slots
// N2 k1 + 4 q .. + 3 (zero past the last column), so a warp's loads are
// consecutive 16-byte words.
template <int N>
__global__ void k_kernel_quads(const float* kern, float* out) {
  using B = PassBR<N>;
  constexpr int NH = N / 2 + 1, N1 = Factor<N>::N1, N2 = Factor<N>::N2, KT = B::KT;
  static_assert(N2 % 4 == 0, "whole quads");
  constexpr int total = N * B::nchunk * 3 * N2 * KT * N1;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    int r = i;
    const int e = r % 4;
    r /= 4;
    const int c = r % KT;
    r /= KT;
    const int k1 = r % N1;
    r /= N1;
    const int q = r % (N2 / 4);
    r /= N2 / 4;
    const int d = r % 3;
    r /= 3;
    const int ch = r % B::nchunk, ys = r / B::nchunk;
    const int kx = ch * KT + c, zs = N2 * k1 + 4 * q + e;
    out[i] = kx < NH ? kern[(((size_t)d * N + zs) * N + ys) * NH + kx] : 0.f;
  }
}
template <int N>
static size_t quads_n(const float* kern, float* out, cudaStream_t st) {
  using B = PassBR<N>;
  if (out) {
    k_kernel_quads<N><<<152 * 4, 256, 0, st>>>(kern, out);
    note_launches(1);
  }
  return (size_t)N * B::nchunk * 3 * Factor<N>::N2 * B::KT * Factor<N>::N1 * sizeof(float);
}
size_t kernel_quads(int N, const float* kern, float* out, cudaStream_t st) {
  switch (N) {
    case 16: return quads_n<16>(kern, out, st);
    case 32: return quads_n<32>(kern, out, st);
    case 48: return quads_n<48>(kern, out, st);
    case 64: return quads_n<64>(kern, out, st);
    case 96: return quads_n<96>(kern, out, st);
    case 128: return quads_n<128>(kern, out, st);
    default: return 0;
  }
}

template <int N>
static cudaError_t solve_n(const SolvePlan& p, const void* src, bool fixed, float* dst, cudaStream_t st, Timer* tm,
                           unsigned int* amax, const Prolong* pro) {
  using C = SolveCfg<N>;
  static bool attr_done = false;
  if (!attr_done) {
    cudaFuncSetAttribute(k_solve_a<N, SRC_FLOAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassA<N>::smem);
    cudaFuncSetAttribute(k_solve_a<N, SRC_FIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassA<N>::smem);
    cudaFuncSetAttribute(k_solve_b<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassBR<N>::smem);
    cudaFuncSetAttribute(k_solve_c<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassC<N>::smem_max());
    if constexpr (N == 96) {
      cudaFuncSetAttribute(k_solve_a<N, SRC_BOXES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassA<N>::smem);
      cudaFuncSetAttribute(k_solve_c<N, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassC<N>::smem_max());
    }
    attr_done = true;
  }
  // 96^3 passes staged by TMA: pass A wants window origins and the source
  // mesh on 16-cell boundaries (float source); pass B reads boxes of the spectrum.
  bool tma_a = false;
  CUtensorMap src_map{}, spec_map{};
  if constexpr (N == 96) {
    const int n = p.src_n;
    tma_a = !fixed && n % kBox == 0 && p.t % kBox == 0 && p.b % kBox == 0 &&
            map_3d(&src_map, src, n, n, n, (uint64_t)n * 4, (uint64_t)n * n * 4, kBox, kBox, 1);
    if (!map_3d(&spec_map, p.spec, 2 * C::NH, N, (uint64_t)p.batch * N, (uint64_t)C::NP * 8, (uint64_t)N * C::NP * 8,
                2 * PassBR<N>::KT, 1, N))
      return cudaErrorInvalidValue;
  }
  const int nprob = p.nts * p.nts * p.nts;
  for (int p0 = 0; p0 < nprob; p0 += p.batch) {
    int nb = (nprob - p0 < p.batch) ? (nprob - p0) : p.batch;
    SolveArgs a{src, p.src_n, p.nts, p.t, p.b, p0, p.spec, p.spec3, p.kern, p.kern_quads, p.tw, dst, 0, amax,
                pro ? pro->coarse : nullptr, pro ? pro->nc : 0, pro ? pro->rc : 1, p.status};
    {
      TimedScope ts(tm, N == p.src_n && p.b == 0 ? "fft_a_mesh" : "fft_a_tiles", st);
      using A = PassA<N>;
      const auto ka = fixed ? k_solve_a<N, SRC_FIXED> : k_solve_a<N, SRC_FLOAT>;
      if constexpr (N == 96) {
        if (tma_a) k_solve_a<N, SRC_BOXES><<<dim3(N, nb), A::threads, A::smem, st>>>(a, src_map);
      }
      if (!tma_a) ka<<<dim3(N, nb), A::threads, A::smem, st>>>(a, src_map);
    }
    {
      TimedScope ts(tm, N == p.src_n && p.b == 0 ? "fft_b_mesh" : "fft_b_tiles", st);
      using B = PassBR<N>;
      k_solve_b<N><<<dim3(N, B::nchunk, nb), B::threads, B::smem, st>>>(a, spec_map);
    }
    if (pro && pro->ready && p0 == 0) {
      cudaError_t e = cudaStreamWaitEvent(st, pro->ready, 0);   // the coarse force must be complete
      if (e != cudaSuccess) return e;
    }
    {
      TimedScope ts(tm, N == p.src_n && p.b == 0 ? "fft_c_mesh" : "fft_c_tiles", st);
      const size_t smem = PassC<N>::smem(p.t, p.b, a.prc, a.pc != nullptr);
      if constexpr (N == 96) {
        if (PassC<N>::narrow(p.t, p.b)) k_solve_c<N, 256><<<dim3(p.t, 3, nb), 256, smem, st>>>(a);
        else k_solve_c<N><<<dim3(p.t, 3, nb), PassC<N>::threads, smem, st>>>(a);
      } else {
        k_solve_c<N><<<dim3(p.t, 3, nb), PassC<N>::threads, smem, st>>>(a);
      }
    }
    note_launches(3);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t solve_launch(const SolvePlan& p, const void* src, bool fixed, float* dst, cudaStream_t st, Timer* tm,
                         unsigned int* amax, const Prolong* pro) {
  if (pro && (p.t % pro->rc || (pro->rc & (pro->rc - 1)))) return cudaErrorInvalidValue;
  switch (p.N) {
    case 16: return solve_n<16>(p, src, fixed, dst, st, tm, amax, pro);
    case 32: return solve_n<32>(p, src, fixed, dst, st, tm, amax, pro);
    case 48: return solve_n<48>(p, src, fixed, dst, st, tm, amax, pro);
    case 64: return solve_n<64>(p, src, fixed, dst, st, tm, amax, pro);
    case 96: return solve_n<96>(p, src, fixed, dst, st, tm, amax, pro);
    case 128: return solve_n<128>(p, src, fixed, dst, st, tm, amax, pro);
    case 192: return pro ? cudaErrorInvalidValue : solve_large_n<192>(p, src, fixed, dst, st, tm, amax);
    case 256: return pro ? cudaErrorInvalidValue : solve_large_n<256>(p, src, fixed, dst, st, tm, amax);
    case 384: return pro ? cudaErrorInvalidValue : solve_large_n<384>(p, src, fixed, dst, st, tm, amax);
    default: return cudaErrorInvalidValue;
  }
}

template <int N>
static cudaError_t solve_adjoint_n(const SolvePlan& p, const float* lam_acc, bool interleaved, float* lam_rho,
                                   float2* spec3comp, cudaStream_t st) {
  const auto ka = interleaved ? k_solve_a<N, SRC_INTERLEAVED> : k_solve_a<N, SRC_FLOAT>;
  cudaFuncSetAttribute(ka, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassA<N>::smem);
  cudaFuncSetAttribute(k_solve_b_adj<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float2) * (N + 2 * (size_t)N * PassB<N>::KC)));
  cudaFuncSetAttribute(k_solve_c<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PassC<N>::smem_max());
  SolveArgs a{lam_acc, p.src_n, 1, N, 0, 0, spec3comp, p.spec3, p.kern, p.kern_quads, p.tw, lam_rho, 1, nullptr, nullptr, 0, 1,
              p.status};
  ka<<<dim3(N, 3), PassA<N>::threads, PassA<N>::smem, st>>>(a, CUtensorMap{});
  a.comp_mode = 0;
  k_solve_b_adj<N><<<dim3(N, 2, 1), PassB<N>::threads, sizeof(float2) * (N + 2 * (size_t)N * PassB<N>::KC), st>>>(a);
  k_solve_c<N><<<dim3(N, 1, 1), PassC<N>::threads, PassC<N>::smem(N, 0, 1, false), st>>>(a);
  note_launches(3);
  return cudaGetLastError();
}

cudaError_t solve_adjoint_launch(const SolvePlan& p, const float* lam_acc, bool interleaved, float* lam_rho,
                                 float2* spec3comp, cudaStream_t st) {
  if (p.nts != 1 || p.b != 0 || p.t != p.N) return cudaErrorInvalidValue;
  switch (p.N) {
    case 16: return solve_adjoint_n<16>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    case 32: return solve_adjoint_n<32>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    case 48: return solve_adjoint_n<48>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    case 64: return solve_adjoint_n<64>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    case 96: return solve_adjoint_n<96>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    case 128: return solve_adjoint_n<128>(p, lam_acc, interleaved, lam_rho, spec3comp, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t tile_window_launch(const SolvePlan& p, const float* src, int64_t tile, float* out, cudaStream_t st) {
  int blocks = 256;
  switch (p.N) {
    case 16: k_tile_window<16><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    case 32: k_tile_window<32><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    case 48: k_tile_window<48><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    case 64: k_tile_window<64><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    case 96: k_tile_window<96><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    case 128: k_tile_window<128><<<blocks, 256, 0, st>>>(src, p.src_n, p.nts, p.t, p.b, tile, out); break;
    default: return cudaErrorInvalidValue;
  }
  note_launches(1);
  return cudaGetLastError();
}

// Coarse CIC density from the fine one (exact for CIC: the coarse tent is the
// fine-node interpolation of itself): rho_c(C) = sum_k w(kx) w(ky) w(kz)
// rho_f(rc C + k), w(k) = 1 - |k| / rc, k = -(rc-1) .. rc-1, periodic.  One
// block per coarse (y, z) row: threads sum the (2 rc - 1)^2 fine rows with
// their y, z weights along x into shared memory, then the x weights.
template <int RC>   // RC > 0: compile-time ratio (loops unrolled); 0: runtime ratio rc
__global__ void __launch_bounds__(256, 1) k_restrict(const float* rho_f, int nf, int rc_rt, float* rho_c) {
  extern __shared__ float acc[];   // [nf]
  const int rc = RC > 0 ? RC : rc_rt;
  const int nc = nf / rc;
  const int cy = blockIdx.x % nc, cz = blockIdx.x / nc;
  const float inv = 1.0f / (float)rc;
  int zrow[2 * (RC > 0 ? RC : 16) - 1], yrow[2 * (RC > 0 ? RC : 16) - 1];
#pragma unroll
  for (int k = 1 - rc; k < rc; ++k) {
    int z = rc * cz + k, y = rc * cy + k;
    z += z < 0 ? nf : (z >= nf ? -nf : 0);
    y += y < 0 ? nf : (y >= nf ? -nf : 0);
    zrow[k + rc - 1] = z;
    yrow[k + rc - 1] = y;
  }
  for (int x = threadIdx.x; x < nf; x += blockDim.x) {
    float s = 0.f;
#pragma unroll
    for (int kz = 1 - rc; kz < rc; ++kz) {
      const float wz = 1.0f - (float)(kz < 0 ? -kz : kz) * inv;
      const float* zp = rho_f + (size_t)zrow[kz + rc - 1] * nf * nf + x;
#pragma unroll
      for (int ky = 1 - rc; ky < rc; ++ky) {
        const float wy = 1.0f - (float)(ky < 0 ? -ky : ky) * inv;
        s = fmaf(wz * wy, __ldg(zp + (size_t)yrow[ky + rc - 1] * nf), s);
      }
    }
    acc[x] = s;
  }
  __syncthreads();
  for (int cx = threadIdx.x; cx < nc; cx += blockDim.x) {
    float t = 0.f;
#pragma unroll
    for (int kx = 1 - rc; kx < rc; ++kx) {
      int x = rc * cx + kx;
      x += x < 0 ? nf : (x >= nf ? -nf : 0);
      t = fmaf(1.0f - (float)(kx < 0 ? -kx : kx) * inv, acc[x], t);
    }
    rho_c[((size_t)cz * nc + cy) * nc + cx] = t;
  }
}

cudaError_t launch_restrict(const float* rho_f, int nf, int rc, float* rho_c, cudaStream_t st) {
  if (rc < 1 || rc > 16 || nf % rc) return cudaErrorInvalidValue;
  const int nc = nf / rc;
  if (rc == 4) k_restrict<4><<<nc * nc, 256, (size_t)nf * sizeof(float), st>>>(rho_f, nf, rc, rho_c);
  else k_restrict<0><<<nc * nc, 256, (size_t)nf * sizeof(float), st>>>(rho_f, nf, rc, rho_c);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pm
