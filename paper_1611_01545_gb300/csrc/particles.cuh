// Device-side views and launchers of the particle kernels (particles.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pm_common.cuh"

namespace pm {

// Geometry as the particle kernels see it (plain values, passed by value).
struct Geo {
  int nf, rc, nc, rcmp, ncmp;
  int64_t ncell;
  bool two;
};

// Cell-block decomposition of the compression mesh for the fused passes.
struct Blk {
  int RX, RY, RZ;     // cells per block along x, y, z
  int nbx, nby, nbz;  // blocks along x, y, z
  int D;              // half-width (cells) of the new-cell histogram window; -1: no window
  int wx, wy, wz;     // that window's extents (set by the recompress launchers; 0: no window)
  int brick;          // blocks are handed out in bricks of brick x brick (y, z) block rows (1: row order)
  int* work;          // persistent launch: device counter of cell blocks taken (zeroed before the launch); null: one CTA per block
};

struct PCodes {
  const uint32_t* pos;
  const void* vel;
  const float* vmax;
  int64_t n;
  bool vel16;
};

struct PCodesOut {
  uint32_t* pos;
  void* vel;
  float* vmax;
  bool vel16;
};

// Scans (scan.cu).  state: scan_state_bytes(ncell) per species, zeroed once before
// its first scan; every scan on it has the same ncell, and they follow one another.
size_t scan_state_bytes(int64_t ncell);
// Arrays that a step's first scan clears on the way: the new-cell counts of
// both species, window and far movers, and `small_words` 32-bit words (null: nothing).
struct ScanClear {
  uint32_t* counts[2];
  uint32_t* far[2];
  uint32_t* small;
  int small_words;
  void* mesh;            // 16-byte aligned
  int64_t mesh_words;    // 16-byte words
};
cudaError_t scan_codes(const pm_codes_t& in, int64_t ncell, int64_t* off, void* state, int* status, cudaStream_t st);
// vmax_bits (float bits): copied to out.vmax when set.
cudaError_t scan_counts(const uint32_t* counts, int64_t ncell, int64_t expect, int64_t* off, pm_codes_t& out,
                        const uint32_t* vmax_bits, void* state, int* status, cudaStream_t st);
// Both species in one launch (2 scan_state_bytes of state).
cudaError_t scan_codes2(const pm_codes_t in[2], int64_t ncell, int64_t* off0, int64_t* off1, void* state, int* status,
                        const ScanClear* clear, cudaStream_t st);
// (counts: far movers apart)
cudaError_t scan_counts2(const uint32_t* const counts[2], const uint32_t* const far[2], int64_t ncell, const int64_t expect[2],
                         int64_t* off0, int64_t* off1, pm_codes_t out[2], const uint32_t* vmax_bits, void* state,
                         int* status, cudaStream_t st);

cudaError_t launch_decompress(const PCodes& in, const int64_t* off, const Geo& g, float* x, float* v, cudaStream_t st);
cudaError_t launch_deposit(const float* x, int64_t n, float m, const Geo& g, float* rho_c, float* rho_f,
                           cudaStream_t st);
cudaError_t launch_deposit_weights(const float* x, int64_t n, const float* w, int nw, const Geo& g, float* out,
                                  cudaStream_t st);
cudaError_t launch_deposit_fixed(const float* x, int64_t n, long long M, const Geo& g, long long* rho_c,
                                 long long* rho_f, cudaStream_t st);
// The acceleration mesh [3][n3] with its components next to each other.
cudaError_t launch_interleave(const float* acc, int64_t n3, float4* out, cudaStream_t st);
// acc4: acc_f interleaved, or null.
cudaError_t launch_interpolate(const float* x, int64_t n, const Geo& g, const float* acc_c, const float* acc_f,
                               const float4* acc4, float* a, cudaStream_t st);
cudaError_t launch_kick_drift(float* x, float* v, int64_t n, const Geo& g, const float* acc_c, const float* acc_f,
                              const float4* acc4, float ck, float cd, cudaStream_t st);
cudaError_t launch_compress(const float* x, const float* v, int64_t n, const Geo& g, uint32_t* counts,
                            uint32_t* vmax_bits, const float* vmax_in, int64_t* off, pm_codes_t& out, bool vel16,
                            void* scan_state, int* status, cudaStream_t st);
size_t deposit_codes_smem(const Geo& g, const Blk& bk, bool fixed);
// Recompress passes (kick.cu).
size_t kick_count_smem(const Geo& g, const Blk& bk);
size_t kick_scatter_smem(const Geo& g, const Blk& bk);
int window_cells(const Geo& g, const Blk& bk);
// New-cell tables between the count pass and the scatter, per species: window
// movers and far movers per cell, and the start of each block's share.
struct RecompressTables {
  uint32_t* counts0;
  uint32_t* counts1;
  uint32_t* far0;
  uint32_t* far1;
  uint32_t* start;   // null: no window (half-width -1)
  int kb;            // rank bits of a key (set by the launchers)
};
size_t table_bytes(const Geo& g, const Blk& bk);
constexpr int kKickRowCells = 32;
Blk kick_blocks(const Geo& g, Blk bk, int64_t particles);
// Brick edge (block rows) of the block order for a block grid (1: row order).
int block_brick(const Blk& bk);
cudaError_t launch_deposit_codes(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1,
                                 const Geo& g, const Blk& bk, float m0, float m1, long long M0, long long M1,
                                 void* rho_c, void* rho_f, bool fixed, cudaStream_t st);
cudaError_t launch_kick_count(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1,
                              const Geo& g, const Blk& bk, const float* acc_c, const float* acc_f, float ck, float cd,
                              const RecompressTables& t, uint32_t* vmax_bits, uint32_t* tkey, uint4* tpv,
                              const float* vq0, const float* vq1, const float4* app, bool coarse, cudaStream_t st);
cudaError_t launch_kick_scatter(int64_t n0, int64_t n1, const int64_t* off0, const int64_t* off1, const Geo& g,
                                const Blk& bk, const RecompressTables& t, const int64_t* newoff0,
                                const int64_t* newoff1, const PCodesOut& o0, const PCodesOut& o1, const uint32_t* tkey,
                                const uint4* tpv, bool coded, int* status, cudaStream_t st);
// v_max' bound of both species from v_max and the maxima amax[3] (coarse mesh,
// fine mesh, PP accelerations; float bits).
// PP acceleration (Eq. 4) of every particle of both species into acc[t] (stream index t,
// species 0 first; float4, w = 0); max |a_d| into *amax when set.  pp.cu.
size_t pp_smem(const Geo& g);
cudaError_t launch_pp(const PCodes& c0, const PCodes& c1, const int64_t* off0, const int64_t* off1, const Geo& g,
                      float m0, float m1, float G, float r_soft, float4* acc, uint32_t* amax, cudaStream_t st);
// Packed codes (pack.cu): padded position / velocity words <-> record bytes.
cudaError_t launch_pack(const uint32_t* pos, const void* vel, bool vel16, int64_t n, uint8_t* ppos, uint8_t* pvel,
                        cudaStream_t st);
cudaError_t launch_unpack(const uint8_t* ppos, const uint8_t* pvel, bool vel16, int64_t n, uint32_t* pos, void* vel,
                          cudaStream_t st);
cudaError_t launch_vmax_bound(const float* vin0, const float* vin1, const uint32_t* amax, float ck, float* vout0,
                              float* vout1, cudaStream_t st);
cudaError_t launch_adj_deposit(const float* x, int64_t n, float m, int nf, const float* lam_rho, float* lam_x,
                               cudaStream_t st);
// lam_A is [3][n^3], or float4 [n^3] (x, y, z, unused) when interleaved (one vector
// reduction per corner instead of three).
// acc4: acc interleaved, or null.
cudaError_t launch_adj_interp(const float* x, int64_t n, int nf, const float* acc, const float4* acc4, float ck, float cd, float* lam_x,
                              float* lam_v, float* lam_A, bool interleaved, cudaStream_t st);

}  // namespace pm
