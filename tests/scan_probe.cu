// Scans of count bytes on one state, for tests/test_gpu_scan_state.py: launched as
// the library does, or with the blocks of two launches at once, which is what two
// scans that overlap on one state come to.
#include <cuda_runtime.h>

#include "scan.cu"

namespace pm {
void note_launches(int) {}
}  // namespace pm

// Device memory: cnt [ncell], off [ncell + 1], state (scan_probe_state(ncell) bytes,
// zeroed), status.  expect: the particles that the counts add up to.  launches: blocks
// of this many scans in one launch; skip: tiles that count as drawn but never run;
// limit: cycles after which a wait is given up (0: the library's own limit).
extern "C" long long scan_probe_state(long long ncell) { return (long long)pm::scan_state_bytes(ncell); }
extern "C" int scan_probe(const void* cnt, const void* vmax, const void* n_esc, const void* esc, long long ncell,
                          long long expect, void* off, void* state, void* status, int launches, int skip, long long limit) {
  using namespace pm;
  Pair<CodesCount> get{};
  Pair<PutOffsets> put{};
  Pair<FinishArgs> fin{};
  get.v[0] = CodesCount{(const uint8_t*)cnt, (const uint32_t*)esc, (const uint32_t*)n_esc, 1, (const float*)vmax, (int*)status};
  put.v[0] = PutOffsets{(int64_t*)off, nullptr, nullptr};
  fin.v[0] = FinishArgs{expect, (int64_t*)off, nullptr, 0, nullptr, nullptr, nullptr, 0, nullptr, 0};
  const int tiles = scan_tiles(ncell);
  if (skip > 0) {
    ScanState s;
    if (cudaMemcpy(&s, state, sizeof(s), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    s.ticket += skip;
    if (cudaMemcpy(state, &s, sizeof(s), cudaMemcpyHostToDevice) != cudaSuccess) return -1;
  }
  k_scan<<<dim3(launches * tiles - skip, 1), SCAN_THREADS>>>(get, put, fin, ncell, tiles, (unsigned char*)state,
                                                             scan_state_bytes(ncell), limit ? limit : kWaitLimit,
                                                             (int*)status);
  const cudaError_t e = cudaGetLastError();
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
