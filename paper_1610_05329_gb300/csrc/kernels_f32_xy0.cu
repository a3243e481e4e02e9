// Staged FP32 kernels of every eighth general line length, from number 0 of the list on
// (dgpe_stages.cuh); eight translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y0(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<0>::y(dir, a, ga, members, st);
}
bool stage_x0(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<0>::x(a, ga, members, st);
}
bool stage_z0(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<0>::z(which, a, ga, members, st);
}
cudaError_t stage_init0(int nx, int ny, int nz) { return StageLaunch<0>::init(nx, ny, nz); }
cudaError_t stage_tables(void *tw, int n, cudaStream_t st) {
  if (st_index(n) < 0) return cudaSuccess;
  k_stage_twiddles<<<(2 * n + 127) / 128, 128, 0, st>>>(static_cast<cplx<float> *>(tw), n, st_radix(n, 0), st_radix(n, 1),
                                                       st_radix(n, 2));
  return cudaGetLastError();
}
bool stage_own_z(int n) { return st_index(n) >= 0 && st_xy(n) && n != 64 && n != 96 && n != 384; }
}  // namespace dgpe
