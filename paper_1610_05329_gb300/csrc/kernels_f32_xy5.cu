// Staged FP32 kernels of every eighth general line length, from number 5 of the list on
// (dgpe_stages.cuh); eight translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y5(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<5>::y(dir, a, ga, members, st);
}
bool stage_x5(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<5>::x(a, ga, members, st);
}
bool stage_z5(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<5>::z(which, a, ga, members, st);
}
cudaError_t stage_init5(int nx, int ny, int nz) { return StageLaunch<5>::init(nx, ny, nz); }
}  // namespace dgpe
