// Staged FP32 kernels of every eighth general line length, from number 1 of the list on
// (dgpe_stages.cuh); eight translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y1(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<1>::y(dir, a, ga, members, st);
}
bool stage_x1(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<1>::x(a, ga, members, st);
}
bool stage_z1(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<1>::z(which, a, ga, members, st);
}
cudaError_t stage_init1(int nx, int ny, int nz) { return StageLaunch<1>::init(nx, ny, nz); }
}  // namespace dgpe
