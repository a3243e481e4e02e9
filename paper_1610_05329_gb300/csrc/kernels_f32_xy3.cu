// Staged FP32 kernels of every eighth general line length, from number 3 of the list on
// (dgpe_stages.cuh); eight translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y3(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<3>::y(dir, a, ga, members, st);
}
bool stage_x3(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<3>::x(a, ga, members, st);
}
bool stage_z3(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<3>::z(which, a, ga, members, st);
}
cudaError_t stage_init3(int nx, int ny, int nz) { return StageLaunch<3>::init(nx, ny, nz); }
}  // namespace dgpe
