// Staged FP32 kernels of every eighth general line length, from number 2 of the list on
// (dgpe_stages.cuh); eight translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y2(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<2>::y(dir, a, ga, members, st);
}
bool stage_x2(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<2>::x(a, ga, members, st);
}
bool stage_z2(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<2>::z(which, a, ga, members, st);
}
cudaError_t stage_init2(int nx, int ny, int nz) { return StageLaunch<2>::init(nx, ny, nz); }
}  // namespace dgpe
