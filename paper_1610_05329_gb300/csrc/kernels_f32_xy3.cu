// FP32 y and x transforms of every fourth general line length, from number 3 of the list on
// (dgpe_stages.cuh); four translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y3(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<3>::y(dir, a, ga, members, st);
}
bool stage_x3(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<3>::x(a, ga, members, st);
}
cudaError_t stage_init3(int nx, int ny) { return StageLaunch<3>::init(nx, ny); }
}  // namespace dgpe
