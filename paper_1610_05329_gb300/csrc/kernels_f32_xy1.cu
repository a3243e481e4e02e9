// FP32 y and x transforms of every fourth general line length, from number 1 of the list on
// (dgpe_stages.cuh); four translation units, so that they build in parallel.
#include "dgpe_stages.cuh"

namespace dgpe {
bool stage_y1(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<1>::y(dir, a, ga, members, st);
}
bool stage_x1(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
  return StageLaunch<1>::x(a, ga, members, st);
}
cudaError_t stage_init1(int nx, int ny) { return StageLaunch<1>::init(nx, ny); }
}  // namespace dgpe
