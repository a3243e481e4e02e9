// Fixed-point transforms of the FP64 precision: every eighth line length, from number 1 of the
// list on (dgpe_fixed.cuh); eight translation units, so that they build in parallel.
#include "dgpe_fixed.cuh"

namespace dgpe {
bool fx_run1(int which, const KArgs &a, cudaStream_t st) { return FxLaunch<1>::run<double>(which, a, st); }
cudaError_t fx_init1(int nx, int ny, int nz) { return FxLaunch<1>::init<double>(nx, ny, nz); }
}  // namespace dgpe
