// Fixed-point transforms of the FP64 precision: every eighth line length, from number 3 of the
// list on (dgpe_fixed.cuh); eight translation units, so that they build in parallel.
#include "dgpe_fixed.cuh"

namespace dgpe {
bool fx_run3(int which, const KArgs &a, cudaStream_t st) { return FxLaunch<3>::run<double>(which, a, st); }
cudaError_t fx_init3(int nx, int ny, int nz) { return FxLaunch<3>::init<double>(nx, ny, nz); }
}  // namespace dgpe
