// Fixed-point transforms of the FP64 precision: every eighth line length, from number 5 of the
// list on (dgpe_fixed.cuh); eight translation units, so that they build in parallel.
#include "dgpe_fixed.cuh"

namespace dgpe {
bool fx_run5(int which, const KArgs &a, cudaStream_t st) { return FxLaunch<5>::run<double>(which, a, st); }
cudaError_t fx_init5(int nx, int ny, int nz) { return FxLaunch<5>::init<double>(nx, ny, nz); }
}  // namespace dgpe
