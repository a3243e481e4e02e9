// Fixed-point transforms of the FP64 precision: every eighth line length, from number 0 of the
// list on (dgpe_fixed.cuh); eight translation units, so that they build in parallel.
#include "dgpe_fixed.cuh"

namespace dgpe {
bool fx_run0(int which, const KArgs &a, cudaStream_t st) { return FxLaunch<0>::run<double>(which, a, st); }
cudaError_t fx_init0(int nx, int ny, int nz) { return FxLaunch<0>::init<double>(nx, ny, nz); }
bool fx_length(int n) { return fx_index(n) >= 0; }
cudaError_t fx_tables(void *tw, int n, cudaStream_t st) {
  if (!fx_length(n)) return cudaSuccess;
  k_fx_twiddles<<<(2 * n + 127) / 128, 128, 0, st>>>(static_cast<fxw *>(tw), n, st_radix(n, 0), st_radix(n, 1),
                                                    st_radix(n, 2));
  return cudaGetLastError();
}
}  // namespace dgpe
