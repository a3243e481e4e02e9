// Fixed-point transforms of the FP64 precision: every eighth line length, from number 0 of the
// list on (dgpe_fixed.cuh); eight translation units, so that they build in parallel.
#include <algorithm>

#include "dgpe_fixed.cuh"

namespace dgpe {
bool fx_run0(int which, const KArgs &a, cudaStream_t st) { return FxLaunch<0>::run<double>(which, a, st); }
cudaError_t fx_init0(int nx, int ny, int nz) { return FxLaunch<0>::init<double>(nx, ny, nz); }
template <bool CPLX>
static cudaError_t cn_launch(int axis, const KArgs &a, int reduce, int renorm, cudaStream_t st) {
  const int lines = axis == 2 ? a.nx * a.ny : (axis == 0 ? a.ny : a.nx) * a.nz, tiles = (lines + 63) / 64;
  // CTAs per SM: four where they take more than two rounds, else three, with which more of y and psi
  // stays in L2 (y sweep, real time: 256^3, 1024 tiles, 285 us with three and 315 with four;
  // 480x480x250, 1875 tiles, 935 and 872)
  const int nsm = std::max(a.nsm, 1), grid = std::min(tiles, (tiles > 8 * nsm ? 4 : 3) * nsm);
  if (axis == 2) k_cn_fx<CPLX, 2, false><<<grid, kFxcThreads, fx_cn_smem<2>(false, 0), st>>>(a, renorm);
  else if (axis == 1) k_cn_fx<CPLX, 1, false><<<grid, kFxcThreads, fx_cn_smem<1>(false, 0), st>>>(a, renorm);
  else if (reduce) k_cn_fx<CPLX, 0, true><<<grid, kFxcThreads, fx_cn_smem<0>(true, a.nx), st>>>(a, renorm);
  else k_cn_fx<CPLX, 0, false><<<grid, kFxcThreads, fx_cn_smem<0>(false, 0), st>>>(a, renorm);
  return cudaGetLastError();
}
cudaError_t fx_cn(int axis, const KArgs &a, int reduce, int renorm, cudaStream_t st) {
  return a.imag ? cn_launch<false>(axis, a, reduce, renorm, st) : cn_launch<true>(axis, a, reduce, renorm, st);
}
cudaError_t fx_cn_init() {
  cudaError_t e = cudaSuccess;
  auto opt = [&](auto k, size_t sm) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  };
  auto all = [&](auto cplx) {
    constexpr bool Z = decltype(cplx)::value;
    opt(k_cn_fx<Z, 2, false>, fx_cn_smem<2>(false, 0));
    opt(k_cn_fx<Z, 1, false>, fx_cn_smem<1>(false, 0));
    opt(k_cn_fx<Z, 0, false>, fx_cn_smem<0>(false, 0));
    opt(k_cn_fx<Z, 0, true>, fx_cn_smem<0>(true, 512));
  };
  all(std::true_type{});
  all(std::false_type{});
  return e;
}
cudaError_t fx_cn_tables(const CnJobs &jobs, cudaStream_t st) {
  if (jobs.n > 0) k_fx_cn_tables<<<jobs.n, kWarp, 0, st>>>(jobs);
  return cudaGetLastError();
}
bool fx_length(int n) { return fx_index(n) >= 0; }
cudaError_t fx_tables(void *tw, int n, cudaStream_t st) {
  if (!fx_length(n)) return cudaSuccess;
  k_fx_twiddles<<<(2 * n + 127) / 128, 128, 0, st>>>(static_cast<fxw *>(tw), n, st_radix(n, 0), st_radix(n, 1),
                                                    st_radix(n, 2));
  return cudaGetLastError();
}
}  // namespace dgpe
