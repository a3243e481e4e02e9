// dgpe_moments_noalloc: the norm and rms sizes of a caller's psi, computed without any
// device allocation.  The scratch memory of its reduction (per-block partial sums and the
// last-block counter) is a file-scope __device__ array of fixed size, so the call needs
// neither a context nor a workspace.  The paper has no counterpart of this entry point.
//
// Scratch: kNoAllocMaxBlocks x 4 doubles of partial sums + one counter, 256 KiB in all (the
// grid is capped at kNoAllocMaxBlocks blocks whatever the size).
// Every GPU that loads libdgpe.so holds one copy of it until the process exits, and every
// call on that GPU shares it: calls whose work overlaps on the GPU (different streams
// without ordering between them) race on it and give wrong results.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "dgpe.h"
#include "dgpe_device.cuh"

using namespace dgpe;

namespace {

constexpr int kNoAllocThreads = 256;
constexpr int kNoAllocMaxBlocks = 8192;
constexpr int kNoAllocMaxN = 512;   // points per axis (the library's grid limit)

struct NoAllocScratch {
  unsigned int ticket;            // last-block counter: must be 0 when a reduction starts
  unsigned int pad[63];
  double partials[kNoAllocMaxBlocks * 4];
};

__device__ __align__(256) NoAllocScratch g_noalloc_scratch;

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void *g_scratch_addr[kMaxDevices] = {};

// Device address of this GPU's copy of the scratch array, looked up once per device with
// that device current (in host code the symbol itself is only a host-side stand-in).
int scratch_address(NoAllocScratch **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DGPE_ECUDA;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return DGPE_ECUDA;
    g_scratch_addr[dev] = p;
  }
  *out = static_cast<NoAllocScratch *>(g_scratch_addr[dev]);
  return DGPE_OK;
}

// Sums n, x^2 n, y^2 n, z^2 n (FP64, weighted by the quadrature rule) with one warp per
// z-line at a time (grid-stride over the nx*ny lines): the line's (i, j) costs one division
// per line, the z weights come from a shared table.  The last block turns the sums into
// norm = hx hy hz sum w n and rms_d = sqrt(sum w d^2 n / sum w n).
template <typename R>
__global__ void __launch_bounds__(kNoAllocThreads)
    k_moments_noalloc(const cplx<R> *__restrict__ psi, int nx, int ny, int nz, double hx, double hy, double hz,
                      int simpson, NoAllocScratch *scr, double *out) {
  __shared__ double wz[kNoAllocMaxN], wz2[kNoAllocMaxN];   // w_k and w_k z_k^2
  for (int k = threadIdx.x; k < nz; k += blockDim.x) {
    const double z = coordinate(k, nz, hz), w = quad_weight(k, nz, simpson);
    wz[k] = w;
    wz2[k] = w * z * z;
  }
  __syncthreads();
  const int lane = threadIdx.x & (kWarp - 1);
  const long long nlines = (long long)nx * ny;
  const long long nwarps = (long long)gridDim.x * (blockDim.x / kWarp);
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (long long l = (long long)blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp; l < nlines; l += nwarps) {
    const int i = (int)(l / ny), j = (int)(l - (long long)i * ny);
    const cplx<R> *line = psi + l * nz;
    double s0 = 0.0, sz = 0.0;
    for (int k = lane; k < nz; k += kWarp) {
      const cplx<R> w = line[k];
      const double d = (double)w.re * w.re + (double)w.im * w.im;
      s0 = fma(wz[k], d, s0);
      sz = fma(wz2[k], d, sz);
    }
    const double x = coordinate(i, nx, hx), y = coordinate(j, ny, hy);
    const double t = quad_weight(i, nx, simpson) * quad_weight(j, ny, simpson) * s0;
    v[0] += t;
    v[1] += x * x * t;
    v[2] += y * y * t;
    v[3] += quad_weight(i, nx, simpson) * quad_weight(j, ny, simpson) * sz;
  }
  double sum[4];
  if (reduce_across_blocks<4>(v, sum, scr->partials, &scr->ticket) && threadIdx.x == 0) {
    for (int q = 0; q < 4; ++q) v[q] = sum[q];
    out[0] = hx * hy * hz * v[0];
    out[1] = sqrt(v[1] / v[0]);
    out[2] = sqrt(v[2] / v[0]);
    out[3] = sqrt(v[3] / v[0]);
  }
}

// FP32 data.  The kernel above spends six to eight FP64-pipe instructions per point (two
// conversions among them; GB300 issues 2 per clock per SM): 1.42 ms at 512x512x384 against 0.12 ms
// of HBM time.  Here a lane sums its points in integers, in units taken from the largest of them:
//   - a component is m 2^(e - 150) with a 24-bit m; its square, 48 bits, goes to a 64-bit integer
//     under the lane's exponent E: exact where the component is above 2^-4 of the lane's first
//     largest, else rounded at 2^-54 of that one's density (E leaves 3 binades for later ones to grow);
//   - the weights are integers (3 x the quadrature weights, squared signed indices); the sums of
//     products, of the high and of the low words apart, are exact;
//   - a lane passes its sums on to FP64 once per unit of up to 8 lines (or where the x index changes
//     or a point outgrows E).
// So the sums are better than FP64's own.  Lanes that meet an infinity or a NaN take those points in
// FP64.  Bound by integer issue (about 35 instructions per point): 1.42 -> 0.29 ms at 512x512x384.  rms error
// over 36 grids of 2.6e5 to 1.3e6 points, norm and sizes: 1.5e-16, 8e-17 -> 1.05e-16, 7e-17.  (Pairs of FP32
// in place of the integers take 0.25 ms and leave 2.5e-16, 1.0e-16.)
constexpr int kMomentPairs = 2;   // pairs of points in a lane's registers (three leave more of a line's end idle)

// A sum of integers 2^32 h + l, and additions of w d and of w times another sum
struct WideSum {
  unsigned long long h = 0, l = 0;
  __device__ __forceinline__ void add(unsigned w, unsigned long long d) {
    h += (unsigned long long)w * (unsigned)(d >> 32);
    l += (unsigned long long)w * (unsigned)d;
  }
  __device__ __forceinline__ void add(unsigned w, const WideSum &s) {
    h += w * s.h;
    l += w * s.l;
  }
  __device__ __forceinline__ double value() const { return fma((double)h, 4294967296.0, (double)l); }
};
// x^2 in units of 2^(2 (E - 150) - 14) for |x| < 2^(E - 126), rounded (halves up); x comes scaled by a
// power of two that takes E to `base` (63 at least: a zero's or a subnormal's exponent field, 0, then
// shifts everything out).  Shifts by the width and more give 0 (shl.b32, shr.u64).
__device__ __forceinline__ unsigned long long square_units(float x, int base) {
  const unsigned u = __float_as_uint(x), m = ((u & 0x7fffffu) | 0x800000u) << 7;
  const unsigned s = 2 * (base - (int)((u >> 23) & 0xff));
  unsigned lo, hi;   // 2^(s - 1)
  unsigned long long r;
  asm("shl.b32 %0, 1, %1;" : "=r"(lo) : "r"(s - 1));
  asm("shl.b32 %0, 1, %1;" : "=r"(hi) : "r"(s - 33));
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"((unsigned long long)m * m + ((unsigned long long)hi << 32 | lo)), "r"(s));
  return r;
}

template <bool WIDE>
__global__ void __launch_bounds__(kNoAllocThreads, 3)
    k_moments_f32(const float2 *__restrict__ psi, int nx, int ny, int nz, double hx, double hy, double hz, int simpson,
                  int lines_per_unit, NoAllocScratch *scr, double *out) {
  __shared__ uint4 wz[kNoAllocMaxN / 2];   // W and W k'^2 of two consecutive points
  for (int p = threadIdx.x; p < nz / 2; p += blockDim.x) {
    const int k0 = 2 * p - nz / 2, k1 = k0 + 1;
    const unsigned w0 = quad_weight3(2 * p, nz, simpson), w1 = quad_weight3(2 * p + 1, nz, simpson);
    wz[p] = make_uint4(w0, w0 * (unsigned)(k0 * k0), w1, w1 * (unsigned)(k1 * k1));
  }
  __syncthreads();
  const int lane = threadIdx.x & (kWarp - 1), np = nz / 2;
  const int nlines = nx * ny;
  const int nwarps = gridDim.x * (blockDim.x / kWarp);
  const int nunits = (nlines + lines_per_unit - 1) / lines_per_unit;
  double v[4] = {0.0, 0.0, 0.0, 0.0};   // sums of W n, i'^2 W n, j'^2 W n, k'^2 W n
  // the sums of one run of lines of equal x index, under E
  WideSum s0, sy, sz;
  int E = 0;   // 0: empty
  auto flush = [&](int i) {
    if (!E) return;
    const double un = __hiloint2double((1023 + 2 * (E - 150) - 14) << 20, 0);
    const int ii = i - nx / 2;
    const double wx = (double)quad_weight3(i, nx, simpson) * un;
    const double t = wx * s0.value();
    v[0] += t;
    v[1] = fma((double)(ii * ii), t, v[1]);
    v[2] = fma(wx, sy.value(), v[2]);
    v[3] = fma(wx, sz.value(), v[3]);
    s0 = sy = sz = WideSum{};
    E = 0;
  };
  auto load = [&](int l, int p0, float4 (&c)[kMomentPairs]) {
#pragma unroll
    for (int u = 0; u < kMomentPairs; ++u) {
      const int p = p0 + u * kWarp + lane;
      if (p < np) {
        const float2 *q = psi + (size_t)l * nz + 2 * p;
        if constexpr (WIDE) {
          c[u] = __ldg(reinterpret_cast<const float4 *>(q));
        } else {
          const float2 a = __ldg(q), b = __ldg(q + 1);
          c[u] = make_float4(a.x, a.y, b.x, b.y);
        }
      } else {
        c[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  for (int unit = blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp; unit < nunits; unit += nwarps) {
    const int l0 = unit * lines_per_unit, l1 = min(nlines, l0 + lines_per_unit);
    int i = l0 / ny, j = l0 - i * ny;
    float4 c[kMomentPairs], nxt[kMomentPairs];
    load(l0, 0, nxt);
    for (int l = l0; l < l1; ++l) {
      const unsigned wy = quad_weight3(j, ny, simpson), jj2 = (unsigned)((j - ny / 2) * (j - ny / 2));
      WideSum t0, tz;   // this line's sums of W_z n, k'^2 W_z n
      auto fold = [&]() {
        s0.add(wy, t0);
        sy.add(wy * jj2, t0);
        sz.add(wy, tz);
        t0 = tz = WideSum{};
      };
      for (int p0 = 0; p0 < np; p0 += kMomentPairs * kWarp) {
#pragma unroll
        for (int u = 0; u < kMomentPairs; ++u) c[u] = nxt[u];
        // the next points of the line, or the next line's first
        if (p0 + kMomentPairs * kWarp < np) load(l, p0 + kMomentPairs * kWarp, nxt);
        else if (l + 1 < l1) load(l + 1, 0, nxt);
        unsigned m = 0u;   // twice the bits of the largest magnitude
#pragma unroll
        for (int u = 0; u < kMomentPairs; ++u)
          m = max(max(m, max(__float_as_uint(c[u].x) << 1, __float_as_uint(c[u].y) << 1)),
                  max(__float_as_uint(c[u].z) << 1, __float_as_uint(c[u].w) << 1));
        if (m == 0u) continue;
        const int e = max((int)(m >> 24), 1);
        if (e == 255) {   // an infinity or a NaN: in FP64
          const int ii = i - nx / 2, jj = j - ny / 2;
          const double wxy = (double)(quad_weight3(i, nx, simpson) * quad_weight3(j, ny, simpson));
#pragma unroll 1
          for (int u = 0; u < 2 * kMomentPairs; ++u) {
            const int p = p0 + (u >> 1) * kWarp + lane;
            if (p >= np) break;
            const float2 z = psi[(size_t)l * nz + 2 * p + (u & 1)];
            const int k = 2 * p + (u & 1), kk = k - nz / 2;
            const double t = wxy * quad_weight3(k, nz, simpson) * ((double)z.x * z.x + (double)z.y * z.y);
            v[0] += t;
            v[1] += (double)(ii * ii) * t;
            v[2] += (double)(jj * jj) * t;
            v[3] += (double)(kk * kk) * t;
          }
          continue;
        }
        if (e > E) {   // the first points, or one above E: the sums so far stay at the old unit
          fold();
          flush(i);
          E = e + 3;
        }
        // psi scaled so that E becomes base = 200 (by 2^127 at most: base >= 131)
        const int sb = min(327 - E, 254), base = E + sb - 127;
        const float sc = __int_as_float(sb << 23);
#pragma unroll
        for (int u = 0; u < kMomentPairs; ++u) {
          const int p = p0 + u * kWarp + lane;
          const uint4 w = wz[min(p, np - 1)];   // (past the line's end the density is zero)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const unsigned long long d = square_units(__fmul_rn(h ? c[u].z : c[u].x, sc), base) +
                                         square_units(__fmul_rn(h ? c[u].w : c[u].y, sc), base);
            t0.add(h ? w.z : w.x, d);
            tz.add(h ? w.w : w.y, d);
          }
        }
      }
      fold();
      if (++j == ny) {
        flush(i);
        j = 0;
        ++i;
      }
    }
    if (j) flush(i);
  }
  double sum[4];
  if (reduce_across_blocks<4>(v, sum, scr->partials, &scr->ticket) && threadIdx.x == 0) {
    // the factors with their rounding errors carried along, so that the results keep the
    // sums' own accuracy: norm = hx hy hz sum / 27 (the integer Simpson weights' (1/3)^3) ...
    const double a = hx * hy, b = a * hz, c = b * sum[0];
    const double eb = fma(a, hz, -b) + fma(hx, hy, -a) * hz, ec = fma(b, sum[0], -c) + eb * sum[0];
    const double q = c / (simpson ? 27.0 : 1.0);
    out[0] = isfinite(c) ? q + (fma(-q, simpson ? 27.0 : 1.0, c) + ec) / (simpson ? 27.0 : 1.0) : c;
    // ... and rms_d = h_d sqrt(sum_d / sum)
    const double h[3] = {hx, hy, hz};
    for (int d = 0; d < 3; ++d) {
      const double r = sum[1 + d] / sum[0], t = sqrt(r), u = h[d] * t;
      out[1 + d] = t > 0.0 ? u + (fma(h[d], t, -u) + h[d] * (fma(-t, t, r) / (2.0 * t))) : u;
    }
  }
}

// One resident wave of CTAs (three of 256 threads per SM); a warp takes up to 8 lines at a time,
// fewer where that leaves warps without work.
int moments_f32(const void *psi, const dgpe_params *p, int simpson, long long nlines, NoAllocScratch *scr, double *out,
                cudaStream_t st) {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
    return DGPE_ECUDA;
  const long long warps = (long long)nsm * 3 * (kNoAllocThreads / kWarp);
  const int lines = (int)std::max<long long>(1, std::min<long long>(8, nlines / (warps * 4)));
  const long long units = (nlines + lines - 1) / lines, per_block = kNoAllocThreads / kWarp;
  const unsigned blocks = (unsigned)std::min<long long>((units + per_block - 1) / per_block,
                                                        std::min<long long>(nsm * 3, kNoAllocMaxBlocks));
  const float2 *q = static_cast<const float2 *>(psi);
  if (reinterpret_cast<uintptr_t>(psi) % 16 == 0)
    k_moments_f32<true><<<blocks, kNoAllocThreads, 0, st>>>(q, p->nx, p->ny, p->nz, p->hx, p->hy, p->hz, simpson, lines, scr, out);
  else   // (8-byte aligned)
    k_moments_f32<false><<<blocks, kNoAllocThreads, 0, st>>>(q, p->nx, p->ny, p->nz, p->hx, p->hy, p->hz, simpson, lines, scr, out);
  return cudaGetLastError() == cudaSuccess ? DGPE_OK : DGPE_ECUDA;
}

}  // namespace

extern "C" int dgpe_moments_noalloc(const void *psi, const dgpe_params *p, double *out, void *cuda_stream) {
  if (!psi || !p || !out) return DGPE_EINVAL;
  if (p->nx < 1 || p->ny < 1 || p->nz < 1) return DGPE_EINVAL;
  if (!(p->hx > 0 && p->hy > 0 && p->hz > 0) || !isfinite(p->hx) || !isfinite(p->hy) || !isfinite(p->hz))
    return DGPE_EINVAL;
  if (p->precision != DGPE_FP64 && p->precision != DGPE_MIXED && p->precision != DGPE_DF64) return DGPE_EINVAL;
  if (p->integration != DGPE_RECTANGLE && p->integration != DGPE_SIMPSON) return DGPE_EINVAL;
  if (p->nx > kNoAllocMaxN || p->ny > kNoAllocMaxN || p->nz > kNoAllocMaxN) return DGPE_EUNSUPPORTED;
  NoAllocScratch *scr = nullptr;
  int rc = scratch_address(&scr);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // the counter must start at zero (a reduction that was cut short may have left it set)
  if (cudaMemsetAsync(&scr->ticket, 0, sizeof(unsigned int), st) != cudaSuccess) return DGPE_ECUDA;
  const long long nlines = (long long)p->nx * p->ny;
  const long long warps_per_block = kNoAllocThreads / kWarp;
  const unsigned blocks = (unsigned)std::min<long long>((nlines + warps_per_block - 1) / warps_per_block,
                                                        kNoAllocMaxBlocks);
  const int simpson = p->integration == DGPE_SIMPSON;
  if (p->precision != DGPE_MIXED)   // complex128 (FP64, and the double-float mode's caller format)
    k_moments_noalloc<double><<<blocks, kNoAllocThreads, 0, st>>>(static_cast<const cplx<double> *>(psi), p->nx,
                                                                  p->ny, p->nz, p->hx, p->hy, p->hz, simpson,
                                                                  scr, out);
  // Integers where the time is the arithmetic's: below 2^17 points the FP64 kernel takes under 2 us of
  // its pipe.  Odd lines have no pairs of points.
  else if (p->nz % 2 == 0 && nlines * p->nz >= (1 << 17))
    return moments_f32(psi, p, simpson, nlines, scr, out, st);
  else
    k_moments_noalloc<float><<<blocks, kNoAllocThreads, 0, st>>>(static_cast<const cplx<float> *>(psi), p->nx,
                                                                 p->ny, p->nz, p->hx, p->hy, p->hz, simpson,
                                                                 scr, out);
  return cudaGetLastError() == cudaSuccess ? DGPE_OK : DGPE_ECUDA;
}
