// FP32 transforms of the general line lengths 2^a 3^b 5^c 7^d (12 .. 512) in two or three
// stages of radix 2 .. 10, every length its own instance: the y transforms (K2, K4), the x
// transforms with the dipolar kernel between them (K3), and K1 and K5 with the z transforms.
//
// The runtime-length transforms of dgpe_device.cuh take four to five radix-2/3/4/5/7/8 stages
// with every index computed at run time (about 85 instructions per element at 480 = 8 4 3 5),
// each stage a round trip through shared memory.  With radices up to 10 three stages reach every
// length, so only two round trips remain: the first stage reads global memory and the last one
// writes it.  Along x the last forward stage of radix R3 leaves a thread the elements
// j + s N/R3, which are the inputs of a first inverse stage of radix R3: it runs that stage on
// them at once (the inverse takes the radices in reverse order), four round trips in all for
// both transforms and the product by Ut(k).
// Bound by shared-memory latency and HBM.  us, before -> now (and of 6784 GB/s): K2 at 480x480x500
// 326 -> 190 (0.72), K3 520 -> 358 (0.38), with the spherical cutoff 641 -> 493; 384^3 112 -> 88
// (0.76), 183 -> 170; 240^3 41 -> 29, 67 -> 41; 64^3, 16 condensates, a step 128 -> 109.
#pragma once
#include "dgpe_device.cuh"

namespace dgpe {

// ---- butterflies of the composite radices ----------------------------------------------
// Good-Thomas prime-factor forms (no twiddles): 6 = 2 x 3, 10 = 2 x 5.
template <typename R, int DIR>
__device__ __forceinline__ void bf6(cplx<R> *v) {
  cplx<R> a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};   // n = 3 n1 + 2 n2
  bf3<R, DIR>(a);
  bf3<R, DIR>(b);
  v[0] = a[0] + b[0];   // k = 3 k1 + 4 k2 (mod 6)
  v[3] = a[0] - b[0];
  v[4] = a[1] + b[1];
  v[1] = a[1] - b[1];
  v[2] = a[2] + b[2];
  v[5] = a[2] - b[2];
}
template <typename R, int DIR>
__device__ __forceinline__ void bf10(cplx<R> *v) {
  cplx<R> a[5] = {v[0], v[2], v[4], v[6], v[8]}, b[5] = {v[5], v[7], v[9], v[1], v[3]};   // n = 5 n1 + 2 n2
  bf5<R, DIR>(a);
  bf5<R, DIR>(b);
#pragma unroll
  for (int k2 = 0; k2 < 5; ++k2) {   // k = 5 k1 + 6 k2 (mod 10)
    v[(6 * k2) % 10] = a[k2] + b[k2];
    v[(6 * k2 + 5) % 10] = a[k2] - b[k2];
  }
}
// 9 = 3 x 3 with the twiddles w9^(n2 k1)
template <typename R, int DIR>
__device__ __forceinline__ void bf9(cplx<R> *v) {
  const R c1 = R(0.76604444311897804), s1 = R(0.64278760968653933);   // cos, sin of 2 pi / 9
  const R c2 = R(0.17364817766693035), s2 = R(0.98480775301220806);   // of 4 pi / 9
  const R c4 = R(-0.93969262078590838), s4 = R(0.34202014332566873);  // of 8 pi / 9
  auto tw = [](cplx<R> z, R c, R s) {   // z e^{DIR i phi}
    return DIR < 0 ? cplx<R>{z.re * c + z.im * s, z.im * c - z.re * s} : cplx<R>{z.re * c - z.im * s, z.im * c + z.re * s};
  };
  cplx<R> c[3][3];   // [n2][k1]
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    c[n2][0] = v[n2];
    c[n2][1] = v[n2 + 3];
    c[n2][2] = v[n2 + 6];
    bf3<R, DIR>(c[n2]);
  }
  c[1][1] = tw(c[1][1], c1, s1);
  c[1][2] = tw(c[1][2], c2, s2);
  c[2][1] = tw(c[2][1], c2, s2);
  c[2][2] = tw(c[2][2], c4, s4);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cplx<R> t[3] = {c[0][k1], c[1][k1], c[2][k1]};
    bf3<R, DIR>(t);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[k2];
  }
}
template <typename R, int DIR, int P>
__device__ __forceinline__ void bf(cplx<R> *v) {
  if constexpr (P == 6) bf6<R, DIR>(v);
  else if constexpr (P == 9) bf9<R, DIR>(v);
  else if constexpr (P == 10) bf10<R, DIR>(v);
  else butterfly<R, DIR, P>(v);
}

// ---- plans -------------------------------------------------------------------------------
// Radix of stage s (0, 1, 2) of the fewest-stage plan of n: descending radices <= 10, the
// largest as small as possible, then the smallest as large as possible; 1 past the last stage.
__host__ __device__ constexpr int st_radix(int n, int s) {
  for (int a = 2; a <= 10; ++a)
    if (n % a == 0 && n / a <= a && n / a >= 2) return s == 0 ? a : s == 1 ? n / a : 1;
  for (int a = 2; a <= 10; ++a) {
    if (n % a) continue;
    int best = 0;
    for (int c = 2; c <= a; ++c) {
      const int m = n / a;
      if (m % c == 0 && m / c >= c && m / c <= a) best = c;
    }
    if (best) return s == 0 ? a : s == 1 ? n / a / best : best;
  }
  return 0;
}
// (X(n) for every length with such a plan; 128, 256 and 512 have register-resident transforms)
#define DGPE_STAGE_LENGTHS(X) \
  X(12) X(14) X(16) X(18) X(20) X(24) X(28) X(30) X(32) X(36) X(40) X(42) X(48) X(50) X(54) X(56) X(60) X(64) X(70) \
  X(72) X(80) X(84) X(90) X(96) X(98) X(100) X(108) X(112) X(120) X(126) X(140) X(144) X(150) X(160) X(162) X(168) \
  X(180) X(192) X(196) X(200) X(210) X(216) X(224) X(240) X(250) X(252) X(270) X(280) X(288) X(294) X(300) X(320) \
  X(324) X(336) X(350) X(360) X(378) X(384) X(392) X(400) X(420) X(432) X(448) X(450) X(480) X(486) X(490) X(500) X(504)

// and with those: the lengths of the z kernels
#define DGPE_STAGE_ALL(X) X(128) X(256) X(512) DGPE_STAGE_LENGTHS(X)
constexpr bool st_xy(int n) { return n != 128 && n != 256 && n != 512; }

template <int N>
struct Stages {
  static constexpr int R1 = st_radix(N, 0), R2 = st_radix(N, 1), R3 = st_radix(N, 2);
  static_assert(R1 * R2 * R3 == N, "a plan of the length");
};

// Slot of element i of a line after a first stage of radix P1 (outputs j P1 + s on neighbouring
// threads j: one pad slot per P1 where P1 is even, so the stride is odd), and after a second one
// (outputs in blocks of P1 P2: threads k < P1 of neighbouring blocks side by side modulo G, the
// elements that a half-warp's width covers: 16 along a line, 2 rows of 8 columns).
template <int P1>
__host__ __device__ constexpr int st_pad1(int i) { return i + (P1 % 2 == 0 ? i / P1 : 0); }
template <int P1, int P2, int G>
__host__ __device__ constexpr int st_pad2_gap() { return ((P1 - P1 * P2) % G + G) % G; }
template <int P1, int P2, int P3, int G>
__host__ __device__ constexpr int st_slots() {
  const int n = P1 * P2 * P3;
  const int a = st_pad1<P1>(n), b = P3 > 1 ? n + P3 * st_pad2_gap<P1, P2, G>() : 0;
  return a > b ? a : b;
}

// Twiddle tables of a plan (P1, P2, P3): entry of stage 2 (ns = P1), output index k < P1, r: at
// (r - 1) P1 + k; stage 3 (ns = P1 P2) after them, at P1 (P2 - 1) + (r - 1) P1 P2 + k: the threads
// of a warp, neighbouring k, read neighbouring entries.  Two tables per axis: the plan, and its
// radices in reverse order (the inverse x transforms), at st_table(n) entries each.
__host__ __device__ constexpr int st_table(int n) { return n; }

template <int DIR, int P, int NS>
__device__ __forceinline__ void st_twiddle(cplx<float> *v, const cplx<float> *__restrict__ tw, int k) {
#pragma unroll
  for (int r = 1; r < P; ++r) v[r] = twiddle<DIR>(v[r], ldg(tw + (r - 1) * NS + k));
}

// ---- K2 / K4 -----------------------------------------------------------------------------
template <int N>
struct StageY {
  using S = Stages<N>;
  static constexpr int NT = 128;
  static constexpr int L = N <= 32 ? 64 : 2048 / N < 1 ? 1 : 2048 / N;   // lines per CTA
  static constexpr int SLOTS = st_slots<S::R1, S::R2, S::R3, 16>() | 1;
  static constexpr size_t smem = (size_t)(S::R3 > 1 ? 2 : 1) * L * SLOTS * sizeof(cplx<float>);
};

template <int DIR, int N>
__global__ void __launch_bounds__(StageY<N>::NT) k_ffty_st(const __grid_constant__ KArgs a0, const KArgs *ga) {
  using C = cplx<float>;
  using Y = StageY<N>;
  constexpr int R1 = Y::S::R1, R2 = Y::S::R2, R3 = Y::S::R3, SL = Y::SLOTS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const KArgs &a = ga ? ga[blockIdx.z] : a0;
  C *sa = reinterpret_cast<C *>(smem_raw), *sb = sa + Y::L * SL;
  const int total = a.nzh * a.nx, l0 = blockIdx.x * Y::L, nl = min(Y::L, total - l0);
  C *g = reinterpret_cast<C *>(a.spec) + (size_t)l0 * N;
  const C *tw = reinterpret_cast<const C *>(a.tw_st[1]);
  {
    constexpr int NB = N / R1;
    for (int it = threadIdx.x; it < nl * NB; it += Y::NT) {
      const int l = it / NB, j = it - l * NB;
      const C *x = g + l * N + j;
      C v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = x[r * NB];
      bf<float, DIR, R1>(v);
      C *y = sa + l * SL + st_pad1<R1>(j * R1);
#pragma unroll
      for (int s = 0; s < R1; ++s) y[s] = v[s];
    }
  }
  __syncthreads();
  constexpr int GAP = st_pad2_gap<R1, R2, 16>();
  {
    constexpr int NB = N / R2;
    for (int it = threadIdx.x; it < nl * NB; it += Y::NT) {
      const int l = it / NB, j = it - l * NB, jb = j / R1, k = j - jb * R1;
      const C *x = sa + l * SL + st_pad1<R1>(j);
      C v[R2];
#pragma unroll
      for (int r = 0; r < R2; ++r) v[r] = x[st_pad1<R1>(r * NB)];
      st_twiddle<DIR, R2, R1>(v, tw, k);
      bf<float, DIR, R2>(v);
      if constexpr (R3 > 1) {
        C *y = sb + l * SL + jb * (R1 * R2 + GAP) + k;
#pragma unroll
        for (int s = 0; s < R2; ++s) y[s * R1] = v[s];
      } else {
        C *y = g + l * N + k;
#pragma unroll
        for (int s = 0; s < R2; ++s) y[s * R1] = v[s];
      }
    }
  }
  if constexpr (R3 > 1) {
    __syncthreads();
    constexpr int NB = N / R3;
    for (int it = threadIdx.x; it < nl * NB; it += Y::NT) {
      const int l = it / NB, j = it - l * NB;
      const C *x = sb + l * SL + j;
      C v[R3];
#pragma unroll
      for (int r = 0; r < R3; ++r) v[r] = x[r * (NB + GAP)];
      st_twiddle<DIR, R3, R1 * R2>(v, tw + R1 * (R2 - 1), j);
      bf<float, DIR, R3>(v);
      C *y = g + l * N + j;
#pragma unroll
      for (int s = 0; s < R3; ++s) y[s * NB] = v[s];
    }
  }
}

// ---- K3 ------------------------------------------------------------------------------------
template <int N>
struct StageX {
  using S = Stages<N>;
  static constexpr int B = 8;                                       // columns per CTA (64-byte rows)
  static constexpr int NT = N >= 200 ? 256 : N >= 64 ? 128 : 64;
  static constexpr int SLA = st_slots<S::R1, S::R2, S::R3, 2>(), SLB = st_slots<S::R3, S::R2, S::R1, 2>();
  static constexpr int SLOTS = SLA > SLB ? SLA : SLB;
  static constexpr size_t smem = 2 * (size_t)SLOTS * B * sizeof(cplx<float>);
};

// stage 2 of a plan (P1, P2, .) from buffer x to buffer y, element slots of B columns
template <int DIR, int N, int P1, int P2, int P3, int B, int NT>
__device__ __forceinline__ void st_middle(const cplx<float> *x0, cplx<float> *y0, const cplx<float> *tw, int b) {
  using C = cplx<float>;
  constexpr int NB = N / P2, GAP = st_pad2_gap<P1, P2, 2>();
  for (int j = threadIdx.x / B; j < NB; j += NT / B) {
    const int jb = j / P1, k = j - jb * P1;
    const C *x = x0 + st_pad1<P1>(j) * B + b;
    C v[P2];
#pragma unroll
    for (int r = 0; r < P2; ++r) v[r] = x[st_pad1<P1>(r * NB) * B];
    st_twiddle<DIR, P2, P1>(v, tw, k);
    bf<float, DIR, P2>(v);
    C *y = y0 + (jb * (P1 * P2 + GAP) + k) * B + b;
#pragma unroll
    for (int s = 0; s < P2; ++s) y[s * P1 * B] = v[s];
  }
}

template <int N>
__global__ void __launch_bounds__(StageX<N>::NT) k3_st(const __grid_constant__ KArgs a0, const KArgs *ga) {
  using C = cplx<float>;
  using X = StageX<N>;
  constexpr int R1 = X::S::R1, R2 = X::S::R2, R3 = X::S::R3, B = X::B, NT = X::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const KArgs &a = ga ? ga[blockIdx.z] : a0;
  C *sa = reinterpret_cast<C *>(smem_raw), *sb = sa + X::SLOTS * B;
  const int b = threadIdx.x % B, m = blockIdx.y, jy = blockIdx.x * B + b, ny = a.ny;
  const bool on = jy < ny;
  C *g = reinterpret_cast<C *>(a.spec) + (size_t)m * a.nx * ny + (on ? jy : 0);
  const C *tw = reinterpret_cast<const C *>(a.tw_st[0]), *twr = tw + st_table(N);
  {
    constexpr int NB = N / R1;
    for (int j = threadIdx.x / B; j < NB; j += NT / B) {
      C v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = on ? g[(size_t)(j + r * NB) * ny] : czero<float>();
      bf<float, -1, R1>(v);
      C *y = sa + st_pad1<R1>(j * R1) * B + b;
#pragma unroll
      for (int s = 0; s < R1; ++s) y[s * B] = v[s];
    }
  }
  __syncthreads();
  // the last forward stage (radix P, ns = N / P, from `x`), Ut(k) = 3 kz^2 / |k|^2 - 1
  // (Ut(0) = 0, k_d = q_d 2 pi / (n_d h_d) with the signed frequency q_d), the first inverse
  // stage on the same elements, to `y`
  constexpr int P = R3 > 1 ? R3 : R2, NBL = N / P;
  constexpr int GAP = st_pad2_gap<R1, R2, 2>();
  if constexpr (R3 > 1) {
    st_middle<-1, N, R1, R2, R3, B, NT>(sa, sb, tw, b);
    __syncthreads();
  }
  {
    const float fx = a.kf[0], fy = a.kf[1], fz = a.kf[2];
    const float ky = (float)(jy <= ny / 2 ? jy : jy - ny) * fy, kz = (float)m * fz;
    const float kz2 = kz * kz, kyz2 = fmaf(ky, ky, kz2), kz23 = 3.0f * kz2;
    const bool cut = a.has_cutoff;
    const float rc = a.cutoff_f;
    const C *x0 = R3 > 1 ? sb : sa;
    C *y0 = R3 > 1 ? sa : sb;
    for (int j = threadIdx.x / B; j < NBL; j += NT / B) {
      const C *x = x0 + (R3 > 1 ? j : st_pad1<R1>(j)) * B + b;
      C v[P];
#pragma unroll
      for (int r = 0; r < P; ++r) v[r] = x[(R3 > 1 ? r * (NBL + GAP) : st_pad1<R1>(r * NBL)) * B];
      st_twiddle<-1, P, NBL>(v, R3 > 1 ? tw + R1 * (R2 - 1) : tw, j);
      bf<float, -1, P>(v);
#pragma unroll
      for (int s = 0; s < P; ++s) {
        const int i = j + s * NBL;
        const float kx = (float)(i <= N / 2 ? i : i - N) * fx;
        const float k2 = fmaf(kx, kx, kyz2);
        float u = k2 > 0.0f ? __fdividef(kz23, k2) - 1.0f : 0.0f;
        if (cut && k2 > 0.0f) u *= cutoff_factor<float>(sqrtf(k2) * rc);
        v[s] = scale(v[s], u);
      }
      bf<float, +1, P>(v);
      C *y = y0 + st_pad1<P>(j * P) * B + b;
#pragma unroll
      for (int s = 0; s < P; ++s) y[s * B] = v[s];
    }
  }
  __syncthreads();
  // the inverse plan (P, .., R1)
  if constexpr (R3 > 1) {
    st_middle<+1, N, R3, R2, R1, B, NT>(sa, sb, twr, b);
    __syncthreads();
  }
  {
    constexpr int NB = N / R1, GAPR = st_pad2_gap<R3, R2, 2>();
    for (int j = threadIdx.x / B; j < NB; j += NT / B) {
      const C *x = sb + (R3 > 1 ? j : st_pad1<P>(j)) * B + b;
      C v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = x[(R3 > 1 ? r * (NB + GAPR) : st_pad1<P>(r * NB)) * B];
      st_twiddle<+1, R1, NB>(v, R3 > 1 ? twr + R3 * (R2 - 1) : twr, j);
      bf<float, +1, R1>(v);
      if (on) {
#pragma unroll
        for (int s = 0; s < R1; ++s) g[(size_t)(j + s * NB) * ny] = v[s];
      }
    }
  }
}

// ---- K1 and K5 ------------------------------------------------------------------------------
// z lines (K1 and K5's step: of the lengths that have no kernel in dgpe_device.cuh, 64, 96, 128, 256,
// 384 and 512 have), in tiles of 2 PZ real lines packed in pairs.
// Two or three stages instead of the four or five of the runtime lengths, the first one reading global
// memory and the last one feeding the potential step, Phi or the observables in registers; the L2
// prefetch of the tile kernels.  Bound by latency at 16 to 24 warps per SM.  us, runtime-length kernels
// -> these: a step at 480x480x500 (imaginary time) 4.05 -> 3.03 ms, K1 343 there (of 204 at the copy
// bandwidth), K5 938 (of 340); observables at 384x360x320 (5-point gradient) 829 -> 728, Phi 250 -> 116.
template <int N>
struct StageZ {
  using S = Stages<N>;
  static constexpr bool kOwn = N != 64 && N != 96 && N != 128 && N != 256 && N != 384 && N != 512;
  static constexpr int NT = 256;
  static constexpr int P1 = N <= 64 ? 16 : 8;     // pairs per K1 tile: rows of 128 bytes of the spectrum
  static constexpr int P5 = N <= 64 ? 16 : N <= 256 ? 8 : 4;   // per K5 tile: two or three CTAs per SM
  static constexpr int PL = S::R3 > 1 ? S::R3 : S::R2, NBL = N / PL;
  static constexpr int TWL = S::R3 > 1 ? S::R1 * (S::R2 - 1) : 0;
  static constexpr int SLOTS = st_slots<S::R1, S::R2, S::R3, 16>() > N ? st_slots<S::R1, S::R2, S::R3, 16>() : N;
  // line stride: PZ lines by 16 / PZ elements on distinct banks
  __host__ __device__ static constexpr int stride(int pz) { return pz == 16 ? SLOTS | 1 : SLOTS + (16 / pz - SLOTS % 16 + 16) % 16; }
  static constexpr size_t smem1 = 2 * (size_t)P1 * stride(P1) * sizeof(cplx<float>);
  // K5: chunk of the z solve (32 lanes per line, padded to 32 chunks), the solve's tile, which lies
  // over the second transform buffer
  static constexpr int CH = k5_chunk(N);
  static constexpr int LS = (32 * CH + 34) | 1;
  static constexpr int kTile = 2 * P5 * LS > P5 * stride(P5) ? 2 * P5 * LS : P5 * stride(P5);
  static constexpr int kRes5 = CH > 10 ? 2 : 3;   // K5 CTAs per SM (registers)
  static constexpr size_t smem5 = ((size_t)P5 * stride(P5) + kTile + 10 * kWarp) * sizeof(cplx<float>);
};

// the middle of three stages and the last one of a tile of np <= PZ lines; out(line, j, v): elements
// j + s NBL of the result
template <int DIR, int N, int NT, int SL>
__device__ __forceinline__ void st_middle_z(const cplx<float> *x0, cplx<float> *y0, const cplx<float> *tw, int np) {
  using C = cplx<float>;
  using S = Stages<N>;
  constexpr int R1 = S::R1, R2 = S::R2, NB = N / R2, GAP = st_pad2_gap<R1, R2, 16>();
  for (int it = threadIdx.x; it < np * NB; it += NT) {
    const int l = it / NB, j = it - l * NB, jb = j / R1, k = j - jb * R1;
    const C *x = x0 + l * SL + st_pad1<R1>(j);
    C v[R2];
#pragma unroll
    for (int r = 0; r < R2; ++r) v[r] = x[st_pad1<R1>(r * NB)];
    st_twiddle<DIR, R2, R1>(v, tw, k);
    bf<float, DIR, R2>(v);
    C *y = y0 + l * SL + jb * (R1 * R2 + GAP) + k;
#pragma unroll
    for (int s = 0; s < R2; ++s) y[s * R1] = v[s];
  }
}
template <int DIR, int N, int NT, int SL, typename Out>
__device__ __forceinline__ void st_last_z(const cplx<float> *x0, const cplx<float> *tw, int np, Out out) {
  using C = cplx<float>;
  using Z = StageZ<N>;
  constexpr int R1 = Z::S::R1, PL = Z::PL, NB = Z::NBL, GAP = st_pad2_gap<R1, Z::S::R2, 16>();
  for (int it = threadIdx.x; it < np * NB; it += NT) {
    const int l = it / NB, j = it - l * NB;
    const C *x = x0 + l * SL + (Z::S::R3 > 1 ? j : st_pad1<R1>(j));
    C v[PL];
#pragma unroll
    for (int r = 0; r < PL; ++r) v[r] = x[Z::S::R3 > 1 ? r * (NB + GAP) : st_pad1<R1>(r * NB)];
    st_twiddle<DIR, PL, NB>(v, tw + Z::TWL, j);
    bf<float, DIR, PL>(v);
    out(l, j, v);
  }
}

// K1: densities (with a factor 1/2), forward transform, separation of the two real spectra
template <int N>
__global__ void __launch_bounds__(StageZ<N>::NT) k1_st(const __grid_constant__ KArgs a0, const KArgs *ga) {
  using C = cplx<float>;
  using Z = StageZ<N>;
  constexpr int R1 = Z::S::R1, PZ = Z::P1, SL = Z::stride(PZ), NT = Z::NT, NB = N / R1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const KArgs &a = ga ? ga[blockIdx.z] : a0;
  C *sa = reinterpret_cast<C *>(smem_raw), *sb = sa + PZ * SL;
  const int i = blockIdx.y, j0 = blockIdx.x * (2 * PZ), np = min(2 * PZ, a.ny - j0) >> 1;
  const C *psi = reinterpret_cast<const C *>(a.psi) + ((size_t)i * a.ny + j0) * N;
  const float s2 = 0.5f * (a.unit_scale ? 1.0f : scale_sq_of<float>(a.state));
  const C *tw = reinterpret_cast<const C *>(a.tw_st[2]);
  {   // the psi rows of the CTA one resident wave ahead into L2
    constexpr int kRes = (int)(225 * 1024 / (Z::smem1 + 1024)) < 6 ? (int)(225 * 1024 / (Z::smem1 + 1024)) : 6;
    AheadTile t;
    if (threadIdx.x == NT - 1 && ahead_tile(a, ga, kRes * a.nsm, t)) {
      const int j2 = t.bx2 * 2 * PZ;
      prefetch_l2(reinterpret_cast<const C *>(t.b->psi) + ((size_t)t.i2 * a.ny + j2) * N, min(2 * PZ, a.ny - j2) * N * (unsigned)sizeof(C));
    }
  }
  for (int it = threadIdx.x; it < np * NB; it += NT) {
    const int p = it / NB, j = it - p * NB;
    const C *row = psi + (size_t)(2 * p) * N + j;
    C v[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const C x = row[r * NB], y = row[N + r * NB];
      v[r] = {s2 * (x.re * x.re + x.im * x.im), s2 * (y.re * y.re + y.im * y.im)};
    }
    bf<float, -1, R1>(v);
    C *q = sa + p * SL + st_pad1<R1>(j * R1);
#pragma unroll
    for (int s = 0; s < R1; ++s) q[s] = v[s];
  }
  __syncthreads();
  if constexpr (Z::S::R3 > 1) {
    st_middle_z<-1, N, NT, SL>(sa, sb, tw, np);
    __syncthreads();
  }
  C *res = Z::S::R3 > 1 ? sa : sb;
  st_last_z<-1, N, NT, SL>(Z::S::R3 > 1 ? sb : sa, tw, np, [&](int p, int j, const C *v) {
#pragma unroll
    for (int s = 0; s < Z::PL; ++s) res[p * SL + j + s * Z::NBL] = v[s];
  });
  __syncthreads();
  C *spec = reinterpret_cast<C *>(a.spec) + (size_t)i * a.ny + j0;
  const size_t plane = (size_t)a.nx * a.ny;
  const int p = threadIdx.x % PZ;
  if (p < np) {
    for (int m = threadIdx.x / PZ; m <= N / 2; m += NT / PZ) {
      const C zm = res[p * SL + m], zc = res[p * SL + (m ? N - m : 0)];
      // (16-byte aligned: ny and j0 are even)
      *reinterpret_cast<float4 *>(spec + m * plane + 2 * p) =
          make_float4(zm.re + zc.re, zm.im - zc.im, zm.im + zc.im, zc.re - zm.re);
    }
  }
}

// K5: packing of the two half spectra, inverse transform (Phi); then the potential step and
// Crank-Nicolson along z on the tile, or Phi as the output, or the observables' sums (psi from global
// memory: a tile's own lines and their neighbours come from L1 and L2)
enum StageZMode { kStStep, kStPhi, kStObs };
template <int N, typename Coef, StageZMode MODE>
__global__ void __launch_bounds__(StageZ<N>::NT, MODE == kStStep ? StageZ<N>::kRes5 : 3) k5_st(const __grid_constant__ KArgs a0, const KArgs *ga) {
  using C = cplx<float>;
  using Z = StageZ<N>;
  constexpr int R1 = Z::S::R1, PZ = Z::P5, SL = Z::stride(PZ), NT = Z::NT, CH = Z::CH, LS = Z::LS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const KArgs &a = ga ? ga[blockIdx.z] : a0;
  C *sa = reinterpret_cast<C *>(smem_raw), *sb = sa + PZ * SL, *tile = sb;
  Coef *scan_s = reinterpret_cast<Coef *>(sb + Z::kTile);
  const int i = blockIdx.y, j0 = blockIdx.x * (2 * PZ), np = min(2 * PZ, a.ny - j0) >> 1;
  const Coef *tab = reinterpret_cast<const Coef *>(a.cnz_tab ? a.cnz_tab : a.cn[2].tab);
  if constexpr (MODE == kStStep)
    for (int q = threadIdx.x; q < 10 * kWarp; q += NT) scan_s[q] = ldg(tab + 4 * kWarp * CH + q);
  C *z0 = Z::S::R3 > 1 ? sa : sb, *z1 = Z::S::R3 > 1 ? sb : sa;   // the last stage reads sa
  {
    const C *spec = reinterpret_cast<const C *>(a.spec) + (size_t)i * a.ny + j0;
    const size_t plane = (size_t)a.nx * a.ny;
    const int p = threadIdx.x % PZ;
    if (p < np) {
#pragma unroll 4
      for (int m = threadIdx.x / PZ; m <= N / 2; m += NT / PZ) {
        const float4 x = *reinterpret_cast<const float4 *>(spec + m * plane + 2 * p);
        const bool end = m == 0 || m == N / 2;   // real bins of a real field's spectrum
        const float i1 = end ? 0.0f : x.y, i2 = end ? 0.0f : x.w;
        z0[p * SL + m] = {x.x - i2, i1 + x.z};
        if (!end) z0[p * SL + N - m] = {x.x + i2, x.z - i1};
      }
    }
  }
  {   // the rows of the CTA one resident wave ahead into L2
    AheadTile t;
    if (ahead_tile(a, ga, Z::kRes5 * a.nsm, t)) {
      const int j2 = t.bx2 * 2 * PZ, nl2 = min(2 * PZ, a.ny - j2);
      const size_t l2 = (size_t)t.i2 * a.ny + j2, plane = (size_t)a.nx * a.ny;
      const C *sp2 = reinterpret_cast<const C *>(t.b->spec) + l2;
      for (int m = threadIdx.x; m <= N / 2; m += NT) prefetch_l2(sp2 + m * plane, nl2 * (unsigned)sizeof(C));
      if (MODE == kStStep && threadIdx.x == NT - 1)
        prefetch_l2(reinterpret_cast<const C *>(t.b->psi) + l2 * N, nl2 * N * (unsigned)sizeof(C));
    }
  }
  __syncthreads();
  const C *tw = reinterpret_cast<const C *>(a.tw_st[2]);
  {
    constexpr int NB = N / R1;
    for (int it = threadIdx.x; it < np * NB; it += NT) {
      const int p = it / NB, j = it - p * NB;
      C v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = z0[p * SL + j + r * NB];
      bf<float, +1, R1>(v);
      C *q = z1 + p * SL + st_pad1<R1>(j * R1);
#pragma unroll
      for (int s = 0; s < R1; ++s) q[s] = v[s];
    }
  }
  __syncthreads();
  if constexpr (Z::S::R3 > 1) {
    st_middle_z<+1, N, NT, SL>(sb, sa, tw, np);
    __syncthreads();
  }
  if constexpr (MODE == kStPhi) {
    float *out = reinterpret_cast<float *>(a.out) + ((size_t)i * a.ny + j0) * N;
    const float f = a.inv_ntot_f;
    st_last_z<+1, N, NT, SL>(sa, tw, np, [&](int p, int j, const C *v) {
#pragma unroll
      for (int s = 0; s < Z::PL; ++s) {
        out[(size_t)(2 * p) * N + j + s * Z::NBL] = v[s].re * f;
        out[(size_t)(2 * p + 1) * N + j + s * Z::NBL] = v[s].im * f;
      }
    });
  } else if constexpr (MODE == kStObs) {
    constexpr int LP = N + 1;
    float *phi = reinterpret_cast<float *>(sb);
    const float f = a.inv_ntot_f;
    st_last_z<+1, N, NT, SL>(sa, tw, np, [&](int p, int j, const C *v) {
#pragma unroll
      for (int s = 0; s < Z::PL; ++s) {
        phi[2 * p * LP + j + s * Z::NBL] = v[s].re * f;
        phi[(2 * p + 1) * LP + j + s * Z::NBL] = v[s].im * f;
      }
    });
    __syncthreads();
    ObsSums t(a, i);
    for (int b = threadIdx.x / kWarp; b < 2 * np; b += NT / kWarp) {   // a warp per line
      t.begin(j0 + b);
      for (int n = threadIdx.x % kWarp; n < N; n += kWarp) t.add(n, phi[b * LP + n]);
      t.end();
    }
    t.finish();
  } else {
    C *psi = reinterpret_cast<C *>(a.psi) + ((size_t)i * a.ny + j0) * N;
    const float *dtv_y = reinterpret_cast<const float *>(a.dtv[1]) + j0, *dtv_z = reinterpret_cast<const float *>(a.dtv[2]);
    const float dtvx = ldg(reinterpret_cast<const float *>(a.dtv[0]) + i);
    const float sr = scale_of<float>(a.state);
    const bool scaled = sr != 1.0f;
    const float dtg = a.dtg_f, dtgdd = a.dtgdd_n_f;
    constexpr bool IMAG = std::is_same<Coef, float>::value;
    st_last_z<+1, N, NT, SL>(sa, tw, np, [&](int p, int j, const C *v) {
      C w[2][Z::PL];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int s = 0; s < Z::PL; ++s) w[h][s] = psi[(size_t)(2 * p + h) * N + j + s * Z::NBL];
      const float vy[2] = {dtvx + ldg(dtv_y + 2 * p), dtvx + ldg(dtv_y + 2 * p + 1)};
#pragma unroll
      for (int s = 0; s < Z::PL; ++s) {
        const int n = j + s * Z::NBL;
        const float vz = ldg(dtv_z + n);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          C z = w[h][s];
          if (scaled) z = scale(z, sr);
          const float dens = z.re * z.re + z.im * z.im;
          const float theta = fmaf(dtg, dens, fmaf(dtgdd, h ? v[s].im : v[s].re, vy[h] + vz));
          C o;
          if constexpr (IMAG) {
            o = scale(z, exp_r(-theta));
          } else {
            float sn, cs;
            sin_cos(theta, &sn, &cs);
            o = {z.re * cs + z.im * sn, z.im * cs - z.re * sn};
          }
          // slot of grid point n: one pad slot per chunk (the walls are zero)
          if (n > 0 && n < N - 1) tile[(2 * p + h) * LS + n + (n - 1) / CH] = o;
        }
      }
    });
    // the padding past the last unknown
    for (int q = threadIdx.x; q < 2 * np * (32 * CH + 2 - N); q += NT) {
      const int b = q / (32 * CH + 2 - N > 0 ? 32 * CH + 2 - N : 1), n = N - 1 + q - b * (32 * CH + 2 - N);
      tile[b * LS + n + (n - 1) / CH] = czero<float>();
    }
    __syncthreads();
    const Coef c = CnCoef<float, Coef>::make(a.cn_rf[2]);
    for (int b = threadIdx.x / kWarp; b < 2 * np; b += NT / kWarp)
      cn_line<float, Coef, CH, false, true>(tile + b * LS, 1, kWarp * CH, 0, tab, scan_s, c);
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * np * N; e += NT) {
      const int b = e / N, n = e - b * N;
      psi[e] = n > 0 && n < N - 1 ? tile[b * LS + n + (n - 1) / CH] : czero<float>();
    }
  }
}

// ---- set-up ---------------------------------------------------------------------------------
// The twiddles of both orders of the plan of length n (layout above), by sincospi in FP64.
__global__ inline void k_stage_twiddles(cplx<float> *tw, int n, int r1, int r2, int r3) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const bool rev = t >= n;
  int e = rev ? t - n : t;
  const int nst = r3 > 1 ? 3 : 2;
  const int p1 = rev ? (nst == 3 ? r3 : r2) : r1, p2 = rev ? (nst == 3 ? r2 : r1) : r2, p3 = nst == 3 ? (rev ? r1 : r3) : 1;
  int ns = p1, p = p2;
  if (e >= p1 * (p2 - 1)) {
    e -= p1 * (p2 - 1);
    ns = p1 * p2;
    p = p3;
    if (e >= ns * (p - 1)) return;
  }
  const int r = e / ns + 1, k = e % ns;
  double s, c;
  sincospi(2.0 * (double)(r * k) / (double)(ns * p), &s, &c);
  tw[t] = {(float)c, (float)-s};
}

// One translation unit's lengths: every kStageParts-th of the list.
constexpr int kStageParts = 8;
constexpr int st_index(int n) {
  int i = 0, at = -1;
#define DGPE_AT(m) \
  if (m == n) at = i; \
  ++i;
  DGPE_STAGE_ALL(DGPE_AT)
#undef DGPE_AT
  return at;
}

template <int PART>
struct StageLaunch {
  // f(integral_constant<N>) for the length n; false if it is not one of this part's
  template <typename F>
  static bool with(int n, F &&f) {
    switch (n) {
#define DGPE_CASE(m) \
  case m: \
    if constexpr (st_index(m) % kStageParts == PART) { \
      f(std::integral_constant<int, m>{}); \
      return true; \
    } \
    break;
      DGPE_STAGE_ALL(DGPE_CASE)
#undef DGPE_CASE
      default: break;
    }
    return false;
  }
  template <typename K>
  static void go(K k, dim3 g, int nt, size_t sm, const KArgs &a, const KArgs *ga, cudaStream_t st) {
    k<<<g, nt, sm, st>>>(a, ga);
  }
  static bool y(int dir, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
    return st_xy(a.ny) && with(a.ny, [&](auto len) {
      constexpr int N = st_xy(decltype(len)::value) ? decltype(len)::value : 12;
      using Y = StageY<N>;
      const dim3 g((a.nzh * a.nx + Y::L - 1) / Y::L, 1, members);
      if (dir < 0) k_ffty_st<-1, N><<<g, Y::NT, Y::smem, st>>>(a, ga);
      else k_ffty_st<+1, N><<<g, Y::NT, Y::smem, st>>>(a, ga);
    });
  }
  static bool x(const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
    return st_xy(a.nx) && with(a.nx, [&](auto len) {
      constexpr int N = st_xy(decltype(len)::value) ? decltype(len)::value : 12;
      using X = StageX<N>;
      const dim3 g((a.ny + X::B - 1) / X::B, a.nzh, members);
      k3_st<N><<<g, X::NT, X::smem, st>>>(a, ga);
    });
  }
  // K1 (which = kK1DensityR2Cz), K5's step (kK5C2RzPhaseCnz), the observables (kKObs) or Phi
  // (kKMaterialize)
  static bool z(int which, const KArgs &a, const KArgs *ga, unsigned members, cudaStream_t st) {
    bool done = false;
    with(a.nz, [&](auto len) {
      constexpr int N = decltype(len)::value;
      using Z = StageZ<N>;
      const dim3 g1((a.ny + 2 * Z::P1 - 1) / (2 * Z::P1), a.nx, members), g5((a.ny + 2 * Z::P5 - 1) / (2 * Z::P5), a.nx, members);
      done = true;
      if (which == kKObs) k5_st<N, float, kStObs><<<g5, Z::NT, Z::smem5, st>>>(a, ga);
      else if (which == kKMaterialize) k5_st<N, float, kStPhi><<<g5, Z::NT, Z::smem5, st>>>(a, ga);
      else if constexpr (Z::kOwn) {
        if (which == kK1DensityR2Cz) k1_st<N><<<g1, Z::NT, Z::smem1, st>>>(a, ga);
        else if (a.imag) k5_st<N, float, kStStep><<<g5, Z::NT, Z::smem5, st>>>(a, ga);
        else k5_st<N, cplx<float>, kStStep><<<g5, Z::NT, Z::smem5, st>>>(a, ga);
      } else {
        done = false;
      }
    });
    return done;
  }
  static cudaError_t init(int nx, int ny, int nz) {
    cudaError_t e = cudaSuccess;
    auto opt = [&](auto k, size_t sm) {
      // (48 KB less the reductions' static shared memory)
      if (e == cudaSuccess && sm > 40 * 1024) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    };
    with(nx, [&](auto len) {
      constexpr int N = decltype(len)::value;
      if constexpr (st_xy(N)) opt(k3_st<N>, StageX<N>::smem);
    });
    with(ny, [&](auto len) {
      constexpr int N = decltype(len)::value;
      if constexpr (st_xy(N)) {
        opt(k_ffty_st<-1, N>, StageY<N>::smem);
        opt(k_ffty_st<+1, N>, StageY<N>::smem);
      }
    });
    with(nz, [&](auto len) {
      using Z = StageZ<decltype(len)::value>;
      constexpr int N = decltype(len)::value;
      opt(k5_st<N, float, kStPhi>, Z::smem5);
      opt(k5_st<N, float, kStObs>, Z::smem5);
      if constexpr (Z::kOwn) {
        opt(k1_st<N>, Z::smem1);
        opt(k5_st<N, float, kStStep>, Z::smem5);
        opt(k5_st<N, cplx<float>, kStStep>, Z::smem5);
      }
    });
    return e;
  }
};

}  // namespace dgpe
