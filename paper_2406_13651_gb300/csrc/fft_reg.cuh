// fft_reg.cuh -- two-stage FFTs held in registers, with one exchange through shared memory.
//
// A line of N = R1 * R2 points belongs to R1 threads.  In the middle of a transform pair
// thread j holds the R2 points j + R1 r: exactly what the last stage of an inverse transform
// (radix R2 after radix R1) leaves and the first stage of a forward one (radix R2, then R1)
// takes, and 8 R1 bytes apart in steps of one per thread, so these points are loaded from
// and stored to global memory directly.  The outer stages are R2 butterflies of radix R1 over
// the points b + R2 r.  A transform therefore writes and reads shared memory once, where the
// tile FFT of fft_core.cuh (any radix plan, whole tiles) does so once per stage and again on
// entry and exit.
//
// Stage twiddles come from two tables per length, [r][k] so that a warp's loads are
// consecutive: A (second stage after radix R1): w^(r k) at r R1 + k; B (after radix R2): w^(r k)
// at r R2 + k.
#pragma once
#include "fft_core.cuh"

namespace clamp {

// R1 = threads per line, R2 = points per thread.
template <int N> struct RPlan;
template <> struct RPlan<8>   { static constexpr int R1 = 2,  R2 = 4; };
template <> struct RPlan<16>  { static constexpr int R1 = 4,  R2 = 4; };
template <> struct RPlan<32>  { static constexpr int R1 = 4,  R2 = 8; };
template <> struct RPlan<64>  { static constexpr int R1 = 8,  R2 = 8; };
template <> struct RPlan<96>  { static constexpr int R1 = 8,  R2 = 12; };
template <> struct RPlan<128> { static constexpr int R1 = 8,  R2 = 16; };
template <> struct RPlan<192> { static constexpr int R1 = 16, R2 = 12; };
template <> struct RPlan<256> { static constexpr int R1 = 16, R2 = 16; };
// The first radix of table A, for the host.
constexpr int rplan_r1(int N) { return N == 8 ? 2 : N <= 32 ? 4 : N <= 128 ? 8 : 16; }

// In-register DFT of 12 points (3 x 4): Y[i2][k1] = DFT3 over i1 of x[4 i1 + i2], times w12^(i2 k1),
// X[k1 + 3 k2] = DFT4 over i2.  Other radices: dft of fft_core.cuh.
template <bool INV>
__device__ __forceinline__ float2 w12mul(float2 x, int m) {
  constexpr float H = 0.86602540378443865f;   // sin(pi/3)
  float c, s;   // W = c - i s (forward), c + i s (inverse)
  switch (m) {
    case 0: return x;
    case 1: c = H; s = 0.5f; break;
    case 2: c = 0.5f; s = H; break;
    case 3: return INV ? make_float2(-x.y, x.x) : make_float2(x.y, -x.x);
    case 4: c = -0.5f; s = H; break;
    default: return make_float2(-x.x, -x.y);   // 6
  }
  if (INV) s = -s;
  return make_float2(fmaf(x.x, c, x.y * s), fmaf(x.y, c, -x.x * s));
}

template <int R, bool INV>
__device__ __forceinline__ void rdft(float2 (&v)[R]) {
  if constexpr (R == 12) {
    float2 y[4][3];
#pragma unroll
    for (int i2 = 0; i2 < 4; ++i2) {
      float2 t[3] = {v[i2], v[4 + i2], v[8 + i2]};
      dft<3, INV>(t);
#pragma unroll
      for (int k1 = 0; k1 < 3; ++k1) y[i2][k1] = w12mul<INV>(t[k1], i2 * k1);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      float2 t[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      dft<4, INV>(t);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 3 * k2] = t[k2];
    }
  } else {
    dft<R, INV>(v);
  }
}

// v[r] *= w^(r k) (conjugate for the inverse): tw points at the table's column k, rows `ld` apart.
template <int R, bool INV>
__device__ __forceinline__ void rtwiddle(float2 (&v)[R], const float2* __restrict__ tw, int ld) {
#pragma unroll
  for (int r = 1; r < R; ++r) {
    const float2 w = __ldg(&tw[r * ld]);
    v[r] = INV ? cmulc(v[r], w) : cmul(v[r], w);
  }
}

// ---- rows: the R1 threads of a line are neighbours in a warp, so the exchange needs only
// __syncwarp.  Shared memory per line: N points, one pad after every butterfly (odd strides),
// and a line stride that puts the lines of a half-warp in different banks.
template <int N>
struct RRow {
  static constexpr int R1 = RPlan<N>::R1, R2 = RPlan<N>::R2, T = R1;
  static constexpr int MAXP = R1 > R2 ? R1 : R2;
  static constexpr int LS0 = N + MAXP;
  // line stride: T (mod 16) points, so that 16 / T lines of a half-warp do not collide
  static constexpr int LS = T >= 16 ? LS0 : LS0 + ((T - LS0 % 16) % 16 + 16) % 16;
  static constexpr int NB = (R2 + T - 1) / T;   // outer butterflies per thread (the last ones may idle)
};

// Inverse, first stage: butterfly b (points b + R2 r in v) to shared memory.
template <int N>
__device__ __forceinline__ void rrow_inv_outer(float2 (&v)[RPlan<N>::R1], float2* sl, int b) {
  constexpr int R1 = RPlan<N>::R1;
  rdft<R1, true>(v);
#pragma unroll
  for (int r = 0; r < R1; ++r) sl[b * (R1 + 1) + r] = v[r];
}
// Inverse, second stage: points j + R1 r into u (natural order).
template <int N>
__device__ __forceinline__ void rrow_inv_mid(float2 (&u)[RPlan<N>::R2], const float2* sl, int j,
                                             const float2* __restrict__ twA) {
  constexpr int R1 = RPlan<N>::R1, R2 = RPlan<N>::R2;
#pragma unroll
  for (int r = 0; r < R2; ++r) u[r] = sl[j + r * (R1 + 1)];
  rtwiddle<R2, true>(u, twA + j, R1);
  rdft<R2, true>(u);
}
// Forward, first stage: points j + R1 r (in u) to shared memory.
template <int N>
__device__ __forceinline__ void rrow_fwd_mid(float2 (&u)[RPlan<N>::R2], float2* sl, int j) {
  constexpr int R2 = RPlan<N>::R2;
  rdft<R2, false>(u);
#pragma unroll
  for (int r = 0; r < R2; ++r) sl[j * (R2 + 1) + r] = u[r];
}
// Forward, second stage: butterfly b, points b + R2 r into v.
template <int N>
__device__ __forceinline__ void rrow_fwd_outer(float2 (&v)[RPlan<N>::R1], const float2* sl, int b,
                                               const float2* __restrict__ twB) {
  constexpr int R1 = RPlan<N>::R1, R2 = RPlan<N>::R2;
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = sl[b + r * (R2 + 1)];
  rtwiddle<R1, false>(v, twB + b, R2);
  rdft<R1, false>(v);
}

// ---- columns: a CTA of 16 R1 threads transforms 16 adjacent lines, thread (line = t % 16,
// j = t / 16), first radix R2: points j + R1 r of the thread's line go in, the points
// b + R2 r of the butterflies b = j, j + R1, ... < R2 come out.  One barrier.
constexpr int RCOLS = 16;
template <int N> struct RCol {
  static constexpr int R1 = RPlan<N>::R1, R2 = RPlan<N>::R2, THREADS = RCOLS * R1, LD = N + 1;
  static constexpr int NB = (R2 + R1 - 1) / R1;   // output butterflies per thread
  static constexpr int MINB = 512 / THREADS;      // 16 warps per SM: up to 128 registers
  static constexpr size_t SMEM = (size_t)RCOLS * LD * sizeof(float2);
};

// First stage and exchange: u holds points j + R1 r.  Ends with the barrier.
template <int N, bool INV>
__device__ __forceinline__ void rcol_first(float2 (&u)[RPlan<N>::R2], float2* sm, int line, int j) {
  constexpr int R2 = RPlan<N>::R2;
  rdft<R2, INV>(u);
#pragma unroll
  for (int r = 0; r < R2; ++r) sm[line * RCol<N>::LD + j * R2 + r] = u[r];
  __syncthreads();
}
// Second stage: butterfly b, points b + R2 r into v.
template <int N, bool INV>
__device__ __forceinline__ void rcol_second(float2 (&v)[RPlan<N>::R1], const float2* sm, int line, int b,
                                            const float2* __restrict__ twB) {
  constexpr int R1 = RPlan<N>::R1, R2 = RPlan<N>::R2;
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = sm[line * RCol<N>::LD + b + r * R2];
  rtwiddle<R1, INV>(v, twB + b, R2);
  rdft<R1, INV>(v);
}

}  // namespace clamp
