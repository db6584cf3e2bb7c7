// band_agent.cu -- the forward agents' gradient on the aperture's support only.
//
// The gradient direction of Eq. (h-gradient) splits as
//     d = F^H [ a (y - a M) ] / sigma_w^2 - D mu,      M = F mu,
// because F^H F = I.  The bracket is zero wherever the aperture a is, so only the
// support of the lateral pupil (about 10 % of the (ky, kx) columns at a radius of 0.35
// Nyquist) ever needs the z and y transforms, and the x transform of a row only needs
// the band of kx columns the pupil touches.  The step size of Eq. (mu-update) needs
// ||A d||^2 = ||a F d||^2, again on the support only, and the next iteration's spectrum
// is M + gamma F d (F is linear), so F mu itself is formed once per call.
//
// Per look and iteration (state mu, r' in HBM; spectra on the support S = {(ky, kx):
// pupil != 0}, enumerated row by row; the band B = {kx: some pupil(ky, kx) != 0}):
//   P1 z pass on S   : M += gamma_prev F d_prev;  G = a (y - a M) / sigma_w^2;
//                      S4 = ||a y||^2;  inverse z-FFT of G              -> Gz [kz->z][S]
//   P2 y pass on B   : inverse y-FFT of Gz (zero off S)                 -> E  [z][y][B]
//   P3 x pass, rows  : e = inverse x-FFT of E (zero off B);  d = e - D mu -> d [z][y][x];
//                      S1 = ||d||^2, S3 = sum D |d|^2;  forward x-FFT of d, kept on B
//   P4 y pass on B   : forward y-FFT, kept on S                         -> [z][S]
//   P5 z pass on S   : forward z-FFT -> F d on S;  S2 = ||a F d||^2
// whose last CTA per look forms gamma = S1 / (S2 / sigma_w^2 + S3); then the elementwise pass C.  Only P3 touches
// every voxel: it reads mu, r' and writes d, plus two band rows.
#include "clamp_kernels.cuh"
#include "fft_reg.cuh"

#include <math.h>

#include <type_traits>

#include <vector>

namespace clamp {
namespace {

extern __shared__ float4 band_smem[];

constexpr int BC = 16;   // support / band columns per CTA in the y and z passes

__device__ __forceinline__ float warp_sum_b(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// FP32 per thread and warp, FP64 across the NTH / 32 warps in fixed order; writes out[k][idx].
template <int NTH, int NV>
__device__ __forceinline__ void block_sums(const float (&v)[NV], double* const (&out)[NV], long long idx) {
  constexpr int NW = (NTH + 31) / 32;
  __shared__ double red[NW][NV];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const float s = warp_sum_b(v[k]);
    if (lane == 0) red[warp][k] = (double)s;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double acc = 0.0;
    for (int w = 0; w < NW; ++w) acc += red[w][threadIdx.x];
    out[threadIdx.x][idx] = acc;
  }
}

// ---------------------------------------------------------------- support tables

// One CTA builds the tables of the support and the band from the pupil, in the order the
// host counted them (row by row, kx ascending; band columns by ascending kx).  The pupil is
// read once, a warp per row, into bit masks in shared memory; every position is then a count
// of mask bits.  Bound by trips to memory and the one SM's stores of the tables: 24 us at
// 256x256, 17 at 192x192 (118 and 66 where a thread walked its row or column, a chain of loads).
constexpr int MAXC = 256 / 32;   // 32-column words of a row
__global__ void __launch_bounds__(1024) k_band_tables(const float* __restrict__ pupil, int nx, int ny, BandTables t) {
  __shared__ unsigned s_mask[256][MAXC];
  __shared__ unsigned s_any[MAXC];        // columns any row of the support touches
  __shared__ int s_first[MAXC];           // band columns before a word
  __shared__ int s_rowstart[256];
  __shared__ int s_warp[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nc = (nx + 31) / 32;
  const unsigned below = (1u << lane) - 1u;
  if (tid < MAXC) s_any[tid] = 0;
  __syncthreads();
  for (int ky = warp; ky < ny; ky += 32) {
    float v[MAXC];
#pragma unroll
    for (int c = 0; c < MAXC; ++c) v[c] = 32 * c + lane < nx ? __ldg(&pupil[ky * nx + 32 * c + lane]) : 0.f;
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      const unsigned m = __ballot_sync(0xffffffffu, v[c] != 0.0f);
      if (lane == 0) {
        s_mask[ky][c] = m;
        if (m) atomicOr(&s_any[c], m);
      }
    }
  }
  __syncthreads();
  int incl = 0;   // support points of the rows up to this one (threads 0 .. ny - 1)
  if (tid < 256) {
    int cnt = 0;
    if (tid < ny)
#pragma unroll
      for (int c = 0; c < MAXC; ++c) cnt += __popc(s_mask[tid][c]);
    incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane == 31) s_warp[warp] = incl;
    incl -= cnt;
  }
  if (tid == 0) {
    int b = 0;
    for (int c = 0; c < MAXC; ++c) {
      s_first[c] = b;
      b += __popc(s_any[c]);
    }
  }
  __syncthreads();
  if (tid < 256) {
    for (int w = 0; w < warp; ++w) incl += s_warp[w];
    s_rowstart[tid] = incl;
  }
  if (tid < nx) {
    const unsigned any = s_any[tid >> 5];
    const int b = s_first[tid >> 5] + __popc(any & below);
    const bool in_band = any >> lane & 1u;
    t.bpos[tid] = in_band ? b : -1;
  }
  __syncthreads();
  for (int ky = warp; ky < ny; ky += 32) {
    int* row = t.sidx + (long long)ky * t.nbxp;
    int s0 = s_rowstart[ky];
    for (int c = 0; c < nc; ++c) {
      const unsigned m = s_mask[ky][c], any = s_any[c];
      const int kx = 32 * c + lane;
      const bool set = m >> lane & 1u;
      const int s = s0 + __popc(m & below);
      if (any >> lane & 1u) row[s_first[c] + __popc(any & below)] = set ? s : -1;
      if (set) {
        t.s_kykx[s] = ky * nx + kx;
        t.s_pup[s] = __ldg(&pupil[ky * nx + kx]);
      }
      s0 += __popc(m);
    }
    for (int b = t.nbx + lane; b < t.nbxp; b += 32) row[b] = -1;
  }
  for (int s = t.nS + tid; s < t.nSp; s += (int)blockDim.x) {   // padding columns: a = 0
    t.s_kykx[s] = 0;
    t.s_pup[s] = 0.0f;
  }
}

// ---------------------------------------------------------------- P1: z pass on the support (inverse)

template <int N>
__global__ void __launch_bounds__(RCol<N>::THREADS, RCol<N>::MINB) k_band_z_inv(BandArgs a, const float2* __restrict__ twB) {
  after_previous();
  [[maybe_unused]] const long long nL = (long long)a.L * a.n, sL = (long long)a.L * a.nz * a.t.nSp;   // buffer extents
  constexpr int R1 = RCol<N>::R1, R2 = RCol<N>::R2;
  float2* sm = reinterpret_cast<float2*>(band_smem);
  const int col = threadIdx.x % BC, j = threadIdx.x / BC;
  const int s = blockIdx.x * BC + col, l = blockIdx.y;
  const long long cbase = (long long)l * N * a.t.nSp + s;   // compact [l][kz][s]
  const float gp = a.gamma_prev ? a.gamma_prev[l] : 0.0f;
  const bool valid = s < a.t.nS;   // padding columns hold stale values: read as zero
  const bool step = valid && a.gamma_prev;
  const float pup = __ldg(&a.t.s_pup[s]);
  const long long ybase = (long long)l * a.n + __ldg(&a.t.s_kykx[s]);
  float2 u[R2], fv[R2];
#pragma unroll
  for (int r = 0; r < R2; ++r) {
    const long long ci = cbase + (long long)(j + r * R1) * a.t.nSp;
    u[r] = valid && CLAMP_IN_BOUNDS(ci, sL, 101) ? a.Ms[ci] : make_float2(0.f, 0.f);
    fv[r] = step && CLAMP_IN_BOUNDS(ci, sL, 102) ? a.Fd[ci] : make_float2(0.f, 0.f);
  }
  float2 yv[R2];
#pragma unroll
  for (int r = 0; r < R2; ++r) {
    const long long yi = ybase + (long long)(j + r * R1) * a.plane;
    yv[r] = CLAMP_IN_BOUNDS(yi, nL, 103) ? a.y[yi] : make_float2(0.f, 0.f);
  }
  float acc[1] = {0.f};
#pragma unroll
  for (int r = 0; r < R2; ++r) {
    float2 M = u[r];
    if (step) {   // the previous step's spectrum update M += gamma F d
      M.x = fmaf(gp, fv[r].x, M.x);
      M.y = fmaf(gp, fv[r].y, M.y);
      const long long mi = cbase + (long long)(j + r * R1) * a.t.nSp;
      if (CLAMP_IN_BOUNDS(mi, sL, 104)) a.Ms[mi] = M;
    }
    const float av = pup * __ldg(&a.window[j + r * R1]), f = av * a.inv_nv;
    u[r] = make_float2(f * fmaf(-av, M.x, yv[r].x), f * fmaf(-av, M.y, yv[r].y));
    acc[0] += av * av * cabs2(yv[r]);
  }
  rcol_first<N, true>(u, sm, col, j);
#pragma unroll
  for (int i = 0; i < RCol<N>::NB; ++i) {
    const int b = j + i * R1;
    if (R2 % R1 != 0 && b >= R2) continue;
    float2 v[R1];
    rcol_second<N, true>(v, sm, col, b, twB);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const long long fi = cbase + (long long)(b + r * R2) * a.t.nSp;
      if (CLAMP_IN_BOUNDS(fi, sL, 105)) a.Fd[fi] = cscale(v[r], a.sc_z);   // Gz, in place
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<unsigned*>(&a.mures[l]) = 0u;   // look_step's count
  double* const outs[1] = {a.s4};
  block_sums<RCol<N>::THREADS, 1>(acc, outs, (long long)l * gridDim.x + blockIdx.x);
}

// ---------------------------------------------------------------- P2 / P4: y passes on the band

// INV: Gz on the support -> E on the band (zero off the support).  !INV: band -> support.
template <int N, bool INV>
__global__ void __launch_bounds__(RCol<N>::THREADS, RCol<N>::MINB) k_band_y(BandArgs a, const float2* __restrict__ twB) {
  after_previous();
  [[maybe_unused]] const long long sL = (long long)a.L * a.nz * a.t.nSp,
                                   bL = (long long)a.L * a.nz * a.ny * a.t.nbxp;   // buffer extents
  constexpr int R1 = RCol<N>::R1, R2 = RCol<N>::R2;
  float2* sm = reinterpret_cast<float2*>(band_smem);
  const int col = threadIdx.x % BC, j = threadIdx.x / BC;
  const int bc = blockIdx.x * BC + col, z = blockIdx.y, l = blockIdx.z;
  const long long cplane = ((long long)l * a.nz + z) * a.t.nSp;               // compact [l][z][s]
  const long long bbase = (((long long)l * a.nz + z) * N) * a.t.nbxp + bc;    // band [l][z][y][b]
  float2 u[R2];
#pragma unroll
  for (int r = 0; r < R2; ++r) {
    const int yi = j + r * R1;
    if constexpr (INV) {
      const int s = __ldg(&a.t.sidx[yi * a.t.nbxp + bc]);
      u[r] = s >= 0 && CLAMP_IN_BOUNDS(cplane + s, sL, 111) ? a.Fd[cplane + s] : make_float2(0.f, 0.f);
    } else {
      const long long bi = bbase + (long long)yi * a.t.nbxp;
      u[r] = CLAMP_IN_BOUNDS(bi, bL, 112) ? a.band[bi] : make_float2(0.f, 0.f);
    }
  }
  rcol_first<N, INV>(u, sm, col, j);
#pragma unroll
  for (int i = 0; i < RCol<N>::NB; ++i) {
    const int b = j + i * R1;
    if (R2 % R1 != 0 && b >= R2) continue;
    float2 v[R1];
    rcol_second<N, INV>(v, sm, col, b, twB);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const int yi = b + r * R2;
      const float2 o = cscale(v[r], a.sc_y);
      if constexpr (INV) {
        const long long bi = bbase + (long long)yi * a.t.nbxp;
        if (CLAMP_IN_BOUNDS(bi, bL, 113)) a.band[bi] = o;
      } else {
        const int s = __ldg(&a.t.sidx[yi * a.t.nbxp + bc]);
        if (s >= 0 && CLAMP_IN_BOUNDS(cplane + s, sL, 114)) a.Fd[cplane + s] = o;
      }
    }
  }
}

// ---------------------------------------------------------------- P3: x pass over whole rows

enum BandRowMode { BAND_GRAD = 0, BAND_SPEC = 1 };

// BAND_GRAD: e = inverse x-FFT of the band row, d = e - D mu (written), S1/S3, forward x-FFT
// of d kept on the band.  BAND_SPEC: forward x-FFT of mu kept on the band (F mu's first axis).
// A row's threads hold its voxels in registers between the two transforms (fft_reg.cuh), each
// row within one warp: no block barrier, no tile staging.  Launch variant V = 0:
// rows_per_cta(N) rows per CTA, two CTAs per SM; V = 1: half as many rows and threads, four
// CTAs per SM (the same warps in smaller units); V = 2: mu and r' prefetched to L2 and read
// after the inverse transform, so no registers hold them across it and three CTAs share an SM.
// An iteration with V = 0, 1, 2 takes 56.1, 54.3, 57.3 us at 64x64x32 (L = 16), 269, 264, 285 at 128x128x64 (16), 537, 511,
// 558 at 192x192x96 (9) and 3.85, 3.79, 4.17 ms at 256x256x128 (32); the autotuner chooses, 0 without it.
template <int N, int V> struct RowCta {
  static constexpr int THREADS = V == 1 ? NT / 2 : NT, LINES = THREADS / RRow<N>::T, MINB = V == 0 ? 2 : V == 1 ? 4 : 3;
  static constexpr size_t SMEM = (size_t)LINES * RRow<N>::LS * sizeof(float2);
  static_assert(LINES == (V == 1 ? variant_rows(N, 2) : rows_per_cta(N)), "rows per CTA");
};

template <int N, int MODE, int V>
__global__ void __launch_bounds__(RowCta<N, V>::THREADS, RowCta<N, V>::MINB)
    k_band_x(BandArgs a, const float2* __restrict__ twA, const float2* __restrict__ twB) {
  after_previous();
  [[maybe_unused]] const long long nL = (long long)a.L * a.n, bL = (long long)a.L * a.nz * a.ny * a.t.nbxp;   // buffer extents
  constexpr int R1 = RRow<N>::R1, R2 = RRow<N>::R2, T = RRow<N>::T, LINES = RowCta<N, V>::LINES;
  constexpr bool LATE = V == 2 && MODE == BAND_GRAD;   // mu, r' read after the inverse transform
  const int line = threadIdx.x / T, j = threadIdx.x % T;
  float2* sl = reinterpret_cast<float2*>(band_smem) + line * RRow<N>::LS;
  const long long row0 = (long long)blockIdx.x * LINES;   // rows over [L][nz][ny]
  const long long row = row0 + line, e0 = row * N + j, b0 = row * a.t.nbxp;
  float2 mv[LATE ? 1 : R2];
  float rv[LATE ? 1 : R2];
  if constexpr (LATE) {   // the row's 128-byte lines of mu (8 B per element) and r' (4 B)
    for (int i = j; i < N / 16; i += T) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.mu + row * N + 16 * i));
    for (int i = j; i < N / 32; i += T) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.rprev + row * N + 32 * i));
  }
  if constexpr (!LATE) {
#pragma unroll
    for (int r = 0; r < R2; ++r) {
      mv[r] = CLAMP_IN_BOUNDS(e0 + r * R1, nL, 121) ? a.mu[e0 + r * R1] : make_float2(0.f, 0.f);
      if constexpr (MODE == BAND_GRAD) rv[r] = CLAMP_IN_BOUNDS(e0 + r * R1, nL, 122) ? a.rprev[e0 + r * R1] : 1.0f;
    }
  }
  float acc[2] = {0.f, 0.f};
  float2 u[R2];
  if constexpr (MODE == BAND_GRAD) {
#pragma unroll
    for (int i = 0; i < RRow<N>::NB; ++i) {
      const int b = j + i * T;
      if (R2 % T != 0 && b >= R2) continue;
      float2 v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) {
        const int bp = __ldg(&a.t.bpos[b + r * R2]);
        v[r] = bp >= 0 && CLAMP_IN_BOUNDS(b0 + bp, bL, 123) ? a.band[b0 + bp] : make_float2(0.f, 0.f);
      }
      rrow_inv_outer<N>(v, sl, b);
    }
    __syncwarp();
    rrow_inv_mid<N>(u, sl, j, twA);
#pragma unroll
    for (int r = 0; r < R2; ++r) {
      const long long e = e0 + r * R1;
      const bool ok = !LATE || CLAMP_IN_BOUNDS(e, nL, 124);
      const float2 m = LATE ? (ok ? a.mu[e] : make_float2(0.f, 0.f)) : mv[LATE ? 0 : r];
      const float D = __frcp_rn((LATE ? (ok ? a.rprev[e] : 1.0f) : rv[LATE ? 0 : r]) + a.floor);
      const float2 dv = make_float2(fmaf(-D, m.x, u[r].x * a.sc_x), fmaf(-D, m.y, u[r].y * a.sc_x));
      if (CLAMP_IN_BOUNDS(e, nL, 126)) a.d[e] = dv;
      const float d2 = cabs2(dv);
      acc[0] += d2;
      acc[1] += D * d2;
      u[r] = dv;
    }
    __syncwarp();   // the line's reads of the exchange are done
  } else {
#pragma unroll
    for (int r = 0; r < R2; ++r) u[r] = mv[LATE ? 0 : r];
  }
  rrow_fwd_mid<N>(u, sl, j);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < RRow<N>::NB; ++i) {
    const int b = j + i * T;
    if (R2 % T != 0 && b >= R2) continue;
    float2 v[R1];
    rrow_fwd_outer<N>(v, sl, b, twB);
#pragma unroll
    for (int r = 0; r < R1; ++r) {   // the band's padding columns stay as they are: nothing reads them
      const int bp = __ldg(&a.t.bpos[b + r * R2]);
      if (bp >= 0 && CLAMP_IN_BOUNDS(b0 + bp, bL, 127)) a.band[b0 + bp] = cscale(v[r], a.sc_x);
    }
  }
  if constexpr (MODE == BAND_GRAD) {
    double* const outs[2] = {a.s1, a.s3};
    const long long rows_per_look = (long long)a.nz * a.ny;
    const long long look = row0 / rows_per_look;
    block_sums<RowCta<N, V>::THREADS, 2>(acc, outs, look * a.px + (row0 - look * rows_per_look) / LINES);
  }
}

// ---------------------------------------------------------------- P5: z pass on the support (forward)

// gamma_l = S1 / (S2 / sigma_w^2 + S3) and the floored mu-residual sqrt(S1) / (sqrt(S4) / sigma_w^2) from
// the look's partial sums: by the last of the look's CTAs of the forward z pass (a kernel of its
// own cost a launch and 7 us on a small scene, where the passes are a chain of such latencies).
// The CTAs are counted in the look's mu-residual slot, which k_band_z_inv zeroes.
template <int NTH>
__device__ __forceinline__ void look_step(const BandArgs& a, int l, int pS) {
  constexpr int NW = (NTH + 31) / 32;
  __shared__ bool s_last;
  __shared__ double red[NW][4];
  unsigned* ticket = reinterpret_cast<unsigned*>(&a.mures[l]);
  if (threadIdx.x == 0) {   // this thread wrote the CTA's partial sum
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double v[4] = {0, 0, 0, 0};
  for (int i = threadIdx.x; i < a.px; i += NTH) {
    v[0] += __ldcg(&a.s1[(long long)l * a.px + i]);
    v[2] += __ldcg(&a.s3[(long long)l * a.px + i]);
  }
  for (int i = threadIdx.x; i < pS; i += NTH) {
    v[1] += __ldcg(&a.s2[(long long)l * pS + i]);
    v[3] += __ldcg(&a.s4[(long long)l * pS + i]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double S[4] = {0, 0, 0, 0};
  for (int w = 0; w < NW; ++w)
    for (int k = 0; k < 4; ++k) S[k] += red[w][k];
  const double den = S[1] / (double)a.nv + S[2];
  a.gamma[l] = den > 0 ? (float)(S[0] / den) : 0.0f;
  a.mures[l] = S[3] > 0 ? sqrt(S[0]) / (sqrt(S[3]) / (double)a.nv) : 0.0;
}

// BAND_GRAD: F d on the support (in place), S2 = ||a F d||^2 and the look's step.  BAND_SPEC: writes M.
template <int N, int MODE>
__global__ void __launch_bounds__(RCol<N>::THREADS, RCol<N>::MINB) k_band_z_fwd(BandArgs a, const float2* __restrict__ twB) {
  after_previous();
  [[maybe_unused]] const long long sL = (long long)a.L * a.nz * a.t.nSp;   // buffer extent
  constexpr int R1 = RCol<N>::R1, R2 = RCol<N>::R2;
  float2* sm = reinterpret_cast<float2*>(band_smem);
  const int col = threadIdx.x % BC, j = threadIdx.x / BC;
  const int s = blockIdx.x * BC + col, l = blockIdx.y;
  const long long cbase = (long long)l * N * a.t.nSp + s;
  const bool valid = s < a.t.nS;
  float2 u[R2];
#pragma unroll
  for (int r = 0; r < R2; ++r) {
    const long long fi = cbase + (long long)(j + r * R1) * a.t.nSp;
    u[r] = valid && CLAMP_IN_BOUNDS(fi, sL, 131) ? a.Fd[fi] : make_float2(0.f, 0.f);
  }
  rcol_first<N, false>(u, sm, col, j);
  float acc[1] = {0.f};
#pragma unroll
  for (int i = 0; i < RCol<N>::NB; ++i) {
    const int b = j + i * R1;
    if (R2 % R1 != 0 && b >= R2) continue;
    float2 v[R1];
    rcol_second<N, false>(v, sm, col, b, twB);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const int kz = b + r * R2;
      const float2 o = cscale(v[r], a.sc_z);
      const long long ci = cbase + (long long)kz * a.t.nSp;
      if constexpr (MODE == BAND_GRAD) {
        if (CLAMP_IN_BOUNDS(ci, sL, 132)) a.Fd[ci] = o;
        const float av = __ldg(&a.t.s_pup[s]) * __ldg(&a.window[kz]);
        acc[0] += av * av * cabs2(o);
      } else {
        if (CLAMP_IN_BOUNDS(ci, sL, 133)) a.Ms[ci] = o;
      }
    }
  }
  if constexpr (MODE == BAND_GRAD) {
    double* const outs[1] = {a.s2};
    block_sums<RCol<N>::THREADS, 1>(acc, outs, (long long)l * gridDim.x + blockIdx.x);
    look_step<RCol<N>::THREADS>(a, l, gridDim.x);
  }
}

template <class F>
cudaError_t dispatch_n(int N, F&& f) {
  switch (N) {
    case 8: return f(std::integral_constant<int, 8>{});
    case 16: return f(std::integral_constant<int, 16>{});
    case 32: return f(std::integral_constant<int, 32>{});
    case 64: return f(std::integral_constant<int, 64>{});
    case 96: return f(std::integral_constant<int, 96>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 192: return f(std::integral_constant<int, 192>{});
    case 256: return f(std::integral_constant<int, 256>{});
    default: return cudaErrorInvalidValue;
  }
}

#define BAND_TRY(x)                   \
  do {                                \
    cudaError_t _e = (x);             \
    if (_e != cudaSuccess) return _e; \
  } while (0)

cudaError_t run_z(const BandArgs& a, int L, bool inverse, int mode, cudaStream_t st) {
  return dispatch_n(a.nz, [&](auto NC) -> cudaError_t {
    constexpr int N = decltype(NC)::value, TH = RCol<N>::THREADS;
    constexpr size_t smem = RCol<N>::SMEM;   // at most 33 KB: within the default limit
    const dim3 grid(a.t.nSp / BC, L);
    if (inverse) return launch_after(k_band_z_inv<N>, grid, TH, smem, st, a, twiddle_table_b(N));
    if (mode == BAND_GRAD) return launch_after(k_band_z_fwd<N, BAND_GRAD>, grid, TH, smem, st, a, twiddle_table_b(N));
    return launch_after(k_band_z_fwd<N, BAND_SPEC>, grid, TH, smem, st, a, twiddle_table_b(N));
  });
}

cudaError_t run_y(const BandArgs& a, int L, bool inverse, cudaStream_t st) {
  return dispatch_n(a.ny, [&](auto NC) -> cudaError_t {
    constexpr int N = decltype(NC)::value, TH = RCol<N>::THREADS;
    constexpr size_t smem = RCol<N>::SMEM;
    const dim3 grid(a.t.nbxp / BC, a.nz, L);
    if (inverse) return launch_after(k_band_y<N, true>, grid, TH, smem, st, a, twiddle_table_b(N));
    return launch_after(k_band_y<N, false>, grid, TH, smem, st, a, twiddle_table_b(N));
  });
}

template <int N, int MODE, int V>
cudaError_t launch_x(const BandArgs& a, int L, cudaStream_t st) {
  using Cta = RowCta<N, V>;
  static_assert(Cta::SMEM <= 48 * 1024, "default shared-memory limit");
  const unsigned grid = (unsigned)((long long)L * a.nz * a.ny / Cta::LINES);
  return launch_after(k_band_x<N, MODE, V>, grid, Cta::THREADS, Cta::SMEM, st, a, twiddle_table_a(N), twiddle_table_b(N));
}

cudaError_t run_x(const BandArgs& a, int L, int mode, int variant, cudaStream_t st) {
  return dispatch_n(a.nx, [&](auto NC) -> cudaError_t {
    constexpr int N = decltype(NC)::value;
    if constexpr (N < 16) {   // nx is a multiple of 16
      return cudaErrorInvalidValue;
    } else {
      if (mode == BAND_SPEC) return launch_x<N, BAND_SPEC, 0>(a, L, st);
      if (variant == 1) return launch_x<N, BAND_GRAD, 1>(a, L, st);
      if (variant == 2) return launch_x<N, BAND_GRAD, 2>(a, L, st);
      return launch_x<N, BAND_GRAD, 0>(a, L, st);
    }
  });
}

}  // namespace

// One pass along the rows, eight columns at a time (independent sums, so the loop vectorises): the GPU
// waits meanwhile.  A chain of additions and a second, column-wise walk took about 100 us at
// 192x192, an eighth of a caller's iteration there.
BandShape band_shape(const float* pupil_host, int nx, int ny, double* sum_sq) {
  BandShape b{};
  constexpr int K = 8;
  std::vector<int> any(nx, 0);
  double s[K] = {};
  int cnt[K] = {};
  for (int ky = 0; ky < ny; ++ky) {
    const float* row = pupil_host + (size_t)ky * nx;
    int kx = 0;
    for (; kx + K <= nx; kx += K)
      for (int j = 0; j < K; ++j) {
        const float v = row[kx + j];
        const int set = v != 0.0f;
        s[j] += (double)v * v;
        cnt[j] += set;
        any[kx + j] |= set;
      }
    for (; kx < nx; ++kx) {
      s[0] += (double)row[kx] * row[kx];
      cnt[0] += row[kx] != 0.0f;
      any[kx] |= row[kx] != 0.0f;
    }
  }
  int nS = 0, nbx = 0;
  double sum = 0;
  for (int j = 0; j < K; ++j) {
    nS += cnt[j];
    sum += s[j];
  }
  for (int kx = 0; kx < nx; ++kx) nbx += any[kx];
  *sum_sq = sum;
  b.nS = nS;
  b.nSp = (nS + BC - 1) / BC * BC;
  b.nbx = nbx;
  b.nbxp = (nbx + BC - 1) / BC * BC;
  return b;
}

size_t band_table_bytes(const BandShape& b, int nx, int ny) {
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  return al(sizeof(int) * (size_t)ny * b.nbxp) + al(sizeof(int) * (size_t)b.nSp) + al(sizeof(float) * (size_t)b.nSp) +
         al(sizeof(int) * (size_t)nx);
}

BandTables band_tables_at(const BandShape& b, int nx, int ny, void* base) {
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  char* p = static_cast<char*>(base);
  BandTables t{};
  t.nS = b.nS;
  t.nSp = b.nSp;
  t.nbx = b.nbx;
  t.nbxp = b.nbxp;
  t.sidx = reinterpret_cast<int*>(p);
  p += al(sizeof(int) * (size_t)ny * b.nbxp);
  t.s_kykx = reinterpret_cast<int*>(p);
  p += al(sizeof(int) * (size_t)b.nSp);
  t.s_pup = reinterpret_cast<float*>(p);
  p += al(sizeof(float) * (size_t)b.nSp);
  t.bpos = reinterpret_cast<int*>(p);
  return t;
}

int band_px(int nx, int ny, int nz, int x_variant) {
  return (int)((long long)nz * ny / (x_variant == 1 ? variant_rows(nx, 2) : rows_per_cta(nx)));
}

cudaError_t launch_band_tables(const float* pupil, int nx, int ny, const BandTables& t, cudaStream_t st) {
  k_band_tables<<<1, 1024, 0, st>>>(pupil, nx, ny, t);
  return cudaGetLastError();
}

cudaError_t launch_band_spectrum(const BandArgs& a0, int L, cudaStream_t st) {
  BandArgs a = a0;
  a.L = L;
  BAND_TRY(run_x(a, L, BAND_SPEC, 0, st));
  BAND_TRY(run_y(a, L, false, st));
  return run_z(a, L, false, BAND_SPEC, st);
}

cudaError_t launch_band_agent(const BandArgs& a, int L, float nv, float* gamma, double* mures, int x_variant,
                              cudaStream_t st) {
  BandArgs b = a;
  b.L = L;
  b.px = band_px(a.nx, a.ny, a.nz, x_variant);
  b.nv = nv;
  b.gamma = gamma;
  b.mures = mures;
  BAND_TRY(run_z(b, L, true, BAND_GRAD, st));
  BAND_TRY(run_y(b, L, true, st));
  BAND_TRY(run_x(b, L, BAND_GRAD, x_variant, st));
  BAND_TRY(run_y(b, L, false, st));
  return run_z(b, L, false, BAND_GRAD, st);
}

cudaError_t bounds_site_band(unsigned int* site, bool reset) { return bounds_site_local(site, reset); }

}  // namespace clamp
