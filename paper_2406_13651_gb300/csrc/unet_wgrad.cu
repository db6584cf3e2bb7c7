// unet_wgrad.cu -- the U-Net's 3x3x3 weight gradients on the 5th-generation tensor cores
// (tcgen05) for BF16 networks:
//     dW[co][ci][tap] = sum over samples and voxels v of G[co][v] X[ci][v + tap],
// both operands rounded to bfloat16 as the CUDA-core kernel rounds them, FP32 sums.
//
// The GEMM's K is the voxels.  Channel-planar tensors with x fastest are K-major as they
// are, so staging is a rounding copy: eight x voxels of one channel are one 16-byte row of a
// no-swizzle core matrix, stored by one thread.  A tap's shift along y or z is then a whole
// number of rows, i.e. an offset of the operand's start; a shift along x would not start on
// a 16-byte row, so G is staged in three x-shifted copies (copy dx holds G[x - dx + 1]) and
// the copies are stacked along M:
//     M = 3 copies x 32 output channels (rows 32 dx + co; 16 channels leave half unused),
//     N = 3 dy x 16 input channels (X rows y, y + 1, y + 2 of the plane lie at one stride),
//     one accumulator per dz, all 27 taps of 16 x 16..32 channels from 3 MMAs per 16 voxels.
// A CTA owns one (output, input) channel chunk and marches along z through a span of
// (sample, y tile, x tile) columns with the three X planes it needs in shared memory, so
// every X and G plane is read and rounded once per chunk; the next step's loads are in
// flight in registers while the current step's MMAs run.
//
// The tensor core truncates its FP32 accumulator at every MMA (measured: a chain of S
// same-signed K = 16 steps loses about 2.5e-8 S of its value), so the sums are kept short:
//   * a step is 128 voxels, eight MMAs per accumulator;
//   * the planes of a pair share their accumulators, the second with G negated: after the first
//     the accumulator holds D1 = S1, after the second D2 = S1 - S2, and S1 + S2 = 2 D1 - D2 loses
//     S1's truncation and gains S2's, which are alike in neighbouring planes;
//   * each step's accumulators are added in FP32 (round to nearest) to sums in shared memory, and
//     the CTAs' sums pairwise in a fixed order by a second kernel.
// Against the FP64 sum of the same rounded operands (U-Net training at 2 x 16^3 .. 24 x 64x64x32,
// relative error of a layer's gradient): 4e-8 .. 9e-8, the CUDA cores' chains 3e-8 .. 1e-4.  With 256-voxel
// steps, each cleared, and atomics between the CTAs it was 7e-8 .. 3.4e-7, two to three times the
// CUDA cores' on small volumes.  The second kernel is also the faster: the ten layers at 24 x 32^3
// take 0.76 ms, 0.81 with atomics (0.66 with 256-voxel steps for 16 outputs, at 1.4e-7 .. 1.7e-7).
// Bound by a step's round (load, wait, take the sums, store, MMAs) at two CTAs per SM: 16 -> 16 at 24 x 32^3 takes
// 0.10 ms with the tensor pipe 12 % busy, issue slots 35 %, DRAM 1.0 TB/s.
#include "../../include/clamp.h"
#include "clamp_internal.cuh"
#include "clamp_kernels.cuh"
#include "packed.cuh"
#include "tc_core.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace clamp {
namespace unet_wg {

constexpr int WT = 256;   // threads per CTA
constexpr uint32_t kWaitLimit = 1u << 22;

// CO: output channels per CTA (16 or 32); NCG: groups of 8 input channels per CTA (1 or 2).
template <int CO, int NCG>
struct WgCfg {
  static constexpr int VOX = 128;                           // voxels (K) per step
  static constexpr int GS = VOX * 16;                       // bytes of one 8-channel group of a G copy
  static constexpr int A_BYTES = 12 * GS;                   // groups 4 dx + (co / 8)
  static constexpr int NCOL = NCG == 2 ? 48 : 32;           // N: (dy, ci); NCG = 1 has a fourth, unused dy
  static constexpr int TCOLS = NCG == 2 ? 256 : 128;        // 3 NCOL, rounded up to a power of two
  static constexpr int ACC = 3 * 3 * NCG * 8 * 3 * CO;      // FP32 sums: [dz][dy][ci][dx][co]
  // X plane: rows y0 - 1 .. y0 + R (and one the unused dy reads), [row][group][W / 8][8 channels][8 voxels]
  __host__ __device__ static int x_bytes(int w, int r) { return (r + 3) * NCG * w * 16; }
  static size_t smem(int w, int r) { return 1024 + A_BYTES + 3 * (size_t)x_bytes(w, r) + 4 * (size_t)ACC + 64; }
};

// Eight consecutive voxels p[0..7] of a row, zeros where x + i >= nx or !ok.
template <bool VEC>
__device__ __forceinline__ void load8(const float* __restrict__ p, int x, int nx, bool ok, float (&v)[8]) {
  if constexpr (VEC) {   // nx a multiple of 8 and 16-byte aligned rows
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (ok && x < nx) {
      a = __ldg(reinterpret_cast<const float4*>(p));
      b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    }
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ok && x + i < nx ? __ldg(p + i) : 0.f;
  }
}

template <int CO, int NCG, bool VEC>
__global__ void __launch_bounds__(WT, 2)
    k_wgrad3_tc(const float* __restrict__ in, long long in_bs, int ci_n, const float* __restrict__ G, long long g_bs,
                int co_n, float* __restrict__ part, int B, int nx, int ny, int nz, int lw, int* err) {
  using Cfg = WgCfg<CO, NCG>;
  constexpr int NCH = NCG * 8;
  const int W = 8 << lw, R = Cfg::VOX >> (3 + lw);   // tile: W x voxels in R rows of one plane
  const int S = W * 16;                              // bytes of one (row, group) of X
  extern __shared__ unsigned char wg_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)wg_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* s_a = base;                          // [12 groups][VOX / 8][8 channels] x 16 B
  unsigned char* s_x = base + Cfg::A_BYTES;           // 3 planes (plane z in slot z % 3)
  const int xb = Cfg::x_bytes(W, R);
  float* s_acc = reinterpret_cast<float*>(s_x + 3 * xb);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(s_acc + Cfg::ACC);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
  int* abort_flag = reinterpret_cast<int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int co0 = blockIdx.y * CO, ci0 = blockIdx.z * NCH;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int tx_n = (nx + W - 1) / W, ty_n = (ny + R - 1) / R;
  // this CTA's steps: whole pairs of planes of the (sample, y tile, x tile) columns
  const int zpairs = (nz + 1) / 2;
  const long long pairs = (long long)B * ty_n * tx_n * zpairs;
  auto first_step = [&](long long p) { return p / zpairs * nz + 2 * (p % zpairs); };
  const long long s_begin = first_step(pairs * blockIdx.x / gridDim.x), s_end = first_step(pairs * (blockIdx.x + 1) / gridDim.x);

  if (tid == 0) {
    tc::mbar_init(mbar, 1);
    *abort_flag = 0;
  }
  for (int e = tid; e < Cfg::ACC; e += WT) s_acc[e] = 0.f;
  if (warp == 0) {
    tc::tmem_alloc(tslot, Cfg::TCOLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = *tslot;
  const uint32_t a_s = tc::smem_addr(s_a), x_s = tc::smem_addr(s_x);

  // Staging tasks: one task is eight voxels of one channel; the channel varies fastest over
  // the threads, so a quarter-warp's 16-byte stores fill one 128-byte core matrix.
  constexpr int XT = ((Cfg::VOX / 8 + 8) * NCH + WT - 1) / WT;        // X tasks per thread: (R + 2) (W / 8) NCH, W <= 32
  constexpr int GT = (Cfg::VOX / 8) * CO / WT;                        // G tasks per thread
  static_assert((Cfg::VOX / 8) * CO % WT == 0, "G tasks");
  const int x_tasks = (R + 2) * NCH << lw;
  float xv[XT][8], gv[GT][8], gl[GT], gr[GT];
  int b = 0, x0 = 0, y0 = 0, z = 0;
  auto origin = [&](long long s) {
    z = (int)(s % nz);
    long long t = s / nz;
    x0 = (int)(t % tx_n) * W;
    t /= tx_n;
    y0 = (int)(t % ty_n) * R;
    b = (int)(t / ty_n);
  };
  auto load_x = [&](int zp) {
    const bool zin = zp >= 0 && zp < nz;
#pragma unroll
    for (int k = 0; k < XT; ++k) {
      const int t = tid + k * WT;
      const int c8 = t & 7, xg = (t >> 3) & ((1 << lw) - 1), rc = t >> (3 + lw), cg = rc % NCG, row = rc / NCG;
      const int c = ci0 + 8 * cg + c8, gy = y0 + row - 1, gx = x0 + 8 * xg;
      const bool ok = t < x_tasks && zin && c < ci_n && gy >= 0 && gy < ny;
      load8<VEC>(in + (ok ? (long long)b * in_bs + (long long)c * n + (long long)zp * plane + (long long)gy * nx + gx : 0LL),
                 gx, nx, ok, xv[k]);
    }
  };
  auto store_x = [&](int zp) {
    unsigned char* dst = s_x + ((zp + 3) % 3) * xb;
#pragma unroll
    for (int k = 0; k < XT; ++k) {
      const int t = tid + k * WT;
      if (t < x_tasks) {   // task order is the layout's order: [row][group][W / 8][8 channels]
        const float(&v)[8] = xv[k];
        reinterpret_cast<uint4*>(dst)[t] =
            make_uint4(bf16x2(v[0], v[1]), bf16x2(v[2], v[3]), bf16x2(v[4], v[5]), bf16x2(v[6], v[7]));
      }
    }
  };
  auto load_g = [&]() {
#pragma unroll
    for (int k = 0; k < GT; ++k) {
      const int t = tid + k * WT;
      const int c8 = t & 7, v8 = (t >> 3) % (Cfg::VOX / 8), cog = t / Cfg::VOX;
      const int xg = v8 & ((1 << lw) - 1), row = v8 >> lw;
      const int c = co0 + 8 * cog + c8, gy = y0 + row, gx = x0 + 8 * xg;
      const bool ok = c < co_n && gy < ny;
      const float* p = G + (ok ? (long long)b * g_bs + (long long)c * n + (long long)z * plane + (long long)gy * nx + gx : 0LL);
      load8<VEC>(p, gx, nx, ok, gv[k]);
      gl[k] = ok && gx > 0 && gx - 1 < nx ? __ldg(p - 1) : 0.f;
      gr[k] = ok && gx + 8 < nx ? __ldg(p + 8) : 0.f;
    }
  };
  auto store_g = [&](uint32_t neg) {   // neg: the sign bits of a pair, to store -G
#pragma unroll
    for (int k = 0; k < GT; ++k) {
      const int t = tid + k * WT;
      const int cog = t / Cfg::VOX, r = t % Cfg::VOX;   // r: [voxel group][8 channels]
      const float(&v)[8] = gv[k];
      uint4* d = reinterpret_cast<uint4*>(s_a + cog * Cfg::GS) + r;
      constexpr int DX = 4 * Cfg::GS / 16;
      auto pack = [&](float a, float b) { return bf16x2(a, b) ^ neg; };
      d[0] = make_uint4(pack(v[1], v[2]), pack(v[3], v[4]), pack(v[5], v[6]), pack(v[7], gr[k]));
      d[DX] = make_uint4(pack(v[0], v[1]), pack(v[2], v[3]), pack(v[4], v[5]), pack(v[6], v[7]));
      d[2 * DX] = make_uint4(pack(gl[k], v[0]), pack(v[1], v[2]), pack(v[3], v[4]), pack(v[5], v[6]));
    }
  };
  // A step's place: the first of a pair (planes z even and z + 1), the second, or alone.
  enum { ALONE, FIRST, SECOND };
  auto place = [&](int zs) { return zs & 1 ? SECOND : zs + 1 < nz ? FIRST : ALONE; };
  auto has = [&](int zs, int dz) { return zs + dz - 1 >= 0 && zs + dz - 1 < nz; };   // the X plane of dz exists
  // adds the finished step's accumulators (of the dz whose plane exists) to the FP32 sums; a sum that
  // is infinite after the first of a pair stays so
  auto flush = [&](int zf, int pl) {
    const int q = warp & 3, hh = warp >> 2;
    if (q == 3) return;   // rows 96..127 are unused
    constexpr int USED = 3 * NCH, BLKS = USED / 8, PER = (BLKS + 1) / 2;   // 8-column blocks per dz, per half
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
      if (!has(zf, dz)) continue;
      const float wt = pl == SECOND ? -1.f : pl == FIRST && has(zf + 1, dz) ? 2.f : 1.f;
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const int blk = hh * PER + j;
        if (blk >= BLKS) continue;
        float v[8];
        tc::tmem_ld_x8(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(dz * Cfg::NCOL + 8 * blk), v);
        if (lane < CO) {
          float* a = s_acc + ((dz * USED + 8 * blk) * 3 + q) * CO + lane;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float sum = a[i * 3 * CO];
            a[i * 3 * CO] = isinf(sum) && pl == SECOND ? sum : fmaf(wt, v[i], sum);
          }
        }
      }
    }
  };

  bool aborted = false;
  uint32_t phase = 0;
  int zprev = 0, plprev = ALONE;
  for (long long s = s_begin; s < s_end; ++s) {
    origin(s);
    const bool fresh = s == s_begin || z == 0;
    const int pl = place(z);
    load_g();
    load_x(z + 1);
    if (s > s_begin) {   // the previous step's MMAs: wait, then take their sums
      if (tid == 0 && !tc::mbar_wait_bounded(mbar, phase & 1u, kWaitLimit)) *abort_flag = 1;
      __syncthreads();
      if (*abort_flag) {
        aborted = true;
        break;
      }
      ++phase;
      tc::fence_after_sync();
      flush(zprev, plprev);
    }
    store_g(pl == SECOND ? 0x80008000u : 0u);
    store_x(z + 1);
    if (fresh) {
      load_x(z);
      store_x(z);
      load_x(z - 1);
      store_x(z - 1);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t idesc = tc::idesc_bf16_f32(128, Cfg::NCOL);
      const int rows = min(R, ny - y0);
      const int ks = (rows * W + 15) / 16;   // K steps; the last row pair of W = 8 may end on a zero row
      // rows of M groups GS apart, voxel groups 128 B apart; X: (dy, group) blocks S apart
      const uint64_t ad = tc::make_desc(a_s, 128, Cfg::GS);
      const uint32_t lbo_b = lw == 0 ? NCG * S : 128;
#pragma unroll
      for (int dz = 0; dz < 3; ++dz) {
        const int zp = z + dz - 1;
        if (!has(z, dz)) continue;
        const bool go_on = pl == SECOND && has(z - 1, dz);
        const uint64_t bd = tc::make_desc(x_s + ((zp + 3) % 3) * xb, lbo_b, S);
        for (int k = 0; k < ks; ++k) {
          const int row = (2 * k) >> lw, xg = (2 * k) & ((1 << lw) - 1);
          tc::mma_bf16(tbase + (uint32_t)(dz * Cfg::NCOL), ad + (uint64_t)(16 * k),
                       bd + (uint64_t)((row * NCG * S + xg * 128) >> 4), idesc, k > 0 || go_on ? 1u : 0u);
        }
      }
      tc::mma_commit(mbar);
    }
    zprev = z;
    plprev = pl;
  }
  if (!aborted && s_end > s_begin) {
    if (tid == 0 && !tc::mbar_wait_bounded(mbar, phase & 1u, kWaitLimit)) *abort_flag = 1;
    __syncthreads();
    aborted = *abort_flag != 0;
    tc::fence_after_sync();
    if (!aborted) flush(zprev, plprev);
  }
  if (aborted && tid == 0) {
    if (err) atomicOr(err, 2);
    tc::mbar_wait_bounded(mbar, phase & 1u, kWaitLimit);   // MMAs in flight, before TMEM is freed
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, Cfg::TCOLS);
  // this share's sums (zeros if a wait gave up), as they lie: [pair of channel chunks][share][ACC]
  float4* o = reinterpret_cast<float4*>(part + (((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * Cfg::ACC);
  static_assert(Cfg::ACC % 4 == 0, "whole 16-byte groups");
  for (int e = tid; e < Cfg::ACC / 4; e += WT)
    o[e] = aborted ? make_float4(0.f, 0.f, 0.f, 0.f) : reinterpret_cast<const float4*>(s_acc)[e];
}

// out[map(e)] = sum over the shares of part[share][e], always in the same order: eight threads per element
// take every eighth share, eight shares at a time pairwise.  Atomics added them one by one (rounding
// errors of about 2e-7 at 304 shares) and never twice in the same order.
constexpr int SH_G = 8;
template <class Map>
__global__ void __launch_bounds__(32 * SH_G) k_sum_shares(const float* __restrict__ part, int shares, int len,
                                                         float* __restrict__ out, Map map) {
  __shared__ float red[SH_G][32];
  const int lane = threadIdx.x % 32, gr = threadIdx.x / 32, e = blockIdx.x * 32 + lane;
  const float* p = part + (long long)blockIdx.y * shares * len + e;
  float acc = 0.f;
  if (e < len)
    for (int s0 = gr; s0 < shares; s0 += 8 * SH_G) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = s0 + k * SH_G < shares ? __ldg(p + (long long)(s0 + k * SH_G) * len) : 0.f;
      acc += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
  red[gr][lane] = acc;
  __syncthreads();
  if (gr != 0 || e >= len) return;
  float t[SH_G];
#pragma unroll
  for (int k = 0; k < SH_G; ++k) t[k] = red[k][lane];
  const long long i = map(blockIdx.y, e);
  if (i >= 0) out[i] = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
}

struct Identity {
  __device__ long long operator()(int, int e) const { return e; }
};
// Element e ([dz][dy][ci][dx][co]) of channel-chunk pair `pair` in dW[co][ci][27], or -1.
template <int CO, int NCH>
struct WgMap {
  int ci_n, co_n, co_chunks;
  __device__ long long operator()(int pair, int e) const {
    const int c = pair % co_chunks * CO + e % CO, dx = (e / CO) % 3, t = e / (3 * CO);
    const int ci = pair / co_chunks * NCH + t % NCH, dy = (t / NCH) % 3, dz = t / (3 * NCH);
    return c < co_n && ci < ci_n ? ((long long)c * ci_n + ci) * 27 + dz * 9 + dy * 3 + dx : -1;
  }
};

// Shares (CTAs per pair of channel chunks) of a layer: pairs of planes over two CTAs per SM.
template <int CO, int NCG>
static int wg_shares(int ci, int co, int B, int nx, int ny, int nz) {
  const int W = nx > 16 ? 32 : nx > 8 ? 16 : 8, R = WgCfg<CO, NCG>::VOX / W;
  const int chunks = ((co + CO - 1) / CO) * ((ci + NCG * 8 - 1) / (NCG * 8));
  const long long pairs = (long long)B * ((ny + R - 1) / R) * ((nx + W - 1) / W) * ((nz + 1) / 2);
  return (int)std::min(pairs, (long long)std::max(1, 2 * 152 / chunks));
}

template <int CO, int NCG>
static cudaError_t launch(const float* in, long long in_bs, int ci, const float* G, long long g_bs, int co, float* dW,
                          int B, int nx, int ny, int nz, float* part, int* err, cudaStream_t st) {
  using Cfg = WgCfg<CO, NCG>;
  const int lw = nx > 16 ? 2 : nx > 8 ? 1 : 0, W = 8 << lw, R = Cfg::VOX / W;
  const bool vec = nx % 8 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)G % 16 == 0 && in_bs % 4 == 0 && g_bs % 4 == 0;
  auto kern = vec ? k_wgrad3_tc<CO, NCG, true> : k_wgrad3_tc<CO, NCG, false>;
  const size_t smem = Cfg::smem(W, R);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int chunks_co = (co + CO - 1) / CO, chunks_ci = (ci + NCG * 8 - 1) / (NCG * 8);
  const int shares = wg_shares<CO, NCG>(ci, co, B, nx, ny, nz);
  kern<<<dim3(shares, chunks_co, chunks_ci), WT, smem, st>>>(in, in_bs, ci, G, g_bs, co, part, B, nx, ny, nz, lw, err);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const dim3 grid((Cfg::ACC + 31) / 32, chunks_co * chunks_ci);
  k_sum_shares<<<grid, 32 * SH_G, 0, st>>>(part, shares, Cfg::ACC, dW, WgMap<CO, NCG * 8>{ci, co, chunks_co});
  return cudaGetLastError();
}

template <int CO, int NCG>
static size_t part_floats(int ci, int co, int B, int nx, int ny, int nz) {
  return (size_t)wg_shares<CO, NCG>(ci, co, B, nx, ny, nz) * ((co + CO - 1) / CO) * ((ci + NCG * 8 - 1) / (NCG * 8)) *
         WgCfg<CO, NCG>::ACC;
}

}  // namespace unet_wg

cudaError_t unet_sum_shares(const float* part, int shares, int len, float* out, cudaStream_t st) {
  using namespace unet_wg;
  k_sum_shares<<<(len + 31) / 32, 32 * SH_G, 0, st>>>(part, shares, len, out, Identity{});
  return cudaGetLastError();
}

size_t unet_wgrad3_tc_part(int ci, int co, int B, int nx, int ny, int nz) {
  using namespace unet_wg;
  if (co <= 16) return ci <= 8 ? part_floats<16, 1>(ci, co, B, nx, ny, nz) : part_floats<16, 2>(ci, co, B, nx, ny, nz);
  return ci <= 8 ? part_floats<32, 1>(ci, co, B, nx, ny, nz) : part_floats<32, 2>(ci, co, B, nx, ny, nz);
}

cudaError_t unet_wgrad3_tc(const float* in, long long in_bs, int ci, const float* G, long long g_bs, int co, float* dW,
                           int B, int nx, int ny, int nz, float* part, int* err, cudaStream_t st) {
  using namespace unet_wg;
  if (co <= 16)
    return ci <= 8 ? launch<16, 1>(in, in_bs, ci, G, g_bs, co, dW, B, nx, ny, nz, part, err, st)
                   : launch<16, 2>(in, in_bs, ci, G, g_bs, co, dW, B, nx, ny, nz, part, err, st);
  return ci <= 8 ? launch<32, 1>(in, in_bs, ci, G, g_bs, co, dW, B, nx, ny, nz, part, err, st)
                 : launch<32, 2>(in, in_bs, ci, G, g_bs, co, dW, B, nx, ny, nz, part, err, st);
}

}  // namespace clamp
