// unet_conv.cu -- the U-Net's 3x3x3 convolutions on the CUDA cores: FP32 networks, the first
// layer (one input channel) and the levels whose rows are no whole tensor-core tiles; the
// forward conv and, with flipped weights, the data gradient.
//
//     out[b][co][v] = bias[co] + sum_ci sum_tap W[co][ci][tap] in[b][ci][v + tap]
// (zero padding, optional ReLU), one FP32 chain per output in the order ci, dz, dy, dx.
//
// A thread holds 4 or 8 x voxels x 8 output channels; the accumulators of two channels are one
// packed pair, so an FFMA2 (fma.rn.f32x2: each half rounded as fmaf rounds) does two terms
// and a (row, 3 taps) step is 48 or 96 of them beside six 16-byte weight loads, two or three input
// loads and the packing of the inputs.  A CTA owns TY rows of CX voxels of one plane and 8 CG
// channels; the widths 8, 16 and 32 are chosen by what the level's rows leave unused.  Per
// input channel its three planes and its weights are staged once, the next channel's loads
// in flight in registers while the current one's FMAs run (two buffers, one barrier per
// channel).  Weights come straight from W: runs of 27 taps, transposed on the way to shared
// memory, so a network in use on several streams needs no shared scratch.
//
// Bound by the FMA pipe and the issue of its loads (64 -> 64 at 48x48x24: 165 us of FMAs).  The
// kernel before it had one tile width (32: a quarter of a 48-wide level's and three quarters of
// an 8-wide level's threads idle), scalar FMAs and nothing in flight while it staged: warm
// start at 192x192x96 2.92 -> 2.42 ms (its two 48x48x24 convs 0.87 -> 0.39), training step
// on 24 x 32^3 5.02 -> 4.13 ms (its four at 8^3), the first layer at 256x256x128 0.33 -> 0.23 ms.
#include "../../include/clamp.h"
#include "clamp_internal.cuh"
#include "clamp_kernels.cuh"
#include "packed.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace clamp {
namespace unet_cc {

// BF16 mode: an operand rounded to bfloat16 (round to nearest even) and widened back.
template <bool BF>
__device__ __forceinline__ float opnd(float x) {
  if constexpr (BF) return __bfloat162float(__float2bfloat16_rn(x));
  else return x;
}

// CX: x voxels of a tile, CG: groups of 8 output channels, VX: x voxels of a thread.
template <int CX, int CG, int VX>
struct CcCfg {
  static constexpr int TX = CX / VX, TY = CG == 2 ? 16 : CX == 32 && CG == 8 ? 4 : 8;
  static constexpr int THREADS = TX * TY * CG;
  static constexpr int COT = 8 * CG, WP = COT + 8;                 // channels, weight row pitch (conflict-free stores)
  static constexpr int IX = CX + 2, IY = TY + 2, IP = CX + 4;      // staged rows, row pitch (16-byte aligned rows)
  static constexpr int NIN = (3 * IY * IX + THREADS - 1) / THREADS;
  static constexpr int TPC = THREADS / COT, NW = (27 + TPC - 1) / TPC;   // threads per channel's weights, taps each
  static constexpr int MINB = (VX == 8 ? 384 : 512) / THREADS;      // 12 or 16 warps per SM: up to 168 or 128 registers
};

template <int CX, int CG, int VX, bool BF>
__global__ void __launch_bounds__(CcCfg<CX, CG, VX>::THREADS, CcCfg<CX, CG, VX>::MINB)
    k_conv3(const float* __restrict__ in, long long in_bs, int ci_n, float* __restrict__ out, long long out_bs,
            int co_n, const float* __restrict__ W, const float* __restrict__ bias, int relu, int nx, int ny, int nz,
            int vec) {
  using Cfg = CcCfg<CX, CG, VX>;
  constexpr int T = Cfg::THREADS, TX = Cfg::TX, TY = Cfg::TY, IX = Cfg::IX, IY = Cfg::IY, IP = Cfg::IP, WP = Cfg::WP;
  __shared__ __align__(16) float s_in[2][3 * IY * IP];
  __shared__ __align__(16) float s_w[2][27 * WP];
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = (tid / TX) % TY, cg = tid / (TX * TY);
  const int x0 = blockIdx.x * CX, y0 = blockIdx.y * TY;
  const int ncb = (co_n + Cfg::COT - 1) / Cfg::COT;
  const int zz = blockIdx.z / ncb, co0 = (int)(blockIdx.z % ncb) * Cfg::COT;
  const int b = zz / nz, z = zz % nz;
  const long long plane = (long long)nx * ny, n = plane * nz;

  // what this thread stages of a channel: voxels (offset from the tile's first, in[] valid) and weights
  const float* inb = in + (long long)b * in_bs + z * plane + (long long)y0 * nx + x0;
  int off[Cfg::NIN];
  unsigned valid = 0;
#pragma unroll
  for (int k = 0; k < Cfg::NIN; ++k) {
    const int e = tid + k * T, xi = e % IX - 1, yi = e / IX % IY - 1, zi = e / (IX * IY) - 1;
    const int gx = x0 + xi, gy = y0 + yi, gz = z + zi;
    const bool ok = e < 3 * IY * IX && gx >= 0 && gx < nx && gy >= 0 && gy < ny && gz >= 0 && gz < nz;
    off[k] = ok ? zi * (int)plane + yi * nx + xi : 0;
    valid |= (ok ? 1u : 0u) << k;
  }
  const int wco = tid / Cfg::TPC, wt0 = tid % Cfg::TPC;
  const bool wok = co0 + wco < co_n;
  const float* wsrc = W + (wok ? (long long)(co0 + wco) * ci_n * 27 : 0LL) + wt0;
  float vin[Cfg::NIN], vw[Cfg::NW];
  auto load = [&](int c) {
    const float* src = inb + c * n;
#pragma unroll
    for (int k = 0; k < Cfg::NIN; ++k) vin[k] = valid >> k & 1u ? __ldg(src + off[k]) : 0.f;
    const float* ws = wsrc + c * 27;
#pragma unroll
    for (int k = 0; k < Cfg::NW; ++k) vw[k] = wok && wt0 + k * Cfg::TPC < 27 ? __ldg(ws + k * Cfg::TPC) : 0.f;
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int k = 0; k < Cfg::NIN; ++k) {
      const int e = tid + k * T;
      if (e < 3 * IY * IX) s_in[buf][e + e / IX * (IP - IX)] = opnd<BF>(vin[k]);
    }
#pragma unroll
    for (int k = 0; k < Cfg::NW; ++k)
      if (wt0 + k * Cfg::TPC < 27) s_w[buf][(wt0 + k * Cfg::TPC) * WP + wco] = opnd<BF>(vw[k]);
  };

  f2 acc[VX][4];   // [x voxel][channel pair]
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int co = co0 + 8 * cg + 2 * p;
    const f2 bv = pack2(bias && co < co_n ? __ldg(&bias[co]) : 0.f, bias && co + 1 < co_n ? __ldg(&bias[co + 1]) : 0.f);
#pragma unroll
    for (int v = 0; v < VX; ++v) acc[v][p] = bv;
  }
  load(0);
  store(0);
  __syncthreads();
  for (int c = 0; c < ci_n; ++c) {
    const int buf = c & 1;
    if (c + 1 < ci_n) load(c + 1);
    const float* xs = s_in[buf] + ty * IP + VX * tx;
    const float* ws = s_w[buf] + 8 * cg;
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        const float* row = xs + (dz * IY + dy) * IP;
        f2 x[VX + 2];
#pragma unroll
        for (int q = 0; q < VX / 4; ++q) {
          const float4 xa = *reinterpret_cast<const float4*>(row + 4 * q);
          x[4 * q] = pack2(xa.x, xa.x), x[4 * q + 1] = pack2(xa.y, xa.y);
          x[4 * q + 2] = pack2(xa.z, xa.z), x[4 * q + 3] = pack2(xa.w, xa.w);
        }
        const float2 xb = *reinterpret_cast<const float2*>(row + VX);
        x[VX] = pack2(xb.x, xb.x), x[VX + 1] = pack2(xb.y, xb.y);
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const ulonglong2* wp = reinterpret_cast<const ulonglong2*>(ws + (dz * 9 + dy * 3 + dx) * WP);
          const ulonglong2 w0 = wp[0], w1 = wp[1];
          const f2 w[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int v = 0; v < VX; ++v) acc[v][p] = fma2(x[v + dx], w[p], acc[v][p]);
        }
      }
    }
    if (c + 1 < ci_n) store(buf ^ 1);   // the other buffer: its readers passed the last barrier
    __syncthreads();
  }
  const int gy = y0 + ty;
  if (gy >= ny) return;
  float* row = out + (long long)b * out_bs + z * plane + (long long)gy * nx;
#pragma unroll
  for (int q = 0; q < VX / 4; ++q) {
    const int gx = x0 + VX * tx + 4 * q;
    if (gx >= nx) continue;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      float2 r[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        r[v] = unpack2(acc[4 * q + v][p]);
        if (relu) r[v] = make_float2(fmaxf(r[v].x, 0.f), fmaxf(r[v].y, 0.f));
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int co = co0 + 8 * cg + 2 * p + h;
        if (co >= co_n) continue;
        const float o[4] = {h ? r[0].y : r[0].x, h ? r[1].y : r[1].x, h ? r[2].y : r[2].x, h ? r[3].y : r[3].x};
        float* oc = row + co * n + gx;
        if (vec) {
          *reinterpret_cast<float4*>(oc) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v)
            if (gx + v < nx) oc[v] = o[v];
        }
      }
    }
  }
}

template <int CX, int CG, int VX, bool BF>
static cudaError_t launch(const float* in, long long in_bs, int ci, float* out, long long out_bs, int co,
                          const float* W, const float* bias, bool relu, int B, int nx, int ny, int nz,
                          cudaStream_t st) {
  using Cfg = CcCfg<CX, CG, VX>;
  const int ncb = (co + Cfg::COT - 1) / Cfg::COT;
  // 16-byte stores: whole groups of four voxels in every row, aligned rows
  const int vec = nx % 4 == 0 && (uintptr_t)out % 16 == 0 && out_bs % 4 == 0;
  // grid.z = samples * nz * channel blocks must stay <= 65535: launch sample chunks
  const int per = std::max(1, 65535 / (nz * ncb));
  for (int b0 = 0; b0 < B; b0 += per) {
    const int bc = std::min(per, B - b0);
    const dim3 grid((nx + CX - 1) / CX, (ny + Cfg::TY - 1) / Cfg::TY, bc * nz * ncb);
    k_conv3<CX, CG, VX, BF><<<grid, Cfg::THREADS, 0, st>>>(in + (long long)b0 * in_bs, in_bs, ci,
                                                       out + (long long)b0 * out_bs, out_bs, co, W, bias, relu ? 1 : 0,
                                                       nx, ny, nz, vec);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int CX, int VX, bool BF, typename... A>
static cudaError_t by_channels(int co, A... a) {
  return co <= 16 ? launch<CX, 2, VX, BF>(a...) : co <= 32 ? launch<CX, 4, VX, BF>(a...) : launch<CX, 8, VX, BF>(a...);
}

// Eight voxels per thread where that leaves eight warps per SM: shared memory returns one float per
// lane and clock to the four schedulers together, and 8 x 8 sums take 5.6 FMAs per float loaded, 4 x 8
// only 3.2 (32 -> 64 and 64 -> 64 at 48x48x24 209 -> 194 us each in the mean, 1 -> 16 at 256x256x128 247 -> 230).
template <int CX, bool BF, typename... A>
static cudaError_t by_voxels(long long outputs, int co, A... a) {
  if (outputs / 64 >= 152LL * 8 * 32) return by_channels<CX, 8, BF>(co, a...);
  return by_channels<CX, 4, BF>(co, a...);
}

template <bool BF, typename... A>
static cudaError_t by_width(long long outputs, int nx, int ny, int co, A... a) {
  if (nx <= 8) return by_channels<8, 4, BF>(co, a...);
  // 16 wide where 32-wide tiles would leave half a tile unused, and above the height at which those of 4 rows
  // (64 channels) are more than a grid's y extent holds
  if ((nx + 15) / 16 % 2 || ny > 4 * 65535) return by_voxels<16, BF>(outputs, co, a...);
  return by_voxels<32, BF>(outputs, co, a...);
}

}  // namespace unet_cc

cudaError_t unet_conv3_cc(bool bf, const float* in, long long in_bs, int ci, float* out, long long out_bs, int co,
                          const float* W, const float* bias, bool relu, int B, int nx, int ny, int nz,
                          cudaStream_t st) {
  const long long outputs = (long long)B * nx * ny * nz * co;
  return bf ? unet_cc::by_width<true>(outputs, nx, ny, co, in, in_bs, ci, out, out_bs, co, W, bias, relu, B, nx, ny, nz, st)
            : unet_cc::by_width<false>(outputs, nx, ny, co, in, in_bs, ci, out, out_bs, co, W, bias, relu, B, nx, ny, nz, st);
}

}  // namespace clamp
