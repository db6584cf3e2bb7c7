// unet.cu -- the learned warm start: a 3-level 3D U-Net (encoder: two 3x3x3 conv + ReLU
// per level and 2^3 max-pooling; decoder: 2^3 stride-2 transposed conv, concatenation
// with the encoder skip, two 3x3x3 conv + ReLU; a final 1x1x1 conv), trained on the
// GPU with these forward and backward kernels and Adam (FP32).
//
// Tensors are channel-planar per sample: [B][C][nz][ny][nx].  A concatenation buffer
// holds the decoder's upsampled channels first and the encoder skip after them, so the
// skip's conv writes straight into it (no copy).
#include "../../include/clamp.h"
#include "clamp_internal.cuh"
#include "clamp_kernels.cuh"
#include "exact_sum.cuh"
#include "packed.cuh"

#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <cstring>
#include <vector>

namespace clamp {
namespace unet {

constexpr int UT = 256;

// BF16 mode: an operand rounded to bfloat16 (round to nearest even) and widened back.
__device__ __forceinline__ float opr(float x, int bf) {
  return bf ? __bfloat162float(__float2bfloat16_rn(x)) : x;
}

enum LayerKind { CONV3 = 0, TCONV = 1, CONV1 = 2 };
struct Layer {
  int kind, ci, co;
  int level;    // its volume is the input's divided by this along every axis
  size_t w, b;  // offsets (floats) into the parameter buffer
  size_t nw;    // weight count
};

// Tensor-core path of a network (BF16 only): packed-weight scratch, error word, switch.
struct TcCtx {
  uint4* wpk;
  int* err;
  bool on;
};

static cudaError_t conv3(bool bf, const float* in, long long in_bs, int ci, float* out, long long out_bs, int co,
                         const float* W, const float* bias, bool relu, int B, int nx, int ny, int nz, cudaStream_t st,
                         const TcCtx& tc) {
  if (bf && tc.on && unet_conv3_tc_supported(ci, co, nx, ny))
    return unet_conv3_tc(in, in_bs, ci, out, out_bs, co, W, bias, relu, B, nx, ny, nz, tc.wpk, tc.err, st);
  return unet_conv3_cc(bf, in, in_bs, ci, out, out_bs, co, W, bias, relu, B, nx, ny, nz, st);
}

// W'[ci][co][26 - tap] = W[co][ci][tap]: the dgrad of a 3x3x3 conv is the conv of the output
// gradient with these weights.
__global__ void k_flip(const float* __restrict__ W, float* __restrict__ Wf, int ci_n, int co_n) {
  const int total = ci_n * co_n * 27;
  for (int e = blockIdx.x * UT + threadIdx.x; e < total; e += gridDim.x * UT) {
    const int tap = e % 27, ci = (e / 27) % ci_n, co = e / (27 * ci_n);
    Wf[((long long)ci * co_n + co) * 27 + (26 - tap)] = W[e];
  }
}

// dW[co][ci][tap] += sum_{b, v} G[b][co][v] in[b][ci][v + tap] on the CUDA cores: one FP32 chain
// per (co, ci, tap) and share of the volume, in voxel order over the share's (sample, plane,
// 4-row) chunks; atomics combine the shares.  A CTA takes CIC input channels and COB output
// channels: a consumer warp per input channel, lane = (output channel, half of the taps), 14
// chains per lane in registers.  The x taps come from a window that slides along the row,
// so four voxels cost six 16-byte shared loads and 56 FMAs, where a thread per chain paid
// two loads per FMA (16 -> 16 at 24 x 64x64x32: 12.3 -> 1.46 ms).  Producer warps stage the next
// chunk meanwhile (two buffers where they fit).  Bound by the one consumer warp per scheduler: of its
// instructions per four voxels 56 are FMAs, and it waits for six 16-byte loads (32 -> 16 at 24 x 32^3: FMA
// pipe 42 % busy, issue slots 72 %, shared memory 0.42 wavefronts a clock).  Two chains to an FFMA2 on
// rows staged in pairs was no faster (1.46 -> 1.45 to 1.78 ms).
constexpr int WG_CO = 16, WG_ROWS = 4, WG_NT = 512;
__host__ __device__ constexpr int wg_pitch(int nx) { return (nx + 3) / 4 * 4 + 8; }   // 4 zeros left, >= 4 right
__host__ __device__ constexpr int wg_gstride(int nx) { return (WG_ROWS * ((nx + 3) / 4 * 4) + 31) / 32 * 32 + 4; }
static size_t wg_buf_floats(int cic, int cob, int nx) {
  return (size_t)3 * (WG_ROWS + 2) * cic * wg_pitch(nx) + (size_t)cob * wg_gstride(nx) + 4;
}

template <int CIC, int COB, bool VEC>
__global__ void __launch_bounds__(WG_NT) k_wgrad3(const float* __restrict__ in, long long in_bs, int ci_n,
                                                  const float* __restrict__ G, long long g_bs, int co_n,
                                                  float* __restrict__ dW, int B, int nx, int ny, int nz, int bf,
                                                  int nbuf) {
  extern __shared__ __align__(16) float wg_sm[];
  constexpr int XR = 3 * (WG_ROWS + 2);   // X rows per channel: [dz][row]
  const int nq = (nx + 3) / 4, pitch = wg_pitch(nx), gs = wg_gstride(nx);
  const int buf_floats = XR * CIC * pitch + COB * gs + 4;   // 4: the look-ahead's last read
  const int ci0 = blockIdx.y * CIC, cob = blockIdx.z * COB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int row_blocks = (ny + WG_ROWS - 1) / WG_ROWS;
  const long long chunks = (long long)B * nz * row_blocks;
  for (int e = threadIdx.x; e < nbuf * buf_floats; e += (int)blockDim.x) wg_sm[e] = 0.f;   // halo columns stay zero
  __syncthreads();

  // Where each staged row comes from and goes: {channel, offset of the row from the chunk's first
  // voxel, offset in the buffer, what must lie inside the volume: bits of X rows 0..5, planes
  // 8..10, G rows 16..19; bit 31: no such channel}.
  constexpr int ROWS = XR * CIC + COB * WG_ROWS, UN = 6;
  __shared__ int4 s_row[ROWS];
  for (int r = threadIdx.x; r < ROWS; r += (int)blockDim.x) {
    const int f = r - XR * CIC;
    if (f < 0) {   // X row [channel][dz][row]
      const int row = r % (WG_ROWS + 2), dz = (r / (WG_ROWS + 2)) % 3, c = r / XR;
      s_row[r] = make_int4(c, (int)((dz - 1) * plane) + (row - 1) * nx, r * pitch + 4,
                           ci0 + c < ci_n ? (1 << row) | (1 << (8 + dz)) : (int)0x80000000);
    } else {       // G row [output channel][row]
      const int o = f / WG_ROWS, row = f % WG_ROWS;
      s_row[r] = make_int4(o, row * nx, XR * CIC * pitch + o * gs + row * nq * 4,
                           cob + o < co_n ? 1 << (16 + row) : (int)0x80000000);
    }
  }
  __syncthreads();

  // Threads 0 <= t < nt stage chunk ch into buffer `to`: groups of 2^lq threads along a row's
  // quads, six rows' loads in flight per thread.
  const int lq = nq > 16 ? 5 : nq > 8 ? 4 : nq > 4 ? 3 : 2;
  auto stage = [&](long long ch, float* to, int t, int nt) {
    const int rb = (int)(ch % row_blocks), z = (int)((ch / row_blocks) % nz), b = (int)(ch / ((long long)row_blocks * nz));
    const int y0 = rb * WG_ROWS, q0 = t & ((1 << lq) - 1), rstep = nt >> lq;
    const long long v0 = z * plane + (long long)y0 * nx;
    const float* xb = in + b * in_bs + (long long)ci0 * n + v0;
    const float* gb = G + b * g_bs + (long long)cob * n + v0;
    int inside = (z > 0 ? 1 << 8 : 0) | 1 << 9 | (z + 1 < nz ? 1 << 10 : 0);
#pragma unroll
    for (int r = 0; r < WG_ROWS + 2; ++r) {
      const int gy = y0 + r - 1;
      if (gy >= 0 && gy < ny) inside |= 1 << r;
      if (r < WG_ROWS && y0 + r < ny) inside |= 1 << (16 + r);
    }
    for (int q = q0; q < nq; q += 1 << lq) {
      for (int r0 = t >> lq; r0 < ROWS; r0 += UN * rstep) {
        float4 v[UN];
        int dst[UN];
#pragma unroll
        for (int k = 0; k < UN; ++k) {
          const int r = r0 + k * rstep;
          v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          dst[k] = -1;
          if (r >= ROWS) continue;
          const int4 e = s_row[r];
          dst[k] = e.z;
          if ((e.w & inside) != e.w) continue;
          const float* src = (r < XR * CIC ? xb : gb) + e.x * n + e.y;
          if constexpr (VEC) {
            v[k] = __ldg(reinterpret_cast<const float4*>(src) + q);
          } else {
            v[k].x = __ldg(src + 4 * q);
            if (4 * q + 1 < nx) v[k].y = __ldg(src + 4 * q + 1);
            if (4 * q + 2 < nx) v[k].z = __ldg(src + 4 * q + 2);
            if (4 * q + 3 < nx) v[k].w = __ldg(src + 4 * q + 3);
          }
        }
#pragma unroll
        for (int k = 0; k < UN; ++k)
          if (dst[k] >= 0)
            reinterpret_cast<float4*>(to + dst[k])[q] =
                make_float4(opr(v[k].x, bf), opr(v[k].y, bf), opr(v[k].z, bf), opr(v[k].w, bf));
      }
    }
  };

  // lane (co, h): taps 0..13 (h = 0) or 13..26 (h = 1); COB = 8 leaves half the lanes idle.  Rows of three taps each, and the
  // middle row (dz, dy) = (1, 1), whose taps 0, 1 or 1, 2 the lane takes.
  const int co = lane % COB, h = lane >> 4;
  float acc[14];
#pragma unroll
  for (int j = 0; j < 14; ++j) acc[j] = 0.f;
  auto consume = [&](const float* buf) {
    const float* xc = buf + warp * XR * pitch;
    const float* gc = buf + XR * CIC * pitch + co * gs;
#pragma unroll 1
    for (int r = 0; r < WG_ROWS; ++r) {
      const float4* row[5];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int t = h ? k + 5 : k;   // row index 3 dz + dy
        row[k] = reinterpret_cast<const float4*>(xc + ((t / 3) * (WG_ROWS + 2) + r + t % 3) * pitch);
      }
      row[4] = reinterpret_cast<const float4*>(xc + ((WG_ROWS + 2) + r + 1) * pitch);
      const float4* g4 = reinterpret_cast<const float4*>(gc) + r * nq;
      // window of voxels 4 q - 1 .. 4 q + 4 per row: pw, cur, nxt.x; the loads run one quad ahead
      float pw[5];
      float4 cur[5], nxt[5], g = g4[0];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        pw[k] = row[k][0].w;
        cur[k] = row[k][1];
        nxt[k] = row[k][2];
      }
#pragma unroll 3
      for (int q = 0; q < nq; ++q) {   // the last quad's look-ahead reads past its row, unused
        const float4 gn = g4[q + 1];
        float4 ahead[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) ahead[k] = row[k][q + 3];
        const float gv[4] = {g.x, g.y, g.z, g.w};
        float w[5][6];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const float u[6] = {pw[k], cur[k].x, cur[k].y, cur[k].z, cur[k].w, nxt[k].x};
#pragma unroll
          for (int i = 0; i < 6; ++i) w[k][i] = u[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {   // voxel by voxel: 14 independent FMAs at a time
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[3 * k + d] = fmaf(gv[i], w[k][i + d], acc[3 * k + d]);
#pragma unroll
          for (int d = 0; d < 2; ++d) acc[12 + d] = fmaf(gv[i], h ? w[4][i + d + 1] : w[4][i + d], acc[12 + d]);
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          pw[k] = cur[k].w;
          cur[k] = nxt[k];
          nxt[k] = ahead[k];
        }
        g = gn;
      }
    }
  };

  // two buffers: warps 4.. stage chunk i + 1 while warps 0..3 consume chunk i; one buffer: in turn
  const bool consumer = warp < CIC, producer = warp >= 4;
  const int nt = (int)blockDim.x;
  const int pt = nbuf == 2 ? (int)threadIdx.x - 128 : (int)threadIdx.x, pn = nbuf == 2 ? nt - 128 : nt;
  if (nbuf == 2) {
    if (producer && (long long)blockIdx.x < chunks) stage(blockIdx.x, wg_sm, pt, pn);
    __syncthreads();
    int cur = 0;
    for (long long ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
      if (producer) {
        if (ch + gridDim.x < chunks) stage(ch + gridDim.x, wg_sm + (cur ^ 1) * buf_floats, pt, pn);
      } else if (consumer) {
        consume(wg_sm + cur * buf_floats);
      }
      __syncthreads();
      cur ^= 1;
    }
  } else {
    for (long long ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
      stage(ch, wg_sm, pt, pn);
      __syncthreads();
      if (consumer) consume(wg_sm);
      __syncthreads();
    }
  }
  if (consumer && ci0 + warp < ci_n && cob + co < co_n && (lane & 15) < COB) {
    float* d = dW + ((long long)(cob + co) * ci_n + ci0 + warp) * 27;
#pragma unroll
    for (int j = 0; j < 12; ++j) atomicAdd(&d[h ? j + 15 : j], acc[j]);
    if (!h) atomicAdd(&d[12], acc[12]);
    atomicAdd(&d[h ? 14 : 13], acc[13]);   // tap 13 is in both halves: the first keeps it
  }
}

// Shares of the volume per (input channel, 16 output channels): the length of a chain.
static long long wgrad3_shares(int ci, int co, int B, int ny, int nz) {
  const long long chunks = (long long)B * nz * ((ny + WG_ROWS - 1) / WG_ROWS);
  const long long rest = (long long)ci * ((co + WG_CO - 1) / WG_CO);
  return std::max(1LL, std::min(chunks, (4LL * 152 + rest - 1) / rest));
}

static cudaError_t wgrad3(const float* in, long long in_bs, int ci, const float* G, long long g_bs, int co, float* dW,
                          int B, int nx, int ny, int nz, int bf, cudaStream_t st) {
  constexpr size_t kMax = 224 * 1024;   // beside the row table
  const bool wide = wg_buf_floats(4, 16, nx) * 4 > kMax;   // rows above about 400 voxels: one channel by eight
  const int cic = wide ? 1 : 4, cob = wide ? 8 : 16;
  const size_t buf = wg_buf_floats(cic, cob, nx) * 4;
  const int nbuf = 2 * buf <= kMax ? 2 : 1;
  const size_t smem = nbuf * buf;
  const bool vec = nx % 4 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)G % 16 == 0 && in_bs % 4 == 0 && g_bs % 4 == 0;
  auto kern = wide ? (vec ? k_wgrad3<1, 8, true> : k_wgrad3<1, 8, false>) : (vec ? k_wgrad3<4, 16, true> : k_wgrad3<4, 16, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)wgrad3_shares(ci, co, B, ny, nz), (ci + cic - 1) / cic, (co + cob - 1) / cob);
  // one CTA per SM keeps twelve producer warps; more CTAs than SMs run two to an SM with four each
  const int nt = (long long)grid.x * grid.y * grid.z > 152 ? 256 : WG_NT;
  kern<<<grid, nt, smem, st>>>(in, in_bs, ci, G, g_bs, co, dW, B, nx, ny, nz, bf, nbuf);
  return cudaGetLastError();
}

// Sum over the CTA's threads of v, valid in thread 0 (FP32 within warps, FP32 across them).
__device__ __forceinline__ float block_sum(float v) {
  __shared__ float red[UT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
  if (threadIdx.x == 0)
    for (int w = 0; w < UT / 32; ++w) s += red[w];
  return s;
}

// Grid of the per-channel reductions below: RC_PER float4 (or values) per thread along a
// channel plane in x, channels in y, samples in z.  A one-CTA-per-channel reduction leaves
// 120 to 136 of 152 SMs idle at 16 to 32 channels (3.1 ms for a 0.2 GB tensor at
// 24 x 64x64x32); here every CTA sums one chunk of a plane into `part`, [channel][sample][chunk], and
// one launch at the end of the backward pass adds those of every layer in a fixed order.
constexpr int RC_PER = 4;
static dim3 chan_grid(long long n, int C, int B) {
  const long long units = n % 4 == 0 ? n / 4 : n;
  return dim3((unsigned)((units + UT * RC_PER - 1) / (UT * RC_PER)), C, std::min(B, 65535));
}
static long long chan_parts(long long n, int B) {   // partial sums per channel
  const dim3 g = chan_grid(n, 1, B);
  return (long long)g.x * g.z;
}
__device__ __forceinline__ long long chan_part(int c) {   // this CTA's
  return ((long long)c * gridDim.z + blockIdx.z) * gridDim.x + blockIdx.x;
}

// The sums to take at the end: out[c] = sum of part[c][0 .. per - 1].
struct ChanSums {
  static constexpr int MAX = 14;
  int n = 0, channels[MAX];
  long long per[MAX];
  const float* part[MAX];
  float* out[MAX];
  float* next;   // free scratch
  float* add(float* o, int C, long long vox, int B) {
    float* r = next;
    out[n] = o;
    channels[n] = C;
    per[n] = chan_parts(vox, B);
    part[n] = r;
    next += C * per[n++];
    return r;
  }
};
__global__ void __launch_bounds__(UT) k_chan_sums(ChanSums t) {   // a CTA per channel of every entry
  int k = 0, c = blockIdx.x;
  while (c >= t.channels[k]) c -= t.channels[k++];
  const float* p = t.part[k] + c * t.per[k];
  float acc = 0.f;
  for (long long i = threadIdx.x; i < t.per[k]; i += UT) acc += __ldg(p + i);
  acc = block_sum(acc);
  if (threadIdx.x == 0) t.out[k][c] = acc;
}
static cudaError_t chan_sums(const ChanSums& t, cudaStream_t st) {
  int total = 0;
  for (int k = 0; k < t.n; ++k) total += t.channels[k];
  k_chan_sums<<<total, UT, 0, st>>>(t);
  return cudaGetLastError();
}

// g <- g * (y > 0) for a ReLU output y (MASK; sample strides allow concat views) and
// db[c] = sum_{b, v} g[b][c][v], in one pass (partial sums into part).
template <bool MASK, bool VEC>
__global__ void __launch_bounds__(UT) k_relu_bias_grad(float* __restrict__ g, long long g_bs,
                                                       const float* __restrict__ y, long long y_bs, int B,
                                                       long long n, float* __restrict__ part) {
  const int c = blockIdx.y;
  const long long units = VEC ? n / 4 : n;
  const long long u0 = (long long)blockIdx.x * (UT * RC_PER) + threadIdx.x;
  float acc = 0.f;
  for (int b = blockIdx.z; b < B; b += gridDim.z) {
    float* gp = g + b * g_bs + (long long)c * n;
    const float* yp = MASK ? y + b * y_bs + (long long)c * n : nullptr;
#pragma unroll
    for (int k = 0; k < RC_PER; ++k) {
      const long long u = u0 + k * UT;
      if (u >= units) continue;
      if constexpr (VEC) {
        float4 v = reinterpret_cast<const float4*>(gp)[u];
        if constexpr (MASK) {
          const float4 m = reinterpret_cast<const float4*>(yp)[u];
          v = make_float4(m.x > 0.f ? v.x : 0.f, m.y > 0.f ? v.y : 0.f, m.z > 0.f ? v.z : 0.f, m.w > 0.f ? v.w : 0.f);
          reinterpret_cast<float4*>(gp)[u] = v;
        }
        acc += (v.x + v.y) + (v.z + v.w);
      } else {
        float v = gp[u];
        if constexpr (MASK) {
          v = yp[u] > 0.f ? v : 0.f;
          gp[u] = v;
        }
        acc += v;
      }
    }
  }
  const float s = block_sum(acc);
  if (threadIdx.x == 0) part[chan_part(c)] = s;
}

template <bool MASK>
static cudaError_t relu_bias_grad(float* g, long long g_bs, const float* y, long long y_bs, int C, int B, long long n,
                                  float* db, ChanSums& sums, cudaStream_t st) {
  float* part = sums.add(db, C, n, B);
  if (n % 4 == 0)
    k_relu_bias_grad<MASK, true><<<chan_grid(n, C, B), UT, 0, st>>>(g, g_bs, y, y_bs, B, n, part);
  else
    k_relu_bias_grad<MASK, false><<<chan_grid(n, C, B), UT, 0, st>>>(g, g_bs, y, y_bs, B, n, part);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- pooling, transposed conv, 1x1 conv

// Grid of the pooling kernels: output (y, x) planes along x, output z along y, (sample,
// channel) pairs along z (strided above 65535), so no thread divides 64-bit indices.
static dim3 pool_grid(int nx, int ny, int nz, int C, int B) {
  return dim3((unsigned)(((nx / 2) * (ny / 2) + UT - 1) / UT), nz / 2, (unsigned)std::min((long long)B * C, 65535LL));
}

// 2^3 max-pool: out[b][c][v] over the 8 children of v; arg[] keeps which child won (the first
// of equal ones).  The two children along x are one 8-byte load (nx is even).
__global__ void __launch_bounds__(UT) k_pool_fwd(const float* __restrict__ in, long long in_bs, float* __restrict__ out,
                                                 unsigned char* __restrict__ arg, int C, int B, int nx, int ny, int nz) {
  const int ox = nx / 2, oy = ny / 2, oz = nz / 2;
  const int i = (int)(blockIdx.x * UT + threadIdx.x);
  if (i >= ox * oy) return;
  const int x = i % ox, y = i / ox, z = blockIdx.y;
  const long long n = (long long)nx * ny * nz, on = (long long)ox * oy * oz, plane = (long long)nx * ny;
  for (int bc = blockIdx.z; bc < B * C; bc += gridDim.z) {
    const float* src = in + (long long)(bc / C) * in_bs + (long long)(bc % C) * n + 2 * z * plane + (long long)(2 * y) * nx + 2 * x;
    float2 v[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) v[d] = __ldg(reinterpret_cast<const float2*>(src + (d >> 1) * plane + (d & 1) * nx));
    float best = -INFINITY;
    int bi = 0;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const float val = d & 1 ? v[d >> 1].y : v[d >> 1].x;
      if (val > best) {
        best = val;
        bi = d;
      }
    }
    const long long o = (long long)bc * on + (long long)z * ox * oy + i;
    out[o] = best;
    arg[o] = (unsigned char)bi;
  }
}

// din[child] += dout for the winning child of every pooled voxel (children are disjoint).
__global__ void __launch_bounds__(UT) k_pool_bwd(const float* __restrict__ dout, const unsigned char* __restrict__ arg,
                                                 float* __restrict__ din, long long din_bs, int C, int B, int nx, int ny,
                                                 int nz) {
  const int ox = nx / 2, oy = ny / 2, oz = nz / 2;
  const int i = (int)(blockIdx.x * UT + threadIdx.x);
  if (i >= ox * oy) return;
  const int x = i % ox, y = i / ox, z = blockIdx.y;
  const long long n = (long long)nx * ny * nz, on = (long long)ox * oy * oz, plane = (long long)nx * ny;
  for (int bc = blockIdx.z; bc < B * C; bc += gridDim.z) {
    const long long o = (long long)bc * on + (long long)z * ox * oy + i;
    const int d = arg[o];
    din[(long long)(bc / C) * din_bs + (long long)(bc % C) * n + (2 * z + (d >> 2)) * plane +
        (long long)(2 * y + ((d >> 1) & 1)) * nx + 2 * x + (d & 1)] += dout[o];
  }
}

// Transposed conv, kernel 2^3, stride 2: out[b][co][2v + d] = bias[co] + sum_ci W[ci][co][d] in[b][ci][v].
// (nx, ny, nz) are the OUTPUT dimensions.  A CTA keeps the weights of 16 output channels in shared
// memory and walks runs of 64 VPT input voxels; a thread makes the 8 children of VPT voxels for
// 4 output channels, two children to an FFMA2 (fma.rn.f32x2: each half rounded as fmaf rounds), so
// eight 16-byte weight loads feed 32 VPT multiply-adds.  The next run's inputs are on their
// way (cp.async, two buffers where they fit) while this one's are used.  Bound by the
// multiply-adds and the output's stores: 32 -> 16 at 256x256x128 115 us of FMAs, 99 us of HBM; 434 us
// with one voxel per thread, scalar FMAs and nothing in flight, now 321 (64 -> 32 at half size 213 ->
// 158); the stores of a run wait for its last multiply-add.
constexpr int TF_CO = 16;
static size_t tconv_fwd_smem(int ci, int vpt, int nbuf) { return sizeof(float) * (size_t)ci * (TF_CO * 8 + nbuf * 64 * vpt); }
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <int VPT>
__global__ void __launch_bounds__(UT, 2) k_tconv_fwd(const float* __restrict__ in, int ci_n, float* __restrict__ out, long long out_bs,
                                                     int co_n, const float* __restrict__ W, const float* __restrict__ bias, int B,
                                                     int nx, int ny, int nz, int bf, int nbuf, int vec) {
  constexpr int V = 64 * VPT;
  extern __shared__ __align__(16) float tf_sm[];
  float* s_w = tf_sm;                       // [ci][TF_CO][8]
  float* s_x = tf_sm + ci_n * TF_CO * 8;    // [nbuf][ci][V]
  const int ix = nx / 2, iy = ny / 2, iz = nz / 2, in_n = ix * iy * iz;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int co0 = blockIdx.y * TF_CO, per_b = (in_n + V - 1) / V;
  const long long runs = (long long)B * per_b;
  for (int e = threadIdx.x; e < ci_n * TF_CO * 8; e += UT) {
    const int d = e % 8, co = (e / 8) % TF_CO, ci = e / (8 * TF_CO);
    s_w[e] = co0 + co < co_n ? opr(__ldg(&W[((long long)ci * co_n + co0 + co) * 8 + d]), bf) : 0.f;
  }
  auto stage = [&](long long r, float* to) {   // voxels past the sample's end are left as they are: not used
    const int b = (int)(r / per_b), v0 = (int)(r % per_b) * V;
    const float* src = in + (long long)b * ci_n * in_n + v0;
    if (vec) {   // in_n a multiple of four, 16-byte aligned
      for (int e = threadIdx.x; e < ci_n * (V / 4); e += UT) {
        const int c = e / (V / 4), q = 4 * (e % (V / 4));
        if (v0 + q < in_n) cp_async16(to + c * V + q, src + (long long)c * in_n + q);
      }
    } else {
      for (int e = threadIdx.x; e < ci_n * V; e += UT)
        if (v0 + e % V < in_n) cp_async4(to + e, src + (long long)(e / V) * in_n + e % V);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int vi = threadIdx.x % 64, cog = threadIdx.x / 64;   // this thread's voxels vi + 64 k of the run, its 4 channels
  float bv[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bv[j] = co0 + 4 * cog + j < co_n ? __ldg(&bias[co0 + 4 * cog + j]) : 0.f;
  int cur = 0;
  if (blockIdx.x < runs) stage(blockIdx.x, s_x);
  for (long long r = blockIdx.x; r < runs; r += gridDim.x) {
    const bool more = r + gridDim.x < runs;
    if (nbuf == 2 && more) {
      stage(r + gridDim.x, s_x + (cur ^ 1) * ci_n * V);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    unsigned long long acc[VPT][4][4];   // [voxel][channel][pair of children]
#pragma unroll
    for (int k = 0; k < VPT; ++k)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[k][j][q] = pack2(bv[j], bv[j]);
    const float* xs = s_x + cur * ci_n * V + vi;
#pragma unroll 2
    for (int ci = 0; ci < ci_n; ++ci) {
      unsigned long long x[VPT];
#pragma unroll
      for (int k = 0; k < VPT; ++k) {
        const float xv = opr(xs[ci * V + 64 * k], bf);
        x[k] = pack2(xv, xv);
      }
      const ulonglong2* w = reinterpret_cast<const ulonglong2*>(s_w + (ci * TF_CO + 4 * cog) * 8);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const ulonglong2 w0 = w[2 * j], w1 = w[2 * j + 1];
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
          acc[k][j][0] = fma2(w0.x, x[k], acc[k][j][0]);
          acc[k][j][1] = fma2(w0.y, x[k], acc[k][j][1]);
          acc[k][j][2] = fma2(w1.x, x[k], acc[k][j][2]);
          acc[k][j][3] = fma2(w1.y, x[k], acc[k][j][3]);
        }
      }
    }
    __syncthreads();   // this buffer's readers are done
    if (nbuf == 2) cur ^= 1;
    else if (more) stage(r + gridDim.x, s_x);
    const int b = (int)(r / per_b), v0 = (int)(r % per_b) * V;
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
      const int v = v0 + vi + 64 * k;
      if (v >= in_n) continue;
      const int x = v % ix, y = (v / ix) % iy, z = v / (ix * iy);
      float* o = out + (long long)b * out_bs + (long long)(co0 + 4 * cog) * n + 2 * z * plane + (long long)(2 * y) * nx + 2 * x;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (co0 + 4 * cog + j >= co_n) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float2*>(o + j * n + (q >> 1) * plane + (q & 1) * nx) = unpack2(acc[k][j][q]);
      }
    }
  }
}

static cudaError_t tconv_fwd(const float* in, int ci, float* out, long long out_bs, int co, const float* W, const float* bias,
                             int B, int nx, int ny, int nz, int bf, cudaStream_t st) {
  // two voxels per thread in two buffers where two CTAs fit an SM, else one voxel and one buffer
  const bool two = 2 * (tconv_fwd_smem(ci, 2, 2) + 1024) <= 227 * 1024;
  const int vpt = two ? 2 : 1, nbuf = two ? 2 : 1;
  auto kern = two ? k_tconv_fwd<2> : k_tconv_fwd<1>;
  const size_t smem = tconv_fwd_smem(ci, vpt, nbuf);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long in_n = (long long)nx * ny * nz / 8;
  const long long runs = (long long)B * ((in_n + 64 * vpt - 1) / (64 * vpt));
  const int cb = (co + TF_CO - 1) / TF_CO;
  const int per_sm = two ? 2 : 6;
  const dim3 grid((unsigned)std::min(runs, std::max(1LL, 152LL * per_sm / cb)), cb);
  const int vec = in_n % 4 == 0 && (uintptr_t)in % 16 == 0;
  kern<<<grid, UT, smem, st>>>(in, ci, out, out_bs, co, W, bias, B, nx, ny, nz, bf, nbuf, vec);
  return cudaGetLastError();
}

// din[b][ci][v] = sum_co sum_d W[ci][co][d] dout[b][co][2v + d]  ((nx, ny, nz) = output dims).  A CTA
// keeps the weights of CI = 32 input channels in shared memory (16 above 128 output channels);
// a thread owns TD_K voxels and CI / 4 input channels, so a weight loaded serves TD_K FMAs (shared
// memory returns one float per lane and clock to the SM's four schedulers together) and a
// voxel's 8 children (four 8-byte loads, shared by the voxel's four threads through L1)
// CI / 4 each.  The two at 24 x 64x64x32 (65 us of FMAs): 1.22 ms, 0.38 with one voxel per
// thread (still the better where four leave an SM without two CTAs: 64 -> 32 at 24 x 16^3 41
// against 48 us), now 0.23.
template <int CI, int TD_K>
__global__ void __launch_bounds__(UT, 2) k_tconv_dgrad(const float* __restrict__ dout, long long dout_bs, int co_n, float* __restrict__ din,
                                                       int ci_n, const float* __restrict__ W, int B, int nx, int ny, int nz, int bf) {
  constexpr int PER = CI / 4, TD_V = 64 * TD_K;
  extern __shared__ __align__(16) float td_sm[];   // [co][CI][8]
  const int ix = nx / 2, iy = ny / 2, iz = nz / 2, in_n = ix * iy * iz;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int ci0 = blockIdx.y * CI, runs = (in_n + TD_V - 1) / TD_V;
  for (int e = threadIdx.x; e < co_n * CI * 8; e += UT) {
    const int d = e % 8, ci = (e / 8) % CI, co = e / (8 * CI);
    td_sm[e] = ci0 + ci < ci_n ? opr(__ldg(&W[((long long)(ci0 + ci) * co_n + co) * 8 + d]), bf) : 0.f;
  }
  __syncthreads();
  const int vi = threadIdx.x % 64, cig = threadIdx.x / 64;
  for (long long r = blockIdx.x; r < (long long)B * runs; r += gridDim.x) {
    const int b = (int)(r / runs), v0 = (int)(r % runs) * TD_V + vi;
    const float* gb = dout + (long long)b * dout_bs;
    long long off[TD_K];   // the first child of voxel v0 + 64 k; past the sample's end: its first voxel's, dropped below
#pragma unroll
    for (int k = 0; k < TD_K; ++k) {
      const int v = v0 + 64 * k < in_n ? v0 + 64 * k : 0;
      const int x = v % ix, y = (v / ix) % iy, z = v / (ix * iy);
      off[k] = 2 * z * plane + (long long)(2 * y) * nx + 2 * x;
    }
    float acc[TD_K][PER];
#pragma unroll
    for (int k = 0; k < TD_K; ++k)
#pragma unroll
      for (int j = 0; j < PER; ++j) acc[k][j] = 0.f;
#pragma unroll 1
    for (int co = 0; co < co_n; ++co) {
      const float* g = gb + (long long)co * n;
      float gv[TD_K][8];
#pragma unroll
      for (int k = 0; k < TD_K; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 t = __ldg(reinterpret_cast<const float2*>(g + off[k] + (q >> 1) * plane + (q & 1) * nx));
          gv[k][2 * q] = opr(t.x, bf);
          gv[k][2 * q + 1] = opr(t.y, bf);
        }
      const float4* w = reinterpret_cast<const float4*>(td_sm + (co * CI + PER * cig) * 8);
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const float4 w0 = w[2 * j], w1 = w[2 * j + 1];
#pragma unroll
        for (int k = 0; k < TD_K; ++k) {
          float s = acc[k][j];
          s = fmaf(w0.x, gv[k][0], s);
          s = fmaf(w0.y, gv[k][1], s);
          s = fmaf(w0.z, gv[k][2], s);
          s = fmaf(w0.w, gv[k][3], s);
          s = fmaf(w1.x, gv[k][4], s);
          s = fmaf(w1.y, gv[k][5], s);
          s = fmaf(w1.z, gv[k][6], s);
          acc[k][j] = fmaf(w1.w, gv[k][7], s);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < TD_K; ++k) {
      if (v0 + 64 * k >= in_n) continue;
      float* o = din + ((long long)b * ci_n + ci0 + PER * cig) * in_n + v0 + 64 * k;
#pragma unroll
      for (int j = 0; j < PER; ++j)
        if (ci0 + PER * cig + j < ci_n) o[(long long)j * in_n] = acc[k][j];
    }
  }
}

static cudaError_t tconv_dgrad(const float* dout, long long dout_bs, int co, float* din, int ci, const float* W, int B, int nx,
                               int ny, int nz, int bf, cudaStream_t st) {
  const int cic = co <= 128 ? 32 : 16, cb = (ci + cic - 1) / cic;
  auto runs = [&](int k) { return (long long)B * (((long long)nx * ny * nz / 8 + 64 * k - 1) / (64 * k)); };
  const bool four = runs(4) * cb >= 2 * 152;   // four voxels per thread
  auto kern = cic == 32 ? (four ? k_tconv_dgrad<32, 4> : k_tconv_dgrad<32, 1>) : (four ? k_tconv_dgrad<16, 4> : k_tconv_dgrad<16, 1>);
  const size_t smem = sizeof(float) * (size_t)co * cic * 8;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)std::min(runs(four ? 4 : 1), std::max(1LL, 152LL * 6 / cb)), cb);
  kern<<<grid, UT, smem, st>>>(dout, dout_bs, co, din, ci, W, B, nx, ny, nz, bf);
  return cudaGetLastError();
}

// dW[ci][co][d] = sum_{b, v} in[b][ci][v] dout[b][co][2v + d]: a product of a [ci][voxel] and a
// [voxel][(co, d)] matrix.  A CTA takes 32 input and 16 output channels (32 x 128 sums, 8 x 4 per
// thread, so three 16-byte shared loads feed 32 FMAs) and a share of the 32-voxel chunks of
// the samples' flat voxel order, whatever the rows' width; the next chunk's loads are in
// flight in registers while the current one's FMAs run.  Bound by FMA issue (24 x 64x64x32,
// 32 -> 16: 43 us of FMAs, 30 us of HBM).  Two sums per thread walked 64-voxel rows, mostly
// padding at the coarse levels (16 wide: a quarter used): 807 us there and 765 us for 64 -> 32 at
// half size, now 124 and 63.  A chain is 256 voxels; each is added in FP32 to a second
// register sum, and a second kernel adds the shares' sums (part[share][ci][co][d]) in a fixed order.
constexpr int TW_CI = 32, TW_CO = 16, TW_V = 32, TW_NT = 128, TW_CHAIN = 8;   // TW_CHAIN: chunks per chain
constexpr int TW_XP = TW_CI + 4, TW_GP = TW_CO * 8 + 8;                       // row pitches (floats)
__global__ void __launch_bounds__(TW_NT, 3) k_tconv_wgrad(const float* __restrict__ in, int ci_n,
                                                          const float* __restrict__ dout, long long dout_bs, int co_n,
                                                          float* __restrict__ part, int B, int nx, int ny, int nz, int bf) {
  __shared__ __align__(16) float s_x[2][TW_V][TW_XP];   // [voxel][ci]
  __shared__ __align__(16) float s_g[2][TW_V][TW_GP];   // [voxel][co][d]
  const int ix = nx / 2, iy = ny / 2, iz = nz / 2, in_n = ix * iy * iz;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int ci0 = blockIdx.y * TW_CI, co0 = blockIdx.z * TW_CO;
  const int per_b = (in_n + TW_V - 1) / TW_V;
  const long long chunks = (long long)B * per_b;
  const long long c_begin = chunks * blockIdx.x / gridDim.x, c_end = chunks * (blockIdx.x + 1) / gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int XT = TW_V * TW_CI / TW_NT;              // inputs staged per thread: voxel `lane`, channel warp + 4 k
  constexpr int GT = TW_V * TW_CO * 4 / TW_NT;          // children pairs per thread
  // pair k: voxel lane / 4 + 8 (k % 4), row (co, dz, dy) = lane % 4 + 4 warp + 16 (k / 4)
  const int gv0 = lane >> 2, gr0 = (lane & 3) + 4 * warp;
  float xv[XT];
  float2 gv[GT];
  auto load = [&](long long c) {
    const int b = (int)(c / per_b), v0 = (int)(c % per_b) * TW_V;
    const float* xs = in + ((long long)b * ci_n + ci0) * in_n + v0 + lane;
#pragma unroll
    for (int k = 0; k < XT; ++k) {
      const int ci = warp + 4 * k;
      xv[k] = v0 + lane < in_n && ci0 + ci < ci_n ? __ldg(xs + (long long)ci * in_n) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int v = v0 + gv0 + 8 * j;
      const int x = v % ix, y = v / ix % iy, z = v / (ix * iy);
      const float* gs = dout + b * dout_bs + (long long)(2 * z) * plane + (long long)(2 * y) * nx + 2 * x;
#pragma unroll
      for (int i = 0; i < GT / 4; ++i) {
        const int row = gr0 + 16 * i, co = co0 + row / 4;
        gv[4 * i + j] = v < in_n && co < co_n
                            ? __ldg(reinterpret_cast<const float2*>(gs + co * n + ((row >> 1) & 1) * plane + (row & 1) * nx))
                            : make_float2(0.f, 0.f);
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int k = 0; k < XT; ++k) s_x[buf][lane][warp + 4 * k] = opr(xv[k], bf);
#pragma unroll
    for (int k = 0; k < GT; ++k)
      *reinterpret_cast<float2*>(&s_g[buf][gv0 + 8 * (k % 4)][2 * (gr0 + 16 * (k / 4))]) =
          make_float2(opr(gv[k].x, bf), opr(gv[k].y, bf));
  };
  float acc[8][4], sum[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = sum[i][j] = 0.f;
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sum[i][j] += acc[i][j];
        acc[i][j] = 0.f;
      }
  };
  if (c_begin < c_end) {
    load(c_begin);
    store(0);
  }
  __syncthreads();
  for (long long c = c_begin; c < c_end; ++c) {
    const int buf = (int)(c - c_begin) & 1;
    if (c + 1 < c_end) load(c + 1);
    const float* xp = &s_x[buf][0][8 * warp];
    const float* gp = &s_g[buf][0][4 * lane];
#pragma unroll 4
    for (int v = 0; v < TW_V; ++v) {
      const float4 xa = *reinterpret_cast<const float4*>(xp + v * TW_XP);
      const float4 xb = *reinterpret_cast<const float4*>(xp + v * TW_XP + 4);
      const float4 g = *reinterpret_cast<const float4*>(gp + v * TW_GP);
      const float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc[i][0] = fmaf(x[i], g.x, acc[i][0]);
        acc[i][1] = fmaf(x[i], g.y, acc[i][1]);
        acc[i][2] = fmaf(x[i], g.z, acc[i][2]);
        acc[i][3] = fmaf(x[i], g.w, acc[i][3]);
      }
    }
    if ((c - c_begin) % TW_CHAIN == TW_CHAIN - 1) flush();
    if (c + 1 < c_end) store(buf ^ 1);   // the other buffer: its readers passed the last barrier
    __syncthreads();
  }
  flush();
  const int co = co0 + lane / 2;
  if (co >= co_n) return;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int ci = ci0 + 8 * warp + i;
    if (ci >= ci_n) continue;
    *reinterpret_cast<float4*>(part + (((long long)blockIdx.x * ci_n + ci) * co_n + co) * 8 + 4 * (lane & 1)) =
        make_float4(sum[i][0], sum[i][1], sum[i][2], sum[i][3]);
  }
}

static int tconv_shares(int ci, int co, int B, int nx, int ny, int nz) {
  const int tiles = ((ci + TW_CI - 1) / TW_CI) * ((co + TW_CO - 1) / TW_CO);
  const long long chunks = (long long)B * (((long long)nx * ny * nz / 8 + TW_V - 1) / TW_V);
  return (int)std::min(chunks, (long long)std::max(1, 152 * 3 / tiles));   // one wave of three CTAs per SM
}
static size_t tconv_part(int ci, int co, int B, int nx, int ny, int nz) {   // floats of scratch
  return (size_t)tconv_shares(ci, co, B, nx, ny, nz) * ci * co * 8;
}
static cudaError_t tconv_wgrad(const float* in, int ci, const float* dout, long long dout_bs, int co, float* dW, int B,
                               int nx, int ny, int nz, int bf, float* part, cudaStream_t st) {
  const int shares = tconv_shares(ci, co, B, nx, ny, nz);
  k_tconv_wgrad<<<dim3(shares, (ci + TW_CI - 1) / TW_CI, (co + TW_CO - 1) / TW_CO), TW_NT, 0, st>>>(
      in, ci, dout, dout_bs, co, part, B, nx, ny, nz, bf);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : unet_sum_shares(part, shares, ci * co * 8, dW, st);
}

// 1x1x1 conv to one channel: out[b][v] = bias + sum_c W[c] in[b][c][v], four voxels per thread
template <bool VEC>
__global__ void __launch_bounds__(UT) k_conv1_fwd(const float* __restrict__ in, int c_n, const float* __restrict__ W,
                                                  const float* __restrict__ bias, float* __restrict__ out, int B, long long n,
                                                  int bf) {
  const long long u = (long long)blockIdx.x * UT + threadIdx.x;
  if (u >= (VEC ? n / 4 : n)) return;
  const float b0 = __ldg(bias);
  for (int b = blockIdx.y; b < B; b += gridDim.y) {
    const float* ip = in + (long long)b * c_n * n;
    if constexpr (VEC) {
      float4 acc = make_float4(b0, b0, b0, b0);
#pragma unroll 8
      for (int c = 0; c < c_n; ++c) {
        const float w = opr(__ldg(&W[c]), bf);
        const float4 x = __ldg(reinterpret_cast<const float4*>(ip + (long long)c * n) + u);
        acc = make_float4(fmaf(w, opr(x.x, bf), acc.x), fmaf(w, opr(x.y, bf), acc.y), fmaf(w, opr(x.z, bf), acc.z),
                          fmaf(w, opr(x.w, bf), acc.w));
      }
      reinterpret_cast<float4*>(out + (long long)b * n)[u] = acc;
    } else {
      float acc = b0;
      for (int c = 0; c < c_n; ++c) acc = fmaf(opr(__ldg(&W[c]), bf), opr(__ldg(&ip[(long long)c * n + u]), bf), acc);
      out[(long long)b * n + u] = acc;
    }
  }
}

static cudaError_t conv1_fwd(const float* in, int c, const float* W, const float* bias, float* out, int B, long long n, int bf,
                             cudaStream_t st) {
  const bool vec = n % 4 == 0;
  const dim3 grid((unsigned)(((vec ? n / 4 : n) + UT - 1) / UT), std::min(B, 65535));
  if (vec) k_conv1_fwd<true><<<grid, UT, 0, st>>>(in, c, W, bias, out, B, n, bf);
  else k_conv1_fwd<false><<<grid, UT, 0, st>>>(in, c, W, bias, out, B, n, bf);
  return cudaGetLastError();
}
// Backward of the 1x1x1 conv and of the ReLU before it, in one pass over the input `in` (the
// ReLU output): din[b][c][v] = W[c] dout[b][v] where in > 0, else 0; partial sums of dW[c] = sum in dout,
// db = sum dout (once, by channel 0's CTAs) and dbprev[c] = sum din (the bias of the layer
// that made `in`) into pw, pb and pp.
template <bool VEC>
__global__ void __launch_bounds__(UT) k_conv1_bwd(const float* __restrict__ in, int c_n, const float* __restrict__ dout,
                                                  const float* __restrict__ W, float* __restrict__ din,
                                                  float* __restrict__ pw, float* __restrict__ pb,
                                                  float* __restrict__ pp, int B, long long n, int bf) {
  const int c = blockIdx.y;
  const long long units = VEC ? n / 4 : n;
  const long long u0 = (long long)blockIdx.x * (UT * RC_PER) + threadIdx.x;
  const float w = opr(__ldg(&W[c]), bf);
  float sw = 0.f, sb = 0.f, sp = 0.f;
  for (int b = blockIdx.z; b < B; b += gridDim.z) {
    const float* ip = in + ((long long)b * c_n + c) * n;
    float* op = din + ((long long)b * c_n + c) * n;
    const float* gp = dout + (long long)b * n;
    auto one = [&](float x, float g) {
      const float gr = opr(g, bf), d = x > 0.f ? w * gr : 0.f;
      sw = fmaf(opr(x, bf), gr, sw);
      sb += g;
      sp += d;
      return d;
    };
#pragma unroll
    for (int k = 0; k < RC_PER; ++k) {
      const long long u = u0 + k * UT;
      if (u >= units) continue;
      if constexpr (VEC) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(ip) + u), g = __ldg(reinterpret_cast<const float4*>(gp) + u);
        reinterpret_cast<float4*>(op)[u] = make_float4(one(x.x, g.x), one(x.y, g.y), one(x.z, g.z), one(x.w, g.w));
      } else {
        op[u] = one(__ldg(ip + u), __ldg(gp + u));
      }
    }
  }
  sw = block_sum(sw);
  sb = block_sum(sb);
  sp = block_sum(sp);
  if (threadIdx.x == 0) {
    pw[chan_part(c)] = sw;
    pp[chan_part(c)] = sp;
    if (c == 0) pb[chan_part(0)] = sb;
  }
}

// MSE: loss = mean (p - t)^2, g = 2 (p - t) / N; loss accumulated in FP64 partials.
__global__ void __launch_bounds__(UT) k_mse(const float* __restrict__ p, const float* __restrict__ t,
                                            float* __restrict__ g, long long N, double* __restrict__ part) {
  double acc = 0.0;
  for (long long i = (long long)blockIdx.x * UT + threadIdx.x; i < N; i += (long long)gridDim.x * UT) {
    const float d = p[i] - t[i];
    g[i] = 2.0f * d / (float)N;
    acc += (double)d * d;
  }
  __shared__ double red[UT];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = UT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}
// Sum of np FP64 partials over the CTA's UT threads, the same in every thread (and every CTA).
// One thread adding 2432 partials in turn took 0.14 ms.
__device__ double sum_of_parts(const double* __restrict__ part, int np) {
  __shared__ double red[UT];
  double a = 0.0;
  for (int i = threadIdx.x; i < np; i += UT) a += part[i];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int o = UT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  return red[0];
}
__global__ void __launch_bounds__(UT) k_mse_final(const double* part, int nb, long long N, double* loss) {
  const double a = sum_of_parts(part, nb);
  if (threadIdx.x == 0) *loss = a / (double)N;
}

// Adam (Kingma and Ba, 2015): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2; p -= lr_t m / (sqrt(v) + eps_t)
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       long long count, float lr_t, float b1, float b2, float eps_t) {
  for (long long i = (long long)blockIdx.x * UT + threadIdx.x; i < count; i += (long long)gridDim.x * UT) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr_t * mi / (sqrtf(vi) + eps_t);
  }
}

// Per-sample normalisation (one CTA per sample): m = sum(x_b) / norm_count in FP64,
// xo = x / m, to = t / m (m <= 0 leaves the sample unscaled).
constexpr int NORM_T = 1024;
__global__ void __launch_bounds__(NORM_T) k_sample_norm(const float* __restrict__ x, const float* __restrict__ t,
                                                        float* __restrict__ xo, float* __restrict__ to, long long n,
                                                        double norm_count) {
  const long long base = (long long)blockIdx.x * n;
  double acc = 0.0;
  for (long long i = threadIdx.x; i < n; i += NORM_T) acc += (double)x[base + i];
  __shared__ double red[NORM_T];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = NORM_T / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const double m = red[0] / norm_count;
  const float inv = m > 0.0 ? (float)(1.0 / m) : 1.0f;
  for (long long i = threadIdx.x; i < n; i += NORM_T) {
    xo[base + i] = x[base + i] * inv;
    if (t) to[base + i] = t[base + i] * inv;
  }
}

// Partial sums of x (one per CTA, FP64), four elements at a time (exact_sum.cuh): 43 -> 22 us at 256x256x128.
template <bool VEC>
__global__ void __launch_bounds__(UT) k_sum_part(const float* __restrict__ x, long long n, double* __restrict__ part) {
  double acc = 0.0;
  const long long t0 = (long long)blockIdx.x * UT + threadIdx.x, step = (long long)gridDim.x * UT;
  if constexpr (VEC) {
    for (long long i = t0; i < n / 4; i += step) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(x) + i);
      add_four(acc, v.x, v.y, v.z, v.w);
    }
  } else {
    for (long long i = t0; i < n; i += step) acc += x[i];
  }
  __shared__ double red[UT];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = UT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// xo = x / m, m = sum(x) / norm_count from the partials (m <= 0 leaves x unscaled)
template <bool VEC>
__global__ void __launch_bounds__(UT) k_scale_by_mean(const float* __restrict__ x, long long n,
                                                     const double* __restrict__ part, int np, double norm_count,
                                                     float* __restrict__ xo) {
  const double m = sum_of_parts(part, np) / norm_count;
  const float inv = m > 0.0 ? (float)(1.0 / m) : 1.0f;
  const long long t0 = (long long)blockIdx.x * UT + threadIdx.x, step = (long long)gridDim.x * UT;
  if constexpr (VEC) {
    for (long long i = t0; i < n / 4; i += step) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(x) + i);
      reinterpret_cast<float4*>(xo)[i] = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    }
  } else {
    for (long long i = t0; i < n; i += step) xo[i] = x[i] * inv;
  }
}

// r_init = m * max(out, floor): the network's output back in the input's units, kept positive.
template <bool VEC>
__global__ void __launch_bounds__(UT) k_warm_map(const float* __restrict__ out, long long n,
                                                 const double* __restrict__ part, int np, double norm_count,
                                                 float floor_rel, float* __restrict__ r) {
  const double m = sum_of_parts(part, np) / norm_count;
  const float sc = m > 0.0 ? (float)m : 1.0f;
  const long long t0 = (long long)blockIdx.x * UT + threadIdx.x, step = (long long)gridDim.x * UT;
  if constexpr (VEC) {
    for (long long i = t0; i < n / 4; i += step) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(out) + i);
      reinterpret_cast<float4*>(r)[i] = make_float4(sc * fmaxf(v.x, floor_rel), sc * fmaxf(v.y, floor_rel),
                                                    sc * fmaxf(v.z, floor_rel), sc * fmaxf(v.w, floor_rel));
    }
  } else {
    for (long long i = t0; i < n; i += step) r[i] = sc * fmaxf(out[i], floor_rel);
  }
}

static unsigned grid_for(long long work) {
  long long b = (work + UT - 1) / UT;
  return (unsigned)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

}  // namespace unet
}  // namespace clamp

using namespace clamp::unet;

struct clamp_unet {
  int c1, c2, c3, dev, bf;
  std::vector<Layer> layers;
  size_t count = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *flip = nullptr;
  size_t flip_count = 0;
  uint4* wpk = nullptr;   // BF16 packed weights of the conv on the tensor cores
  int* err = nullptr;     // device word: bit 2 = a tensor-core wait gave up
  int tc = 1;             // BF16 convs on the tensor cores where supported
  TcCtx ctx() const { return TcCtx{wpk, err, bf != 0 && tc != 0}; }
};

// Workspace: activations and their gradients for batch B at (nx, ny, nz).
namespace {
struct Acts {
  float *e1a, *cat1, *p1, *e2a, *cat2, *p2, *bta, *btb, *d2a, *d2b, *d1a, *d1b, *out, *xin;
  float *ge1a, *gcat1, *gp1, *ge2a, *gcat2, *gp2, *gbta, *gbtb, *gd2a, *gd2b, *gd1a, *gd1b, *gout;
  unsigned char *arg1, *arg2;
  double* part;
  float* shares;   // partial sums of one weight gradient
  float* chan;     // partial sums of the biases' and the 1x1 conv's gradients
  size_t bytes;
};

Acts acts_layout(const clamp_unet* u, int B, int nx, int ny, int nz, void* base, bool with_grads) {
  const long long n1 = (long long)nx * ny * nz, n2 = n1 / 8, n3 = n1 / 64;
  size_t off = 0;
  char* b = static_cast<char*>(base);
  auto take = [&](long long floats) -> float* {
    float* r = b ? reinterpret_cast<float*>(b + off) : nullptr;
    off += ((size_t)floats * sizeof(float) + 255) & ~(size_t)255;
    return r;
  };
  Acts a{};
  const int c1 = u->c1, c2 = u->c2, c3 = u->c3;
  float** fw[] = {&a.e1a, &a.cat1, &a.p1, &a.e2a, &a.cat2, &a.p2, &a.bta, &a.btb, &a.d2a, &a.d2b, &a.d1a, &a.d1b, &a.out};
  const long long sz[] = {c1 * n1, 2LL * c1 * n1, c1 * n2, c2 * n2, 2LL * c2 * n2, c2 * n3, c3 * n3, c3 * n3,
                          c2 * n2, c2 * n2, c1 * n1, c1 * n1, n1};
  for (int i = 0; i < 13; ++i) *fw[i] = take(B * sz[i]);
  a.xin = take(B * n1);
  if (with_grads) {
    float** gw[] = {&a.ge1a, &a.gcat1, &a.gp1, &a.ge2a, &a.gcat2, &a.gp2, &a.gbta, &a.gbtb, &a.gd2a, &a.gd2b, &a.gd1a, &a.gd1b, &a.gout};
    for (int i = 0; i < 13; ++i) *gw[i] = take(B * sz[i]);
  }
  a.arg1 = reinterpret_cast<unsigned char*>(take((B * c1 * n2 + 3) / 4));
  a.arg2 = reinterpret_cast<unsigned char*>(take((B * c2 * n3 + 3) / 4));
  a.part = reinterpret_cast<double*>(take(2 * 152 * 16));
  if (with_grads) {
    size_t m = 0;
    for (const Layer& L : u->layers) {
      const int lx = nx / L.level, ly = ny / L.level, lz = nz / L.level;
      if (L.kind == TCONV) m = std::max(m, tconv_part(L.ci, L.co, B, lx, ly, lz));
      if (L.kind == CONV3 && u->bf) m = std::max(m, clamp::unet_wgrad3_tc_part(L.ci, L.co, B, lx, ly, lz));
    }
    a.shares = take((long long)m);
    // five layers' biases at the first two levels, two's at the third; the 1x1 conv's weights and bias
    a.chan = take((6LL * c1 + 1) * chan_parts(n1, B) + 5LL * c2 * chan_parts(n2, B) + 2LL * c3 * chan_parts(n3, B));
  }
  a.bytes = off;
  return a;
}

bool unet_shape_ok(int B, int nx, int ny, int nz) {
  return B >= 1 && nx >= 4 && ny >= 4 && nz >= 4 && nx % 4 == 0 && ny % 4 == 0 && nz % 4 == 0;
}
}  // namespace

extern "C" clamp_status clamp_unet_create(int32_t c1, int32_t c2, int32_t c3, int32_t dtype, const float* params_host,
                                          clamp_unet** out) {
  if (!out || c1 < 1 || c2 < 1 || c3 < 1 || c1 > 256 || c2 > 256 || c3 > 256)
    return api_fail(CLAMP_EINVAL, "clamp_unet_create: channel counts must be in [1, 256]");
  if (dtype != CLAMP_DENOISER_FP32 && dtype != CLAMP_DENOISER_BF16)
    return api_fail(CLAMP_EINVAL, "clamp_unet_create: dtype must be CLAMP_DENOISER_FP32 or CLAMP_DENOISER_BF16");
  clamp_unet* u = new clamp_unet();
  u->bf = dtype == CLAMP_DENOISER_BF16;
  u->c1 = c1;
  u->c2 = c2;
  u->c3 = c3;
  cudaGetDevice(&u->dev);
  const int spec[13][4] = {{CONV3, 1, c1, 1},  {CONV3, c1, c1, 1}, {CONV3, c1, c2, 2},     {CONV3, c2, c2, 2}, {CONV3, c2, c3, 4},
                           {CONV3, c3, c3, 4}, {TCONV, c3, c2, 2}, {CONV3, 2 * c2, c2, 2}, {CONV3, c2, c2, 2},
                           {TCONV, c2, c1, 1}, {CONV3, 2 * c1, c1, 1}, {CONV3, c1, c1, 1}, {CONV1, c1, 1, 1}};
  size_t off = 0;
  for (auto& s : spec) {
    Layer L{s[0], s[1], s[2], s[3], 0, 0, 0};
    L.nw = (size_t)s[1] * s[2] * (s[0] == CONV3 ? 27 : s[0] == TCONV ? 8 : 1);
    L.w = off;
    off += L.nw;
    L.b = off;
    off += s[2];
    if (s[0] == CONV3) u->flip_count = std::max(u->flip_count, L.nw);
    u->layers.push_back(L);
  }
  u->count = off;
  const size_t bytes = off * sizeof(float);
  size_t wpk_bytes = 16;
  for (const Layer& L : u->layers)
    if (L.kind == CONV3 && L.ci >= 16)   // forward (ci -> co) and data gradient (co -> ci)
      wpk_bytes = std::max({wpk_bytes, clamp::unet_conv3_tc_wpk_bytes(L.ci, L.co),
                            clamp::unet_conv3_tc_wpk_bytes(L.co, L.ci)});
  if (cudaMalloc(&u->p, bytes) != cudaSuccess || cudaMalloc(&u->g, bytes) != cudaSuccess ||
      cudaMalloc(&u->m, bytes) != cudaSuccess || cudaMalloc(&u->v, bytes) != cudaSuccess ||
      cudaMalloc(&u->flip, u->flip_count * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&u->wpk, wpk_bytes) != cudaSuccess || cudaMalloc(&u->err, sizeof(int)) != cudaSuccess) {
    clamp_unet_destroy(u);
    return api_fail(CLAMP_ENOMEM, "clamp_unet_create: device allocation failed");
  }
  cudaError_t e = cudaSuccess;
  for (float* q : {u->g, u->m, u->v})
    if (e == cudaSuccess) e = cudaMemset(q, 0, bytes);
  if (e == cudaSuccess) e = cudaMemset(u->err, 0, sizeof(int));
  if (e == cudaSuccess)
    e = params_host ? cudaMemcpy(u->p, params_host, bytes, cudaMemcpyHostToDevice) : cudaMemset(u->p, 0, bytes);
  if (e != cudaSuccess) {
    clamp_unet_destroy(u);
    return api_fail(CLAMP_ECUDA, "clamp_unet_create: %s", cudaGetErrorString(e));
  }
  *out = u;
  return CLAMP_OK;
}

extern "C" void clamp_unet_destroy(clamp_unet* u) {
  if (!u) return;
  for (float* q : {u->p, u->g, u->m, u->v, u->flip})
    if (q) cudaFree(q);
  if (u->wpk) cudaFree(u->wpk);
  if (u->err) cudaFree(u->err);
  delete u;
}

extern "C" int64_t clamp_unet_param_count(const clamp_unet* u) { return u ? (int64_t)u->count : 0; }

static float* unet_state(const clamp_unet* u, int which) {
  switch (which) {
    case 0: return u->p;
    case 1: return u->g;
    case 2: return u->m;
    case 3: return u->v;
    default: return nullptr;
  }
}

extern "C" clamp_status clamp_unet_get(const clamp_unet* u, int32_t which, float* host) {
  if (!u || !host || !unet_state(u, which)) return api_fail(CLAMP_EINVAL, "clamp_unet_get: bad arguments");
  const cudaError_t e = cudaMemcpy(host, unet_state(u, which), u->count * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? CLAMP_OK : api_fail(CLAMP_ECUDA, "clamp_unet_get: %s", cudaGetErrorString(e));
}

extern "C" clamp_status clamp_unet_set(clamp_unet* u, int32_t which, const float* host) {
  if (!u || !host || !unet_state(u, which)) return api_fail(CLAMP_EINVAL, "clamp_unet_set: bad arguments");
  const cudaError_t e = cudaMemcpy(unet_state(u, which), host, u->count * sizeof(float), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? CLAMP_OK : api_fail(CLAMP_ECUDA, "clamp_unet_set: %s", cudaGetErrorString(e));
}

extern "C" size_t clamp_unet_workspace_size(const clamp_unet* u, int32_t batch, int32_t nx, int32_t ny, int32_t nz,
                                            int32_t training) {
  if (!u || !unet_shape_ok(batch, nx, ny, nz)) return 0;
  return acts_layout(u, batch, nx, ny, nz, nullptr, training != 0).bytes;
}

// The network's buffers live on the device it was created on.
static bool on_unet_device(const clamp_unet* u, const char* where) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != u->dev) {
    api_fail(CLAMP_EINVAL, "%s: the network was created on device %d, current device is %d", where, u->dev, dev);
    return false;
  }
  return true;
}

// The kernels access the workspace 16 bytes at a time.
static clamp_status check_unet_ws(const void* ws, size_t have, size_t need, const char* where) {
  if (!ws || have < need) return api_fail(CLAMP_ENOMEM, "%s: workspace too small", where);
  if ((uintptr_t)ws & 255) return api_fail(CLAMP_EINVAL, "%s: workspace must be 256-byte aligned", where);
  return CLAMP_OK;
}

#define U_TRY(x)                                                                       \
  do {                                                                                 \
    cudaError_t _e = (x);                                                              \
    if (_e != cudaSuccess) return api_fail(CLAMP_ECUDA, "unet: %s", cudaGetErrorString(_e)); \
  } while (0)

static clamp_status unet_forward(clamp_unet* u, const float* x, int B, int nx, int ny, int nz, const Acts& a,
                                 cudaStream_t st) {
  const bool bf = u->bf != 0;
  const int c1 = u->c1, c2 = u->c2, c3 = u->c3;
  const long long n1 = (long long)nx * ny * nz, n2 = n1 / 8, n3 = n1 / 64;
  const int hx = nx / 2, hy = ny / 2, hz = nz / 2, qx = nx / 4, qy = ny / 4, qz = nz / 4;
  auto W = [&](int i) { return u->p + u->layers[i].w; };
  auto Bi = [&](int i) { return u->p + u->layers[i].b; };
  U_TRY(conv3(bf, x, n1, 1, a.e1a, c1 * n1, c1, W(0), Bi(0), true, B, nx, ny, nz, st, u->ctx()));
  U_TRY(conv3(bf, a.e1a, c1 * n1, c1, a.cat1 + c1 * n1, 2 * c1 * n1, c1, W(1), Bi(1), true, B, nx, ny, nz, st, u->ctx()));  // s1
  k_pool_fwd<<<pool_grid(nx, ny, nz, c1, B), UT, 0, st>>>(a.cat1 + c1 * n1, 2 * c1 * n1, a.p1, a.arg1, c1, B, nx, ny, nz);
  U_TRY(cudaGetLastError());
  U_TRY(conv3(bf, a.p1, c1 * n2, c1, a.e2a, c2 * n2, c2, W(2), Bi(2), true, B, hx, hy, hz, st, u->ctx()));
  U_TRY(conv3(bf, a.e2a, c2 * n2, c2, a.cat2 + c2 * n2, 2 * c2 * n2, c2, W(3), Bi(3), true, B, hx, hy, hz, st, u->ctx()));  // s2
  k_pool_fwd<<<pool_grid(hx, hy, hz, c2, B), UT, 0, st>>>(a.cat2 + c2 * n2, 2 * c2 * n2, a.p2, a.arg2, c2, B, hx, hy, hz);
  U_TRY(cudaGetLastError());
  U_TRY(conv3(bf, a.p2, c2 * n3, c2, a.bta, c3 * n3, c3, W(4), Bi(4), true, B, qx, qy, qz, st, u->ctx()));
  U_TRY(conv3(bf, a.bta, c3 * n3, c3, a.btb, c3 * n3, c3, W(5), Bi(5), true, B, qx, qy, qz, st, u->ctx()));
  U_TRY(tconv_fwd(a.btb, c3, a.cat2, 2 * c2 * n2, c2, W(6), Bi(6), B, hx, hy, hz, bf, st));
  U_TRY(conv3(bf, a.cat2, 2 * c2 * n2, 2 * c2, a.d2a, c2 * n2, c2, W(7), Bi(7), true, B, hx, hy, hz, st, u->ctx()));
  U_TRY(conv3(bf, a.d2a, c2 * n2, c2, a.d2b, c2 * n2, c2, W(8), Bi(8), true, B, hx, hy, hz, st, u->ctx()));
  U_TRY(tconv_fwd(a.d2b, c2, a.cat1, 2 * c1 * n1, c1, W(9), Bi(9), B, nx, ny, nz, bf, st));
  U_TRY(conv3(bf, a.cat1, 2 * c1 * n1, 2 * c1, a.d1a, c1 * n1, c1, W(10), Bi(10), true, B, nx, ny, nz, st, u->ctx()));
  U_TRY(conv3(bf, a.d1a, c1 * n1, c1, a.d1b, c1 * n1, c1, W(11), Bi(11), true, B, nx, ny, nz, st, u->ctx()));
  U_TRY(conv1_fwd(a.d1b, c1, W(12), Bi(12), a.out, B, n1, bf, st));
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_forward(clamp_unet* u, const float* x, float* y, int32_t batch, int32_t nx,
                                           int32_t ny, int32_t nz, void* ws, size_t ws_bytes, void* stream) {
  if (!u || !x || !y) return api_fail(CLAMP_EINVAL, "clamp_unet_forward: NULL argument");
  if (!on_unet_device(u, "clamp_unet_forward")) return CLAMP_EINVAL;
  if (!unet_shape_ok(batch, nx, ny, nz))
    return api_fail(CLAMP_EINVAL, "clamp_unet_forward: nx, ny, nz must be multiples of 4");
  const Acts a = acts_layout(u, batch, nx, ny, nz, ws, false);
  if (const clamp_status w = check_unet_ws(ws, ws_bytes, a.bytes, "clamp_unet_forward")) return w;
  cudaStream_t st = (cudaStream_t)stream;
  clamp_status s = unet_forward(u, x, batch, nx, ny, nz, a, st);
  if (s != CLAMP_OK) return s;
  const long long n1 = (long long)nx * ny * nz;
  U_TRY(cudaMemcpyAsync(y, a.out, sizeof(float) * batch * n1, cudaMemcpyDeviceToDevice, st));
  return CLAMP_OK;
}

// conv3 backward for layer li: input `in` (ci channels, sample stride in_bs), output gradient
// `g` (co channels, stride g_bs); writes din (if non-NULL) and accumulates dW.
//
// BF16 networks form dW on the tensor cores (16 -> 16 at 24 x 32^3: 0.11 ms, 0.47 ms on the CUDA
// cores) between two lengths of the CUDA cores' FP32 chains:
//   * below 128 terms a launch more would cost what the tensor cores save (17 against 10 to 17 us), and
//     the CUDA cores' sums are as exact (64 -> 64 at chains of 85: 4.3e-8 of FP64 against 4.5e-8);
//   * the longer chains are the less exact of the two by far (at 21 k terms 2e-6 of a layer's gradient,
//     at 79 k 1e-5 to 4e-5; the tensor cores' stay below 1e-7), but they are what earlier training
//     runs followed, and a gradient that leaves them moves by their whole error.  That error grows
//     with the length to the power 1.5 to 2, fastest at the full-size level, whose activations carry
//     the image's background.  Up to the limits it is below 2e-5 of the whole gradient: measured at
//     most 0.7e-6 at 21 k terms and 1.4e-5 at 41 k there; 9.4e-6 at 79 k and 1.1e-5 at 111 k at the coarser levels.
constexpr long long kTcChainMin = 128, kTcChainFull = 24LL << 10, kTcChainCoarse = 112LL << 10;
static clamp_status conv3_bwd(clamp_unet* u, int li, const float* in, long long in_bs, const float* g, long long g_bs,
                              float* din, long long din_bs, int B, int nx, int ny, int nz, float* part, cudaStream_t st) {
  const Layer& L = u->layers[li];
  const bool bf = u->bf != 0;
  if (din) {
    k_flip<<<grid_for((long long)L.nw), UT, 0, st>>>(u->p + L.w, u->flip, L.ci, L.co);
    U_TRY(cudaGetLastError());
    U_TRY(conv3(bf, g, g_bs, L.co, din, din_bs, L.ci, u->flip, nullptr, false, B, nx, ny, nz, st, u->ctx()));
  }
  const long long shares = wgrad3_shares(L.ci, L.co, B, ny, nz), voxels = (long long)B * nx * ny * nz;
  const long long most = L.level == 1 ? kTcChainFull : kTcChainCoarse;
  if (u->ctx().on && voxels >= kTcChainMin * shares && voxels <= most * shares)
    U_TRY(clamp::unet_wgrad3_tc(in, in_bs, L.ci, g, g_bs, L.co, u->g + L.w, B, nx, ny, nz, part, u->err, st));
  else
    U_TRY(wgrad3(in, in_bs, L.ci, g, g_bs, L.co, u->g + L.w, B, nx, ny, nz, u->bf, st));
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_backward(clamp_unet* u, const float* x, const float* target, int32_t batch,
                                            int32_t nx, int32_t ny, int32_t nz, double* loss, void* ws,
                                            size_t ws_bytes, void* stream) {
  if (!u || !x || !target) return api_fail(CLAMP_EINVAL, "clamp_unet_backward: NULL argument");
  if (!on_unet_device(u, "clamp_unet_backward")) return CLAMP_EINVAL;
  if (!unet_shape_ok(batch, nx, ny, nz))
    return api_fail(CLAMP_EINVAL, "clamp_unet_backward: nx, ny, nz must be multiples of 4");
  const Acts a = acts_layout(u, batch, nx, ny, nz, ws, true);
  if (const clamp_status w = check_unet_ws(ws, ws_bytes, a.bytes, "clamp_unet_backward")) return w;
  cudaStream_t st = (cudaStream_t)stream;
  const int bf = u->bf;
  const int B = batch, c1 = u->c1, c2 = u->c2, c3 = u->c3;
  const long long n1 = (long long)nx * ny * nz, n2 = n1 / 8, n3 = n1 / 64;
  const int hx = nx / 2, hy = ny / 2, hz = nz / 2, qx = nx / 4, qy = ny / 4, qz = nz / 4;
  clamp_status s = unet_forward(u, x, B, nx, ny, nz, a, st);
  if (s != CLAMP_OK) return s;
  U_TRY(cudaMemsetAsync(u->g, 0, u->count * sizeof(float), st));
  // loss and its gradient
  const unsigned nb = grid_for(B * n1);
  k_mse<<<nb, UT, 0, st>>>(a.out, target, a.gout, B * n1, a.part);
  U_TRY(cudaGetLastError());
  if (loss) {
    k_mse_final<<<1, UT, 0, st>>>(a.part, (int)nb, B * n1, loss);
    U_TRY(cudaGetLastError());
  }
  auto W = [&](int i) { return u->p + u->layers[i].w; };
  auto dB = [&](int i) { return u->g + u->layers[i].b; };
  // output 1x1 conv, the ReLU before it and that layer's bias
  ChanSums sums;
  sums.next = a.chan;
  float* pw = sums.add(u->g + u->layers[12].w, c1, n1, B);
  float* pb = sums.add(dB(12), 1, n1, B);
  float* pp = sums.add(dB(11), c1, n1, B);
  (n1 % 4 == 0 ? k_conv1_bwd<true> : k_conv1_bwd<false>)<<<chan_grid(n1, c1, B), UT, 0, st>>>(a.d1b, c1, a.gout, W(12), a.gd1b,
                                                                                              pw, pb, pp, B, n1, bf);
  U_TRY(cudaGetLastError());
  // decoder level 1
  s = conv3_bwd(u, 11, a.d1a, c1 * n1, a.gd1b, c1 * n1, a.gd1a, c1 * n1, B, nx, ny, nz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(relu_bias_grad<true>(a.gd1a, c1 * n1, a.d1a, c1 * n1, c1, B, n1, dB(10), sums, st));
  s = conv3_bwd(u, 10, a.cat1, 2 * c1 * n1, a.gd1a, c1 * n1, a.gcat1, 2 * c1 * n1, B, nx, ny, nz, a.shares, st);
  if (s != CLAMP_OK) return s;
  // transposed conv up1: u1 = cat1[:, :c1] from d2b
  U_TRY(tconv_dgrad(a.gcat1, 2 * c1 * n1, c1, a.gd2b, c2, W(9), B, nx, ny, nz, bf, st));
  U_TRY(tconv_wgrad(a.d2b, c2, a.gcat1, 2 * c1 * n1, c1, u->g + u->layers[9].w, B, nx, ny, nz, bf, a.shares, st));
  U_TRY(relu_bias_grad<false>(a.gcat1, 2 * c1 * n1, nullptr, 0, c1, B, n1, dB(9), sums, st));
  // decoder level 2
  U_TRY(relu_bias_grad<true>(a.gd2b, c2 * n2, a.d2b, c2 * n2, c2, B, n2, dB(8), sums, st));
  s = conv3_bwd(u, 8, a.d2a, c2 * n2, a.gd2b, c2 * n2, a.gd2a, c2 * n2, B, hx, hy, hz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(relu_bias_grad<true>(a.gd2a, c2 * n2, a.d2a, c2 * n2, c2, B, n2, dB(7), sums, st));
  s = conv3_bwd(u, 7, a.cat2, 2 * c2 * n2, a.gd2a, c2 * n2, a.gcat2, 2 * c2 * n2, B, hx, hy, hz, a.shares, st);
  if (s != CLAMP_OK) return s;
  // transposed conv up2: u2 = cat2[:, :c2] from btb
  U_TRY(tconv_dgrad(a.gcat2, 2 * c2 * n2, c2, a.gbtb, c3, W(6), B, hx, hy, hz, bf, st));
  U_TRY(tconv_wgrad(a.btb, c3, a.gcat2, 2 * c2 * n2, c2, u->g + u->layers[6].w, B, hx, hy, hz, bf, a.shares, st));
  U_TRY(relu_bias_grad<false>(a.gcat2, 2 * c2 * n2, nullptr, 0, c2, B, n2, dB(6), sums, st));
  // bottleneck
  U_TRY(relu_bias_grad<true>(a.gbtb, c3 * n3, a.btb, c3 * n3, c3, B, n3, dB(5), sums, st));
  s = conv3_bwd(u, 5, a.bta, c3 * n3, a.gbtb, c3 * n3, a.gbta, c3 * n3, B, qx, qy, qz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(relu_bias_grad<true>(a.gbta, c3 * n3, a.bta, c3 * n3, c3, B, n3, dB(4), sums, st));
  s = conv3_bwd(u, 4, a.p2, c2 * n3, a.gbta, c3 * n3, a.gp2, c2 * n3, B, qx, qy, qz, a.shares, st);
  if (s != CLAMP_OK) return s;
  // pool 2 into the skip s2 = cat2[:, c2:] (its gradient already holds the concat path)
  k_pool_bwd<<<pool_grid(hx, hy, hz, c2, B), UT, 0, st>>>(a.gp2, a.arg2, a.gcat2 + c2 * n2, 2 * c2 * n2, c2, B, hx, hy, hz);
  U_TRY(cudaGetLastError());
  // encoder level 2
  U_TRY(relu_bias_grad<true>(a.gcat2 + c2 * n2, 2 * c2 * n2, a.cat2 + c2 * n2, 2 * c2 * n2, c2, B, n2, dB(3), sums, st));
  s = conv3_bwd(u, 3, a.e2a, c2 * n2, a.gcat2 + c2 * n2, 2 * c2 * n2, a.ge2a, c2 * n2, B, hx, hy, hz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(relu_bias_grad<true>(a.ge2a, c2 * n2, a.e2a, c2 * n2, c2, B, n2, dB(2), sums, st));
  s = conv3_bwd(u, 2, a.p1, c1 * n2, a.ge2a, c2 * n2, a.gp1, c1 * n2, B, hx, hy, hz, a.shares, st);
  if (s != CLAMP_OK) return s;
  // pool 1 into the skip s1 = cat1[:, c1:]
  k_pool_bwd<<<pool_grid(nx, ny, nz, c1, B), UT, 0, st>>>(a.gp1, a.arg1, a.gcat1 + c1 * n1, 2 * c1 * n1, c1, B, nx, ny, nz);
  U_TRY(cudaGetLastError());
  // encoder level 1
  U_TRY(relu_bias_grad<true>(a.gcat1 + c1 * n1, 2 * c1 * n1, a.cat1 + c1 * n1, 2 * c1 * n1, c1, B, n1, dB(1), sums, st));
  s = conv3_bwd(u, 1, a.e1a, c1 * n1, a.gcat1 + c1 * n1, 2 * c1 * n1, a.ge1a, c1 * n1, B, nx, ny, nz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(relu_bias_grad<true>(a.ge1a, c1 * n1, a.e1a, c1 * n1, c1, B, n1, dB(0), sums, st));
  s = conv3_bwd(u, 0, x, n1, a.ge1a, c1 * n1, nullptr, 0, B, nx, ny, nz, a.shares, st);
  if (s != CLAMP_OK) return s;
  U_TRY(chan_sums(sums, st));
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_adam(clamp_unet* u, float lr, float beta1, float beta2, float eps, int32_t t,
                                        void* stream) {
  if (!u || t < 1) return api_fail(CLAMP_EINVAL, "clamp_unet_adam: bad arguments");
  if (!on_unet_device(u, "clamp_unet_adam")) return CLAMP_EINVAL;
  const double bc1 = 1.0 - pow((double)beta1, t), bc2 = 1.0 - pow((double)beta2, t);
  const float lr_t = (float)(lr * sqrt(bc2) / bc1), eps_t = (float)(eps * sqrt(bc2));
  k_adam<<<grid_for((long long)u->count), UT, 0, (cudaStream_t)stream>>>(u->p, u->g, u->m, u->v, (long long)u->count,
                                                                          lr_t, beta1, beta2, eps_t);
  U_TRY(cudaGetLastError());
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_set_tensor_cores(clamp_unet* u, int32_t on) {
  if (!u || (on != 0 && on != 1)) return api_fail(CLAMP_EINVAL, "clamp_unet_set_tensor_cores: bad arguments");
  u->tc = on;
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_check(clamp_unet* u) {
  if (!u) return api_fail(CLAMP_EINVAL, "clamp_unet_check: NULL network");
  if (!on_unet_device(u, "clamp_unet_check")) return CLAMP_EINVAL;
  int h = 0;
  U_TRY(cudaMemcpy(&h, u->err, sizeof(int), cudaMemcpyDeviceToHost));
  if (!h) return CLAMP_OK;
  U_TRY(cudaMemset(u->err, 0, sizeof(int)));
  return api_fail(CLAMP_ETIMEOUT, "clamp_unet_check: a bounded tensor-core wait gave up");
}

extern "C" clamp_status clamp_unet_normalize(int32_t batch, int64_t n, int64_t norm_count, const float* x,
                                             const float* t, float* x_out, float* t_out, void* stream) {
  if (batch < 1 || n < 1 || norm_count < 1 || !x || !x_out || (t && !t_out))
    return api_fail(CLAMP_EINVAL, "clamp_unet_normalize: bad arguments");
  k_sample_norm<<<batch, NORM_T, 0, (cudaStream_t)stream>>>(x, t, x_out, t_out, (long long)n, (double)norm_count);
  U_TRY(cudaGetLastError());
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_warm_start(clamp_unet* u, int32_t nx, int32_t ny, int32_t nz, const float* r0,
                                              float floor_rel, float* r_init, void* ws, size_t ws_bytes,
                                              void* stream) {
  if (!u || !r0 || !r_init) return api_fail(CLAMP_EINVAL, "clamp_unet_warm_start: NULL argument");
  if (!on_unet_device(u, "clamp_unet_warm_start")) return CLAMP_EINVAL;
  if (!unet_shape_ok(1, nx, ny, nz))
    return api_fail(CLAMP_EINVAL, "clamp_unet_warm_start: nx, ny, nz must be multiples of 4");
  const Acts a = acts_layout(u, 1, nx, ny, nz, ws, false);
  if (const clamp_status w = check_unet_ws(ws, ws_bytes, a.bytes, "clamp_unet_warm_start")) return w;
  cudaStream_t st = (cudaStream_t)stream;
  const long long n = (long long)nx * ny * nz;
  // four CTAs per SM: every CTA of the two element-wise passes adds all the partial sums
  const unsigned np = std::min(grid_for(n), 152u * 4);
  const bool vec = n % 4 == 0 && ((uintptr_t)r0 | (uintptr_t)r_init | (uintptr_t)a.xin | (uintptr_t)a.out) % 16 == 0;
  if (vec) k_sum_part<true><<<np, UT, 0, st>>>(r0, n, a.part);
  else k_sum_part<false><<<np, UT, 0, st>>>(r0, n, a.part);
  const double cols = (double)nx * ny;   // m = sum(r0) / (nx ny): energy per (x, y) column
  if (vec) k_scale_by_mean<true><<<np, UT, 0, st>>>(r0, n, a.part, (int)np, cols, a.xin);
  else k_scale_by_mean<false><<<np, UT, 0, st>>>(r0, n, a.part, (int)np, cols, a.xin);
  U_TRY(cudaGetLastError());
  clamp_status s = unet_forward(u, a.xin, 1, nx, ny, nz, a, st);
  if (s != CLAMP_OK) return s;
  if (vec) k_warm_map<true><<<np, UT, 0, st>>>(a.out, n, a.part, (int)np, cols, floor_rel, r_init);
  else k_warm_map<false><<<np, UT, 0, st>>>(a.out, n, a.part, (int)np, cols, floor_rel, r_init);
  U_TRY(cudaGetLastError());
  return CLAMP_OK;
}

extern "C" clamp_status clamp_unet_loss(clamp_unet* u, const float* x, const float* target, int32_t batch,
                                        int32_t nx, int32_t ny, int32_t nz, double* loss, void* ws, size_t ws_bytes,
                                        void* stream) {
  if (!u || !x || !target || !loss) return api_fail(CLAMP_EINVAL, "clamp_unet_loss: NULL argument");
  if (!on_unet_device(u, "clamp_unet_loss")) return CLAMP_EINVAL;
  if (!unet_shape_ok(batch, nx, ny, nz))
    return api_fail(CLAMP_EINVAL, "clamp_unet_loss: nx, ny, nz must be multiples of 4");
  const Acts a = acts_layout(u, batch, nx, ny, nz, ws, true);   // the loss gradient goes to gout
  if (const clamp_status w = check_unet_ws(ws, ws_bytes, a.bytes, "clamp_unet_loss")) return w;
  cudaStream_t st = (cudaStream_t)stream;
  clamp_status s = unet_forward(u, x, batch, nx, ny, nz, a, st);
  if (s != CLAMP_OK) return s;
  const long long N = (long long)batch * nx * ny * nz;
  const unsigned nb = grid_for(N);
  k_mse<<<nb, UT, 0, st>>>(a.out, target, a.gout, N, a.part);
  k_mse_final<<<1, UT, 0, st>>>(a.part, (int)nb, N, loss);
  U_TRY(cudaGetLastError());
  return CLAMP_OK;
}
