// unet_tc.cu -- the U-Net's 3x3x3 convolutions on the 5th-generation tensor cores (tcgen05),
// BF16 operands and FP32 accumulation: the forward conv and, with flipped weights, the data
// gradient of the backward pass (Sec. III-C's U-Net prior and the learned warm start).
//
// The U-Net keeps FP32 channel-planar tensors [batch][C][nz][ny][nx] (pooling, transposed
// convs, skips and the weight gradient read them), so this kernel converts on the fly: it
// loads FP32 halo voxels, rounds them to BF16 (round to nearest even, as the CUDA-core BF16
// path does) and writes them in the no-swizzle K-major layout, and its epilogue writes FP32
// planar outputs with bias and optional ReLU.
//
// Implicit GEMM: an MMA's M = 128 output voxels are a patch of 8 x voxels in 16 rows of one
// plane, N = C_out, K = 16 input channels of one tap.  A staged input plane (16 channels) is
// [2 channel groups][18 rows][XW + 2 voxels] of 16 bytes (8 channels); eight x voxels in a row
// are one core matrix, the next row lies one row pitch further, so a tap (dz, dy, dx) is a
// plane and an offset of the A operand's start, whatever the volume's width: one copy of the
// halo serves all 27 taps.
//
// A CTA owns XW x 16 voxels of up to ZT planes (their accumulators fill 256 TMEM columns, so
// two CTAs share an SM) and, for every 16-channel chunk, marches along z: each plane is
// loaded and rounded once per chunk into a ring of four, and completes the three planes one
// output plane needs.  Seven warps stage: the next plane's loads are in flight in registers
// while a plane's MMAs run, and it is stored once the MMAs of the plane before have completed.
// The eighth warp issues the MMAs (27 per patch, committed to an mbarrier) meanwhile: issued by
// one of the staging threads they held up its warp, and with it all eight at the next barrier,
// for most of the time.  CTAs are persistent: TMEM and barriers are set up once, and the next
// tile's first plane is loaded under the current tile's last MMAs.  Waits are bounded and set an
// error bit instead of hanging.
//
// For one output the MMAs accumulate chunk by chunk in tap order, as the earlier kernel's did
// (three shifted halo copies staged per output plane, no overlap), so results are
// the same bit for bit.  Bound: a 4 KB A operand read per MMA (32 clocks for N = 16; 0.20 ms
// per 16 -> 16 conv at 256x256x128) and the FP32 planes' traffic (0.16 ms); measured there, mean of
// two 16 -> 16 and one 32 -> 16: 0.69 ms with the MMAs issued by a staging thread, now 0.56 (32 -> 32 at
// half size 0.23 -> 0.20).  What is left is the latency of a plane's round (load, store, barrier,
// MMAs) at two CTAs per SM, which registers and shared memory allow (16 -> 16 at 128x128x64: tensor pipe 10 % busy,
// issue slots 39 %, DRAM 1.3 TB/s).
#include "../../include/clamp.h"
#include "clamp_internal.cuh"
#include "clamp_kernels.cuh"
#include "packed.cuh"
#include "tc_core.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace clamp {
namespace unet_tc {

constexpr int UNT = 256;   // threads per CTA
constexpr int UST = 224;   // of these stage; the last warp issues the MMAs
constexpr uint32_t kWaitLimit = 1u << 22;
constexpr int TROWS = 16;  // rows of a tile

// XW: x voxels of a tile.
template <int COUT, int XW>
struct UtCfg {
  static constexpr int P = XW + 2, HR = TROWS + 2, TX = XW / 8;   // row pitch, staged rows, patches per plane
  static constexpr int CG_VEC = HR * P;                           // 16-byte vectors of one channel group of a plane
  static constexpr int PLANE_VEC = 2 * CG_VEC;
  static constexpr int ZT = 256 / (TX * COUT);                    // output planes whose accumulators fit 256 columns
  static constexpr int W_VEC = 27 * 2 * COUT;                     // a chunk's weights [tap][group][C_out]
  static constexpr int TASKS = (PLANE_VEC + UST - 1) / UST;       // staging tasks (8 channels of a voxel) per thread
  static constexpr size_t SMEM = 1024 + 16 * (size_t)(4 * PLANE_VEC + W_VEC) + 64;
  static_assert(ZT >= 1 && TX * COUT * ZT == 256, "TMEM");
  static_assert(2 * (SMEM + 1024) <= 228 * 1024, "two CTAs per SM");
};

// wpk[((c * 27 + tap) * 2 + cg) * C_out + co] = BF16 W[co][16 c + 8 cg + k][tap], k = 0..7.
__global__ void k_pack_weights(const float* __restrict__ W, int ci_n, int co_n, uint4* __restrict__ wpk) {
  const int total = (ci_n / 16) * 27 * 2 * co_n;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int co = e % co_n, cg = (e / co_n) % 2, tap = (e / (2 * co_n)) % 27, c = e / (54 * co_n);
    const int ci0 = 16 * c + 8 * cg;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = W[((long long)co * ci_n + ci0 + k) * 27 + tap];
    wpk[e] = make_uint4(bf16x2(v[0], v[1]), bf16x2(v[2], v[3]), bf16x2(v[4], v[5]), bf16x2(v[6], v[7]));
  }
}

template <int COUT, int XW>
__global__ void __launch_bounds__(UNT, 2)
    k_conv3_unet_tc(const float* __restrict__ in, long long in_bs, int ci_n, float* __restrict__ out,
                    long long out_bs, const uint4* __restrict__ wpk, const float* __restrict__ bias, int relu, int B,
                    int nx, int ny, int nz, int zt, int* err) {
  using Cfg = UtCfg<COUT, XW>;
  constexpr int P = Cfg::P, TX = Cfg::TX;
  extern __shared__ unsigned char ut_smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)ut_smem_raw + 1023) & ~(uintptr_t)1023);
  uint4* s_a = reinterpret_cast<uint4*>(base);          // ring of four planes
  uint4* s_w = s_a + 4 * Cfg::PLANE_VEC;                // the chunk's weights
  uint64_t* mbar = reinterpret_cast<uint64_t*>(s_w + Cfg::W_VEC);   // [2]: commits alternate between them
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 2);
  int* abort_flag = reinterpret_cast<int*>(tslot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long plane = (long long)nx * ny, n = plane * nz;
  const int tiles_x = nx / XW, tiles_y = (ny + TROWS - 1) / TROWS, tiles_z = (nz + zt - 1) / zt;
  const int ntiles = B * tiles_z * tiles_y * tiles_x;
  const int nchunks = ci_n / 16, per_chunk = zt + 2;

  if (tid == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
    *abort_flag = 0;
  }
  if (warp == 0) {
    tc::tmem_alloc(tslot, 256);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = *tslot;
  const uint64_t a0 = tc::make_desc(tc::smem_addr(s_a), Cfg::CG_VEC * 16, P * 16);
  const uint64_t b0 = tc::make_desc(tc::smem_addr(s_w), COUT * 16, 128);

  // the tile being computed, and the (tile, chunk, plane) of the arrival being loaded
  struct Pos {
    int x0, y0, z0, b;
  };
  auto at = [&](int t) {
    Pos p;
    p.x0 = t % tiles_x * XW;
    t /= tiles_x;
    p.y0 = t % tiles_y * TROWS;
    t /= tiles_y;
    p.z0 = t % tiles_z * zt;
    p.b = t / tiles_z;
    return p;
  };
  float v[Cfg::TASKS][8];
  // arrival (chunk c, plane p of the march: z0 - 1 + p) of tile `t` into registers, zeros outside
  auto load = [&](const Pos& t, int c, int p) {
    const int gz = t.z0 - 1 + p;
    const bool zin = gz >= 0 && gz < nz;
    const float* src = in + (long long)t.b * in_bs + (long long)(16 * c) * n + (zin ? gz * plane : 0LL);
#pragma unroll
    for (int k = 0; k < Cfg::TASKS; ++k) {
      const int e = tid + k * UST;
      const int cg = e / Cfg::CG_VEC, r = e % Cfg::CG_VEC;
      const int gx = t.x0 + r % P - 1, gy = t.y0 + r / P - 1;
      const bool ok = e < Cfg::PLANE_VEC && zin && gx >= 0 && gx < nx && gy >= 0 && gy < ny;
      const float* q = src + (ok ? (long long)(8 * cg) * n + (long long)gy * nx + gx : 0LL);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[k][j] = ok ? __ldg(q + (long long)j * n) : 0.f;
    }
  };
  auto store = [&](uint32_t slot) {
#pragma unroll
    for (int k = 0; k < Cfg::TASKS; ++k) {
      const int e = tid + k * UST;
      if (e < Cfg::PLANE_VEC)
        s_a[slot * Cfg::PLANE_VEC + e] = make_uint4(bf16x2(v[k][0], v[k][1]), bf16x2(v[k][2], v[k][3]),
                                                    bf16x2(v[k][4], v[k][5]), bf16x2(v[k][6], v[k][7]));
    }
  };
  auto weights = [&](int c) {
    const uint4* src = wpk + (long long)c * Cfg::W_VEC;
    for (int e = tid; e < Cfg::W_VEC; e += UST) cp_async16(&s_w[e], &src[e]);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // MMAs of output plane o of the tile: planes in ring slots g - 2, g - 1, g
  auto issue = [&](uint32_t g, int c, int o) {
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, COUT);
#pragma unroll 1
    for (int dz = 0; dz < 3; ++dz) {
      const uint64_t ad = a0 + (uint64_t)(((g + 2 + dz) & 3u) * Cfg::PLANE_VEC);   // slot (g - 2 + dz) mod 4
      const uint64_t bd = b0 + (uint64_t)(dz * 9 * 2 * COUT);
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
          for (int t = 0; t < TX; ++t)
            tc::mma_bf16(tbase + (uint32_t)((o * TX + t) * COUT), ad + (uint64_t)(dy * P + dx + 8 * t),
                         bd + (uint64_t)((dy * 3 + dx) * 2 * COUT), idesc,
                         (c > 0 || dz > 0 || dy > 0 || dx > 0) ? 1u : 0u);
    }
  };
  auto epilogue = [&](const Pos& t) {
    const int q = warp & 3, hh = warp >> 2;
    const int gy = t.y0 + 4 * q + (lane >> 3);
    const uint32_t trow = tbase + ((uint32_t)(32 * q) << 16);
    const int units = min(zt, nz - t.z0) * TX;
    for (int u = hh; u < units; u += 2) {   // u = o TX + patch; every lane of the warp loads TMEM
      const int gz = t.z0 + u / TX, gx = t.x0 + 8 * (u % TX) + (lane & 7);
      float* o = out + (long long)t.b * out_bs + gz * plane + (long long)gy * nx + gx;
#pragma unroll
      for (int j = 0; j < COUT / 16; ++j) {
        float r[16];
        tc::tmem_ld_x16(trow + (uint32_t)(u * COUT + 16 * j), r);
        if (gy < ny) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            float w = r[k] + (bias ? __ldg(&bias[16 * j + k]) : 0.f);
            if (relu) w = fmaxf(w, 0.f);
            o[(long long)(16 * j + k) * n] = w;
          }
        }
      }
    }
  };

  uint32_t g = 0;         // arrivals stored (this one's ring slot: g mod 4)
  uint32_t issued = 0;    // commits issued; commit k is on mbar[k & 1], phase k >> 1
  uint32_t waited = 0;    // commits waited for
  bool aborted = false;
  // bounded wait (thread 0) for every commit but the newest `keep`
  auto drain = [&](uint32_t keep) {
    if (tid == 0)
      for (uint32_t k = waited; k + keep < issued; ++k)
        if (!tc::mbar_wait_bounded(&mbar[k & 1u], (k >> 1) & 1u, kWaitLimit)) {
          *abort_flag = 1;
          break;
        }
    if (issued > keep && issued - keep > waited) waited = issued - keep;
  };
  const bool stager = tid < UST;
  int tile = blockIdx.x;   // < ntiles: the grid has at most a CTA per tile
  bool pending = false;    // the previous tile's epilogue is not done (its MMAs may be in flight)
  if (stager) {
    load(at(tile), 0, 0);
    weights(0);
    store(0);
  }
  tc::fence_proxy_async();
  __syncthreads();
  while (tile < ntiles && !aborted) {
    const int next = tile + (int)gridDim.x;
    const Pos cur = at(tile);
    for (int i = 0; i < nchunks * per_chunk; ++i, ++g) {
      const int c = i / per_chunk, p = i % per_chunk;
      // the next arrival's loads
      const bool last = i + 1 == nchunks * per_chunk;
      const bool more = !last || next < ntiles;
      if (stager) {
        if (!last) load(cur, (i + 1) / per_chunk, (i + 1) % per_chunk);
        else if (more) load(at(next), 0, 0);
      }
      const bool did = p >= 2 && cur.z0 + p - 2 < nz;
      if (did) {
        ++issued;
        if (!stager) {
          if (tc::elect_one()) {
            tc::fence_after_sync();
            issue(g, c, p - 2);
            tc::mma_commit(&mbar[(issued - 1) & 1u]);
          }
          __syncwarp();
        }
      }
      // the slot of arrival g + 1 held arrival g - 3, last read by the MMAs of arrival g - 1
      drain(did ? 1u : 0u);
      if (did) {
        if (stager) asm volatile("bar.sync 1, %0;" ::"n"(UST) : "memory");
      } else {
        __syncthreads();
      }
      tc::fence_after_sync();
      if ((did && !stager) || *abort_flag == 0) {   // a wait that gave up: nothing more is written, all leave below
        if (p == 0 && nchunks > 1 && (c > 0 || pending) && stager) weights(c);   // the previous chunk's MMAs are done
        if (p == 0 && pending) {
          epilogue(at(tile - (int)gridDim.x));
          pending = false;
        }
        if (more && stager) store((g + 1) & 3u);
        if (p <= 1) asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      tc::fence_proxy_async();
      tc::fence_before_sync();
      __syncthreads();
      if (*abort_flag != 0) {
        aborted = true;
        break;
      }
    }
    pending = true;
    tile = next;
  }
  if (!aborted && pending) {
    drain(0);
    __syncthreads();
    tc::fence_after_sync();
    if (*abort_flag == 0) epilogue(at(tile - (int)gridDim.x));
    else aborted = true;
  }
  if (aborted && tid == 0) {
    if (err) atomicOr(err, 2);
    // MMAs in flight get a bounded wait before TMEM is freed
    if (issued > 0) tc::mbar_wait_bounded(&mbar[(issued - 1) & 1u], ((issued - 1) >> 1) & 1u, kWaitLimit);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, 256);
}

}  // namespace unet_tc

using namespace unet_tc;

bool unet_conv3_tc_supported(int ci, int co, int nx, int ny) {
  if (ci < 16 || ci % 16 != 0 || (co != 16 && co != 32 && co != 64)) return false;
  return nx == 16 ? ny % 8 == 0 : nx % 32 == 0 && ny % 4 == 0;
}

size_t unet_conv3_tc_wpk_bytes(int ci, int co) { return (size_t)(ci / 16) * 27 * 2 * co * 16; }

template <int COUT, int XW>
static cudaError_t launch_tile(const float* in, long long in_bs, int ci, float* out, long long out_bs,
                               const uint4* wpk, const float* bias, bool relu, int B, int nx, int ny, int nz, int* err,
                               cudaStream_t st) {
  using Cfg = UtCfg<COUT, XW>;
  auto kern = k_conv3_unet_tc<COUT, XW>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
  if (e != cudaSuccess) return e;
  // fewer planes per tile (more halo planes, more CTAs) until two CTAs per SM have work
  const long long cols = (long long)B * (nx / XW) * ((ny + TROWS - 1) / TROWS);
  int zt = std::min(Cfg::ZT, nz);
  while (zt > 1 && cols * ((nz + zt - 1) / zt) < 2 * 152) zt = (zt + 1) / 2;
  const long long ntiles = cols * ((nz + zt - 1) / zt);
  kern<<<(unsigned)std::min(ntiles, 2LL * 152), UNT, Cfg::SMEM, st>>>(in, in_bs, ci, out, out_bs, wpk, bias, relu ? 1 : 0, B,
                                                                     nx, ny, nz, zt, err);
  return cudaGetLastError();
}

cudaError_t unet_conv3_tc(const float* in, long long in_bs, int ci, float* out, long long out_bs, int co,
                          const float* W, const float* bias, bool relu, int B, int nx, int ny, int nz, uint4* wpk,
                          int* err, cudaStream_t st) {
  if (!unet_conv3_tc_supported(ci, co, nx, ny)) return cudaErrorInvalidValue;
  const int total = (ci / 16) * 27 * 2 * co;
  k_pack_weights<<<(total + 255) / 256, 256, 0, st>>>(W, ci, co, wpk);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // tiles are 32 voxels wide where the level allows it; at 64 outputs 16, which leaves TMEM for
  // two planes per tile and shared memory for two CTAs per SM
  const bool wide = nx % 32 == 0;
  switch (co) {
    case 16:
      return wide ? launch_tile<16, 32>(in, in_bs, ci, out, out_bs, wpk, bias, relu, B, nx, ny, nz, err, st)
                  : launch_tile<16, 16>(in, in_bs, ci, out, out_bs, wpk, bias, relu, B, nx, ny, nz, err, st);
    case 32:
      return wide ? launch_tile<32, 32>(in, in_bs, ci, out, out_bs, wpk, bias, relu, B, nx, ny, nz, err, st)
                  : launch_tile<32, 16>(in, in_bs, ci, out, out_bs, wpk, bias, relu, B, nx, ny, nz, err, st);
    default: return launch_tile<64, 16>(in, in_bs, ci, out, out_bs, wpk, bias, relu, B, nx, ny, nz, err, st);
  }
}

}  // namespace clamp
