// Kernels of the learned initial-guess network: the BF16 implicit-GEMM 3D
// convolution on the fifth-generation tensor cores (forward and data
// gradient), the weight gradient on warp-level tensor-core MMAs, and the
// memory-bound glue (pooling, upsampling, skip sums, ReLU masks, input
// scaling, loss, Adam).
//
// Convolution as a GEMM.  For an output tile of M = 128 voxels (8 along x, 16
// along y, one z-plane) the 3x3x3 correlation with 16 input and 16 output
// channels is D[v][co] += sum_ci X[v + o_t][ci] * W[t][ci][co] over 27 taps t.
// A block walks a run of z-planes of one 8 x 16 column.  Input plane z adds
// to the output planes z - 1, z and z + 1 through the same nine shifted views
// (dy, dx), so one MMA of shape 128 x 48 x 16 does the three dz taps of a
// view: their accumulators are three slots of 16 TMEM columns, output plane p
// in slot p mod 3, and the 48 columns of B hold the taps dz in the cyclic
// order that puts each under its slot (a window of three in the stored
// sequence +1, 0, -1, +1, 0).  An input plane takes 9 MMAs instead of 27, and
// each view is read from shared memory once instead of three times, which is
// what bounds a 128 x 16 x 16 MMA (its 4 KB A tile at 128 bytes per SM cycle
// takes 32 cycles, its arithmetic about 9); an output's 27 taps still add up
// in the order of t.  After plane z the slot of output z - 1 is complete: the
// four warps read it with tcgen05.ld, write zeros to it for output z + 2, and
// apply the epilogue and store 32 bytes per voxel while the next plane's MMAs
// run.
//
// A plane with its one-voxel halo in x and y is copied once, two planes ahead,
// by 16-byte cp.async into [channel half][y][x][8 channels]: eight voxels of a
// line are then a 128-byte core matrix of the unswizzled K-major layout from
// any x on, so the A operands of all nine views are descriptors into the same
// copy (start address + 160 bytes per dy, + 16 per dx).  (Tiled TMA needs a
// copy per dx, swizzled, and moves it as 432 rows of 32 bytes per plane, which
// bound the layer at 62 us.)  Out-of-range voxels are zero-filled (the zero
// padding).  Measured on GB300, one 16 -> 16 layer of 8 x 64^3 voxels: 92 us with
// 27 MMAs per plane, 47 us now (134 MB in and out: 20 us at the copy rate; 84
// cycles per MMA on an SM with five blocks, against 44 for its operands at 128
// bytes per cycle); 256 x 128 x 128 voxels 184 -> 86 us.

// The data gradient is the same kernel with the mirrored, transposed taps
// (W'[26 - t][co][ci] = W[t][ci][co]).  The weight gradient
//     dW[t][ci][co] = sum_v X[v + o_t][ci] G[v][co]
// reduces over voxels and has M = 27 x 16 rows whose shared-memory views
// are not a single strided pattern, so it uses m16n8k16 MMAs fed by
// ldmatrix.trans, which gathers any eight 16-byte rows from the same
// swizzled [z][y][x][16 channels] tiles (the swizzle puts the 8 rows of one
// channel group in 8 different bank quads).
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "gn.h"
#include "tma_host.h"
#include "umma.cuh"

namespace npmg {
namespace gn {

namespace {

constexpr int kLine = (kTX + 2) * 16;                        // 8 channels of one line of voxels with halo
constexpr int kHalf = (kTY + 2) * kLine;                     // one channel half of a plane
constexpr int kStage = 2 * kHalf;
constexpr int kStages = 3;                                   // planes in flight or in use
constexpr int kChunks = kStage / 16;                         // 16-byte pieces of a plane
constexpr int kBView = 2 * 5 * 256;                          // B of one (dy, dx): [K half][five dz blocks][2][128 B]
constexpr int kBBytes = 9 * kBView;
constexpr int kConvSmem = kBBytes + kStages * kStage;
constexpr int kConvThreads = 128;
constexpr int kPer = (kChunks + kConvThreads - 1) / kConvThreads;
constexpr uint32_t kConvCols = 64;                           // TMEM columns (three accumulators of 16, a power of two)
static_assert(kTX == 8 && kTX * kTY == kConvThreads, "a line is a core matrix, one voxel per thread");
static_assert(kBBytes % 128 == 0 && kStage % 128 == 0, "operands start on 128-byte boundaries");

constexpr int kXTile = (kWTX + 2) * (kWTY + 2) * (kWTZ + 2) * 32;  // wgrad x tile with halo
constexpr int kGTile = kWTX * kWTY * kWTZ * 32;
constexpr int kWgSmem = kXTile + kGTile + 1024;
constexpr int kWgThreads = 288;  // 9 warps: warp w owns the taps of one (dy, dx), dz = -1, 0, 1
static_assert(kWElems % 32 == 0, "whole blocks of the reduction");
static_assert(kXTile % 256 == 0 && kGTile % 256 == 0, "swizzled TMA destinations stay 256-aligned");

// byte offset of channel group g of voxel v in a 32-byte-swizzled tile
// whose base is 256-byte aligned
__device__ __forceinline__ uint32_t sw32(uint32_t v, uint32_t g) { return v * 32u + ((g ^ ((v >> 2) & 1u)) << 4); }

struct ConvArgs {
  int nx, ny, nz, nn;
  int tx, ty;
  int zc, nzc;  // planes per z-run and runs per column
  long long nitems;
  void* out;
  const __nv_bfloat16* mask;
  const float* scale;
  int* err;
};

struct WgArgs {
  int nx, ny, nz, nn;
  int tx, ty, tz;
  long long ntiles;
  float* partials;
  int* err;
};

__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ bool bf_pos(uint32_t h16) { return !(h16 & 0x8000u) && (h16 & 0x7fffu); }

// 32 bytes to a 16-byte aligned address; one store (a whole sector) where the
// address is 32-byte aligned.
__device__ __forceinline__ void store32(void* p, const uint32_t (&q)[8]) {
  if (((uintptr_t)p & 31) == 0) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(q[0]), "r"(q[1]), "r"(q[2]),
                 "r"(q[3]), "r"(q[4]), "r"(q[5]), "r"(q[6]), "r"(q[7])
                 : "memory");
  } else {
    uint4* o = static_cast<uint4*>(p);
    o[0] = make_uint4(q[0], q[1], q[2], q[3]);
    o[1] = make_uint4(q[4], q[5], q[6], q[7]);
  }
}

template <int EPI>
__device__ __forceinline__ void store_epi(const ConvArgs& a, size_t vox, int n, const float (&v)[16],
                                          const uint4 (&m)[2]) {
  if (EPI == kEpiF32) {
    uint32_t q[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = __float_as_uint(v[8 * h + k]);
      store32(static_cast<float*>(a.out) + vox * kC + 8 * h, q);
    }
  } else if (EPI == kEpiOut0) {
    static_cast<float*>(a.out)[vox] = v[0] * (a.scale ? a.scale[n] : 1.f);
  } else {
    float w[16];
    if (EPI == kEpiMask) {
      const uint32_t mw[8] = {m[0].x, m[0].y, m[0].z, m[0].w, m[1].x, m[1].y, m[1].z, m[1].w};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        w[2 * k] = bf_pos(mw[k] & 0xffffu) ? v[2 * k] : 0.f;
        w[2 * k + 1] = bf_pos(mw[k] >> 16) ? v[2 * k + 1] : 0.f;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) w[k] = EPI == kEpiRelu ? fmaxf(v[k], 0.f) : v[k];
    }
    uint32_t q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = pack_bf2(w[2 * k], w[2 * k + 1]);
    store32(static_cast<__nv_bfloat16*>(a.out) + vox * kC, q);
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Persistent implicit-GEMM convolution (see the file comment).
template <int EPI>
__global__ void __launch_bounds__(kConvThreads) k_conv(const unsigned char* __restrict__ xin,
                                                     const unsigned char* __restrict__ wpack, ConvArgs a) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ __align__(8) uint64_t bar_mma;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t sB_u = smem_u32(dsm), sA_u = sB_u + kBBytes;

  // B of view v = (dy + 1) 3 + dx + 1, K half h, block q = 0 .. 4 (dz = +1, 0,
  // -1, +1, 0): the 256 bytes of packed tap (dz, v), half h
  for (int i = tid; i < kBBytes / 16; i += kConvThreads) {
    const int q = (i >> 4) % 5, h = (i / 80) & 1, v = i / 160;
    const int dz1 = (2 - q + 3) % 3;  // dz + 1
    cp_async16(sB_u + (uint32_t)i * 16u, wpack + (dz1 * 9 + v) * 512 + h * 256 + (i & 15) * 16, true);
  }
  const uint32_t hiA = (uint32_t)(smem_desc(0, kHalf, kLine) >> 32), hiB = (uint32_t)(smem_desc(0, 1280, 128) >> 32);
  const uint32_t loA = (uint32_t)smem_desc(sA_u, kHalf, kLine), loB = (uint32_t)smem_desc(sB_u, 1280, 128);
  if (tid == 0) {
    mbar_init(&bar_mma, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_slot, kConvCols);
    tmem_relinquish();
  }

  // A step is one input plane of an item = (x tile, y tile, z run, sample):
  // planes zr0 - 1 .. zr0 + count, `count` outputs.
  struct Step {
    long long item;
    int x0, y0, zr0, n, count, i;
  };
  auto open = [&](Step& p) {
    if (p.item >= a.nitems) return;
    long long r = p.item;
    p.x0 = (int)(r % a.tx) * kTX;
    r /= a.tx;
    p.y0 = (int)(r % a.ty) * kTY;
    r /= a.ty;
    p.zr0 = (int)(r % a.nzc) * a.zc;
    p.n = (int)(r / a.nzc);
    p.count = min(a.zc, a.nz - p.zr0);
    p.i = 0;
  };
  Step cur, ahead;  // the plane in work and the next one to fetch
  cur.item = blockIdx.x;
  open(cur);
  ahead = cur;
  // this thread's pieces of a plane: shared offsets, and for the item being
  // fetched the offsets in a plane (-1 outside it)
  uint32_t so[kPer];
  long long go[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int c = tid + k * kConvThreads, r = c % (2 * (kTX + 2));
    so[k] = (uint32_t)((r & 1) * kHalf + c / (2 * (kTX + 2)) * kLine + (r >> 1) * 16);
  }
  auto locate = [&]() {
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int c = tid + k * kConvThreads, r = c % (2 * (kTX + 2));
      const int x = ahead.x0 - 1 + (r >> 1), y = ahead.y0 - 1 + c / (2 * (kTX + 2));
      const bool in = x >= 0 && x < a.nx && y >= 0 && y < a.ny;
      go[k] = in ? ((long long)y * a.nx + x) * 32 + (r & 1) * 16 : -1;
    }
  };
  locate();
  // copy the next plane into `stage` (an empty group when none is left)
  auto fetch = [&](int stage) {
    if (ahead.item < a.nitems) {
      const int z = ahead.zr0 - 1 + ahead.i;
      const bool zin = z >= 0 && z < a.nz;
      const unsigned char* src = xin + ((size_t)ahead.n * a.nz + (zin ? z : 0)) * a.ny * a.nx * 32;
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (kChunks % kConvThreads == 0 || tid + k * kConvThreads < kChunks) {
          const bool on = zin && go[k] >= 0;
          cp_async16(sA_u + (uint32_t)(stage * kStage) + so[k], src + (on ? go[k] : 0), on);
        }
      if (++ahead.i >= ahead.count + 2) {
        ahead.item += gridDim.x;
        open(ahead);
        locate();
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int k = 0; k < kStages - 1; ++k) fetch(k);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot, lanes = (uint32_t)(warp * 32) << 16;
  constexpr uint32_t idesc = idesc_bf16(128, 48);
  tmem_zero16(tmem + lanes);  // slot 0, the first output's
  cp_async_wait<kStages - 2>();
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();

  int stage = 0, slot = 0;  // step mod kStages, step mod 3
  uint32_t ph_mma = 0;
  float v[16];
  uint4 msk[2];  // the output's mask, on its way while the next plane is set up
  size_t vox = 0;
  int vn = 0;
  bool have = false;
  while (cur.item < a.nitems) {
    if (tid == 0) {
      tc_fence_after();
      const uint32_t dA = loA + (uint32_t)(stage * kStage >> 4), dB = loB + (uint32_t)((2 - slot) * 256 >> 4);
#pragma unroll
      for (int t = 0; t < 9; ++t)
        umma_bf16(tmem, ((uint64_t)hiA << 32) | (dA + (uint32_t)((t / 3 * kLine + t % 3 * 16) >> 4)),
                  ((uint64_t)hiB << 32) | (dB + (uint32_t)(t * kBView >> 4)), idesc, 1u);
      umma_commit(&bar_mma);
    }
    // while the tensor core works: the plane kStages - 1 ahead into the stage
    // of the previous one, and the previous plane's output
    fetch(stage == 0 ? kStages - 1 : stage - 1);
    if (have) store_epi<EPI>(a, vox, vn, v, msk);
    const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar_mma, ph_mma));
    const int done = slot == 2 ? 0 : slot + 1;
    if (ok) {  // the whole warp
      tc_fence_after();
      // the slot of output i - 2 (its last tap was this plane's) is read and
      // set to zero for the output that starts with the next plane
      tmem_ld16(tmem + lanes + (uint32_t)(done * 16), v);
      tmem_zero16(tmem + lanes + (uint32_t)(done * 16));
    }
    const int x = cur.x0 + (tid & (kTX - 1)), y = cur.y0 + tid / kTX, z = cur.zr0 + cur.i - 2;
    have = ok && cur.i >= 2 && x < a.nx && y < a.ny;
    vox = (((size_t)cur.n * a.nz + (have ? z : 0)) * a.ny + y) * a.nx + x;
    vn = cur.n;
    if (EPI == kEpiMask && have) {
      msk[0] = __ldg(reinterpret_cast<const uint4*>(a.mask + vox * kC));
      msk[1] = __ldg(reinterpret_cast<const uint4*>(a.mask + vox * kC) + 1);
    }
    cp_async_wait<kStages - 2>();  // the next plane has landed
    fence_proxy_async_smem();
    tc_fence_before();
    if (__syncthreads_or(!ok)) {
      // MMAs that never end: report it, give them one more bounded wait, stop
      if (tid == 0) {
        atomicExch(a.err, 2);
        mbar_wait_bounded(&bar_mma, ph_mma);
      }
      have = false;
      break;
    }
    if (++cur.i >= cur.count + 2) {
      cur.item += gridDim.x;
      open(cur);
    }
    slot = done;
    ph_mma ^= 1u;
    if (++stage == kStages) stage = 0;
  }
  if (have) store_epi<EPI>(a, vox, vn, v, msk);
  cp_async_wait<0>();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, kConvCols);
}

// Weight gradient: per-block partial sums of dW over the block's tiles.
// Staged (32-byte swizzled): x as [z][y][18][16 ch] covering x0 - 1 ..
// x0 + 16, g as [z][y][16][16 ch].  Bound by the shared-memory fragment loads:
// a warp keeps one (dy, dx) and walks a column of lines along z, so that one
// fragment of x serves the three dz taps (against the g fragments of the
// planes around it) and a tile's column takes 10 loads for 24 MMAs instead
// of 16 (a warp per (dz, dy) with a load of x per dx): 8 x 64^3 voxels
// 96 -> 76 us.
__global__ void __launch_bounds__(kWgThreads, 4) k_wgrad(const __grid_constant__ CUtensorMap xmap,
                                                    const __grid_constant__ CUtensorMap gmap, WgArgs a) {
  extern __shared__ unsigned char dsm[];
  __shared__ __align__(8) uint64_t bar;
  const uint32_t pad = (1024u - (smem_u32(dsm) & 1023u)) & 1023u;
  unsigned char* sX = dsm + pad;
  unsigned char* sG = sX + kXTile;
  const uint32_t sX_u = smem_u32(sX), sG_u = smem_u32(sG);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int dy = warp / 3 - 1, dx = warp % 3 - 1;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  float acc[3][2][4];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[j][q][k] = 0.f;
  // ldmatrix row of this lane: matrix mi = lane / 8, row rr = lane % 8.
  // G (B operand): matrix mi = (channel group mi / 2, voxels 8 (mi % 2) ..).
  // X (A operand): matrix mi = (channel group mi % 2, voxels 8 (mi / 2) ..).
  const int mi = lane >> 3, rr = lane & 7;
  const uint32_t gk = (uint32_t)((mi & 1) * 8 + rr), gg = (uint32_t)(mi >> 1);
  const uint32_t xk = (uint32_t)((mi >> 1) * 8 + rr), xg = (uint32_t)(mi & 1);
  uint32_t phase = 0;
  for (long long tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    long long r = tile;
    const int bx = (int)(r % a.tx);
    r /= a.tx;
    const int by = (int)(r % a.ty);
    r /= a.ty;
    const int bz = (int)(r % a.tz);
    const int n = (int)(r / a.tz);
    const int x0 = bx * kWTX, y0 = by * kWTY, z0 = bz * kWTZ;
    if (tid == 0) {
      mbar_arrive_expect_tx(&bar, kXTile + kGTile);
      tma_load_5d(sX, &xmap, &bar, 0, x0 - 1, y0 - 1, z0 - 1, n);
      tma_load_5d(sG, &gmap, &bar, 0, x0, y0, z0, n);
    }
    const bool ok = mbar_wait_bounded(&bar, phase);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicExch(a.err, 3);
      mbar_wait_bounded(&bar, phase);
      break;
    }
    for (int yi = 0; yi < kWTY; ++yi) {
      uint32_t b[kWTZ][4];
#pragma unroll
      for (int zi = 0; zi < kWTZ; ++zi)
        ldsm_x4_trans(sG_u + sw32((uint32_t)((zi * kWTY + yi) * kWTX) + gk, gg), b[zi]);
      const uint32_t xl = (uint32_t)((yi + dy + 1) * (kWTX + 2) + dx + 1) + xk;
#pragma unroll
      for (int p = 0; p < kWTZ + 2; ++p) {  // x plane z0 - 1 + p = g plane zi + dz
        uint32_t av[4];
        ldsm_x4_trans(sX_u + sw32(xl + (uint32_t)(p * (kWTY + 2) * (kWTX + 2)), xg), av);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int zi = p - j;  // dz = j - 1
          if (zi < 0 || zi >= kWTZ) continue;
          mma_16816(acc[j][0], av, b[zi][0], b[zi][1]);
          mma_16816(acc[j][1], av, b[zi][2], b[zi][3]);
        }
      }
    }
    __syncthreads();
    phase ^= 1;
  }
  // accumulator fragment: c0, c1 = (row g, cols 2q, 2q+1), c2, c3 = row g + 8
  float* P = a.partials + (size_t)blockIdx.x * kWElems;
  const int g = lane >> 2, c2 = (lane & 3) * 2;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int t = 9 * j + warp;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int co = q * 8 + c2;
      *reinterpret_cast<float2*>(P + (t * kC + g) * kC + co) = make_float2(acc[j][q][0], acc[j][q][1]);
      *reinterpret_cast<float2*>(P + (t * kC + g + 8) * kC + co) = make_float2(acc[j][q][2], acc[j][q][3]);
    }
  }
}

// dw (+)= scale * the sum of the blocks' partials: a block of 256 threads sums
// 32 elements, eight threads each taking every eighth block's partial with
// sixteen loads in flight, their sums added in order (608 blocks, 16.8 MB: one
// thread per element walked its 608 partials in 21 us, now 6.6 us).
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* __restrict__ partials, int nblocks,
                                                      float* __restrict__ dw, float scale, int accumulate) {
  __shared__ float sh[8][32];
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), c = threadIdx.x >> 5;
  const float* __restrict__ p = partials + e;
  float s = 0.f;
  int b = c;
  for (; b + 8 * 15 < nblocks; b += 8 * 16) {
    float v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __ldg(p + (size_t)(b + 8 * k) * kWElems);
#pragma unroll
    for (int k = 0; k < 16; ++k) s += v[k];
  }
  for (; b < nblocks; b += 8) s += __ldg(p + (size_t)b * kWElems);
  sh[c][threadIdx.x & 31] = s;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  s = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) s += sh[k][threadIdx.x];
  dw[e] = (accumulate ? dw[e] : 0.f) + scale * s;
}

// ---------------------------------------------------------------------------
// glue kernels; one thread per (voxel, channel group of 8) = one uint4
__device__ __forceinline__ void unpack8(uint4 u, float (&f)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[k]));
    f[2 * k] = p.x;
    f[2 * k + 1] = p.y;
  }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  return make_uint4(pack_bf2(f[0], f[1]), pack_bf2(f[2], f[3]), pack_bf2(f[4], f[5]), pack_bf2(f[6], f[7]));
}
__device__ __forceinline__ void mask8(uint4 act, float (&f)[8]) {
  const uint32_t w[4] = {act.x, act.y, act.z, act.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!bf_pos(w[k] & 0xffffu)) f[2 * k] = 0.f;
    if (!bf_pos(w[k] >> 16)) f[2 * k + 1] = 0.f;
  }
}

// Element counts below 2^31 (every grid-stride index then fits 32 bits) use
// 32-bit index arithmetic: the 64-bit divisions by the extents bound these
// kernels, which otherwise stream (residual loss of 8 x 64^3 voxels 50 -> 19 us,
// with its neighbours loaded before use; skip sums 17.4 -> 13.7 us).
static bool idx32(size_t total) { return total < (size_t)1 << 31; }
#define GN_INDEXED(total, K, grid, block, s, ...)                        \
  do {                                                                   \
    if (idx32(total)) K<unsigned><<<grid, block, 0, s>>>(__VA_ARGS__);   \
    else K<size_t><<<grid, block, 0, s>>>(__VA_ARGS__);                  \
  } while (0)

// index helpers: element (n, z, y, x, group) of a level with dims (nx, ny, nz)
struct Lv {
  int nx, ny, nz;
  __device__ size_t u4(size_t n, int z, int y, int x, int g) const {
    return ((((n * nz + z) * ny + y) * nx + x) << 1) + g;
  }
};

template <typename I>
__global__ void k_pool(const uint4* __restrict__ fine, uint4* __restrict__ coarse, Lv F, Lv Cc, size_t total) {
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int g = (int)(i & 1);
    I v = i >> 1;
    const int x = (int)(v % (I)Cc.nx);
    v /= (I)Cc.nx;
    const int y = (int)(v % (I)Cc.ny);
    v /= (I)Cc.ny;
    const int z = (int)(v % (I)Cc.nz);
    const I n = v / (I)Cc.nz;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float f[8];
      unpack8(fine[F.u4(n, 2 * z + (c >> 2), 2 * y + ((c >> 1) & 1), 2 * x + (c & 1), g)], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] += f[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] *= 0.125f;
    coarse[i] = pack8(s);
  }
}

template <typename I>
__global__ void k_up_add(const uint4* __restrict__ coarse, const uint4* __restrict__ fine, uint4* __restrict__ out,
                         Lv F, Lv Cc, size_t total) {
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int g = (int)(i & 1);
    I v = i >> 1;
    const int x = (int)(v % (I)F.nx);
    v /= (I)F.nx;
    const int y = (int)(v % (I)F.ny);
    v /= (I)F.ny;
    const int z = (int)(v % (I)F.nz);
    const I n = v / (I)F.nz;
    float a[8], b[8];
    unpack8(coarse[Cc.u4(n, z >> 1, y >> 1, x >> 1, g)], a);
    unpack8(fine[i], b);
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] += b[k];
    out[i] = pack8(a);
  }
}

template <typename I>
__global__ void k_upbwd_mask(const uint4* __restrict__ gfine, const uint4* __restrict__ act, uint4* __restrict__ out,
                             Lv F, Lv Cc, size_t total) {
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int g = (int)(i & 1);
    I v = i >> 1;
    const int x = (int)(v % (I)Cc.nx);
    v /= (I)Cc.nx;
    const int y = (int)(v % (I)Cc.ny);
    v /= (I)Cc.ny;
    const int z = (int)(v % (I)Cc.nz);
    const I n = v / (I)Cc.nz;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float f[8];
      unpack8(gfine[F.u4(n, 2 * z + (c >> 2), 2 * y + ((c >> 1) & 1), 2 * x + (c & 1), g)], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] += f[k];
    }
    mask8(act[i], s);
    out[i] = pack8(s);
  }
}

template <typename I>
__global__ void k_poolbwd_add_mask(const uint4* __restrict__ gskip, const uint4* __restrict__ gcoarse,
                                   const uint4* __restrict__ act, uint4* __restrict__ out, Lv F, Lv Cc,
                                   size_t total) {
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int g = (int)(i & 1);
    I v = i >> 1;
    const int x = (int)(v % (I)F.nx);
    v /= (I)F.nx;
    const int y = (int)(v % (I)F.ny);
    v /= (I)F.ny;
    const int z = (int)(v % (I)F.nz);
    const I n = v / (I)F.nz;
    float a[8], b[8];
    unpack8(gskip[i], a);
    unpack8(gcoarse[Cc.u4(n, z >> 1, y >> 1, x >> 1, g)], b);
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] += 0.125f * b[k];
    mask8(act[i], a);
    out[i] = pack8(a);
  }
}

__device__ __forceinline__ const float* field(const float* base, const Fields& f, int n) {
  const size_t s = f.idx ? (size_t)f.idx[n] : (size_t)n;
  return base + s * f.stride;
}

// per-sample sums of squares of b (blockIdx.z = 0) and p (= 1): grid
// (blocks, n, 2), partials[(field * n + sample) * blocks + block]
__global__ void k_sumsq(Fields f, size_t vox, float* __restrict__ partials) {
  __shared__ double sh[32];
  const float* a = field(blockIdx.z ? f.p : f.b, f, blockIdx.y);
  float acc = 0.f;
  // few blocks per sample: sixteen loads in flight per thread (256 x 128 x 128:
  // 117 -> 18.5 us), added in the order of i
  const size_t step = (size_t)gridDim.x * blockDim.x;
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (; i + 15 * step < vox; i += 16 * step) {
    float v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __ldg(a + i + k * step);
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fmaf(v[k], v[k], acc);
  }
  for (; i < vox; i += step) acc = fmaf(a[i], a[i], acc);
  const double t = block_sum((double)acc, sh);
  if (threadIdx.x == 0) partials[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = (float)t;
}

// rms / inverse rms per (field, sample), pooled over the samples if asked;
// 1 for an all-zero field
__global__ void k_rms_final(const float* __restrict__ partials, int nblk, size_t vox, int n, int pooled,
                            float* __restrict__ rms, float* __restrict__ inv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n) return;
  const int fld = i / n, s = i % n;
  double acc = 0.0;
  const int s0 = pooled ? 0 : s, s1 = pooled ? n : s + 1;
  for (int q = s0; q < s1; ++q)
    for (int b = 0; b < nblk; b += 16) {  // nblk is a multiple of 16
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = partials[(fld * n + q) * nblk + b + k];
#pragma unroll
      for (int k = 0; k < 16; ++k) acc += (double)v[k];
    }
  const double r = sqrt(acc / ((double)vox * (s1 - s0)));
  rms[i] = r > 0.0 ? (float)r : 1.f;
  inv[i] = r > 0.0 ? (float)(1.0 / r) : 1.f;
}

template <typename I>
__global__ void k_pack_input(Fields f, const float* __restrict__ inv, uint4* __restrict__ x0, size_t vox, int n) {
  const size_t total = vox * (size_t)n;
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int s = (int)(i / (I)vox);
    const I v = i - (I)s * (I)vox;
    const float bv = field(f.b, f, s)[v] * inv[s], pv = field(f.p, f, s)[v] * inv[n + s];
    const uint32_t q[8] = {pack_bf2(bv, pv), 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    store32(x0 + 2 * (size_t)i, q);
  }
}

template <typename I>
__global__ void k_loss_grad(const float* __restrict__ y, Fields f, const float* __restrict__ inv,
                            uint4* __restrict__ gy, size_t vox, int n, double* __restrict__ partials) {
  __shared__ double sh[32];
  const size_t total = vox * (size_t)n;
  float acc = 0.f;
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int s = (int)(i / (I)vox);
    const I v = i - (I)s * (I)vox;
    const float d = y[i] - field(f.t, f, s)[v] * inv[s];
    acc = fmaf(d, d, acc);
    const uint32_t q[8] = {pack_bf2(d, 0.f), 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    store32(gy + 2 * (size_t)i, q);
  }
  const double t = block_sum((double)acc, sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

__global__ void k_sum_partials(const double* __restrict__ partials, int nblk, double scale,
                               double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) acc += partials[b];
  const double t = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = scale * t;
}

// (A_crop v)_c * h^2 on a fluid cell c: sum over fluid face neighbours n in
// the crop of (v_c - v_n).
__device__ __forceinline__ float crop_stencil(const float* v, const float* fl, size_t i, int x, int y, int z, int nx,
                                              int ny, int nz) {
  // every load before the first use (a missing neighbour loads the cell)
  const size_t sy = (size_t)nx, sz = (size_t)nx * ny;
  const bool in[6] = {x > 0, x < nx - 1, y > 0, y < ny - 1, z > 0, z < nz - 1};
  const size_t j[6] = {in[0] ? i - 1 : i,  in[1] ? i + 1 : i,  in[2] ? i - sy : i,
                       in[3] ? i + sy : i, in[4] ? i - sz : i, in[5] ? i + sz : i};
  float vn[6], fn[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    vn[k] = v[j[k]];
    fn[k] = fl ? fl[j[k]] : 1.f;
  }
  const float vc = v[i];
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k)
    if (in[k] && fn[k] > 0.5f) acc += vc - vn[k];
  return acc;
}

template <typename I>
__global__ void k_residual(const float* __restrict__ y, Fields f, const float* __restrict__ inv, int nx, int ny,
                           int nz, int n, float inv_h2, float* __restrict__ r, double* __restrict__ partials) {
  __shared__ double sh[32];
  const size_t vox = (size_t)nx * ny * nz, total = vox * n;
  float acc = 0.f;
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int s = (int)(i / (I)vox);
    const I v = i - (I)s * (I)vox;
    const I row = v / (I)nx;
    const int x = (int)(v % (I)nx), yy = (int)(row % (I)ny), z = (int)(row / (I)ny);
    const float* fl = f.fluid ? field(f.fluid, f, s) : nullptr;
    const bool inner = x > 0 && x < nx - 1 && yy > 0 && yy < ny - 1 && z > 0 && z < nz - 1;
    float rv = 0.f;
    if (inner && (!fl || fl[v] > 0.5f)) {
      rv = crop_stencil(y + (size_t)s * vox, fl, v, x, yy, z, nx, ny, nz) * inv_h2 - field(f.b, f, s)[v] * inv[s];
      acc = fmaf(rv, rv, acc);
    }
    r[i] = rv;
  }
  const double t = block_sum((double)acc, sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

template <typename I>
__global__ void k_apply_crop(const float* __restrict__ r, Fields f, int nx, int ny, int nz, int n, float inv_h2,
                             uint4* __restrict__ gy) {
  const size_t vox = (size_t)nx * ny * nz, total = vox * n;
  for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < (I)total; i += (I)(gridDim.x * blockDim.x)) {
    const int s = (int)(i / (I)vox);
    const I v = i - (I)s * (I)vox;
    const I row = v / (I)nx;
    const int x = (int)(v % (I)nx), yy = (int)(row % (I)ny), z = (int)(row / (I)ny);
    const float* fl = f.fluid ? field(f.fluid, f, s) : nullptr;
    float g = 0.f;
    if (!fl || fl[v] > 0.5f) g = crop_stencil(r + (size_t)s * vox, fl, v, x, yy, z, nx, ny, nz) * inv_h2;
    const uint32_t q[8] = {pack_bf2(g, 0.f), 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    store32(gy + 2 * (size_t)i, q);
  }
}

// fwd operand: [t][ci / 8][co][ci % 8]; data-gradient operand: tap 26 - t,
// [co / 8][ci][co % 8] (K = output channel, N = input channel).
__global__ void k_adam_pack(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ grad, int update, AdamArgs a, __nv_bfloat16* __restrict__ wf,
                            __nv_bfloat16* __restrict__ wd) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= kLayers * kWElems) return;
  float wv = w[e];
  if (update) {
    const float g = grad[e];
    const float mv = a.b1 * m[e] + a.omb1 * g;
    const float vv = a.b2 * v[e] + a.omb2 * g * g;
    m[e] = mv;
    v[e] = vv;
    wv -= a.lr * (mv * a.c1) / (sqrtf(vv * a.c2) + a.eps);
    w[e] = wv;
  }
  const int k = e / kWElems, rem = e % kWElems;
  const int t = rem / (kC * kC), ci = (rem / kC) % kC, co = rem % kC;
  const __nv_bfloat16 h = __float2bfloat16_rn(wv);
  const size_t lb = (size_t)k * kTaps;
  wf[((lb + t) * 2 + (ci >> 3)) * 128 + co * 8 + (ci & 7)] = h;
  wd[((lb + (kTaps - 1 - t)) * 2 + (co >> 3)) * 128 + ci * 8 + (co & 7)] = h;
}

__global__ void k_pack_layer(const float* __restrict__ w, __nv_bfloat16* __restrict__ wf,
                             __nv_bfloat16* __restrict__ wd) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= kWElems) return;
  const int t = e / (kC * kC), ci = (e / kC) % kC, co = e % kC;
  const __nv_bfloat16 h = __float2bfloat16_rn(w[e]);
  wf[(t * 2 + (ci >> 3)) * 128 + co * 8 + (ci & 7)] = h;
  wd[((kTaps - 1 - t) * 2 + (co >> 3)) * 128 + ci * 8 + (co & 7)] = h;
}

__global__ void k_crop(const float* __restrict__ b, const float* __restrict__ p_next, const float* __restrict__ dp,
                       const uint8_t* __restrict__ solid, long long fx, long long fy, long long cx, long long cy,
                       long long cz, long long ox, long long oy, long long oz, float* __restrict__ dst) {
  const size_t vox = (size_t)(cx * cy * cz);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < vox; i += (size_t)gridDim.x * blockDim.x) {
    const long long x = (long long)(i % cx), y = (long long)((i / cx) % cy), z = (long long)(i / (cx * cy));
    const size_t src = (size_t)(((z + oz) * fy + (y + oy)) * fx + (x + ox));
    const float d = dp[src];
    dst[i] = b[src];
    dst[vox + i] = p_next[src] - d;
    dst[2 * vox + i] = d;
    dst[3 * vox + i] = (solid && solid[src]) ? 0.f : 1.f;
  }
}

// Resident blocks of `kernel` on all SMs, from its shared memory (dynamic +
// static + the per-block reservation), registers and threads.
template <typename K>
int occupancy_blocks(K kernel, int threads, size_t smem) {
  int dev = 0, nsm = 0, smem_sm = 0, reserved = 0, regs_sm = 0, thr_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return nsm;
  const size_t per_block = smem + fa.sharedSizeBytes + (size_t)reserved;
  int occ = (int)((size_t)smem_sm / per_block);
  const int regs_block = ((fa.numRegs * 32 + 255) / 256) * 256 * ((threads + 31) / 32);
  if (regs_block > 0) occ = std::min(occ, regs_sm / regs_block);
  occ = std::min(occ, thr_sm / threads);
  return nsm * std::max(occ, 1);
}

int grid_1d(size_t work, int threads = 256) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const size_t want = (work + threads - 1) / threads;
  const size_t cap = (size_t)nsm * 8;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace

std::atomic<int64_t> g_launches{0};

bool encode_act(CUtensorMap* m, const void* base, const Dims& d, int bx, int by, int bz) {
  auto fn = (PFN_cuTensorMapEncodeTiled_v12000)tensor_map_encoder();
  if (!fn || ((uintptr_t)base & 15)) return false;
  cuuint64_t gdim[5] = {(cuuint64_t)kC, (cuuint64_t)d.nx, (cuuint64_t)d.ny, (cuuint64_t)d.nz, (cuuint64_t)d.n};
  cuuint64_t gstride[4] = {(cuuint64_t)kC * 2, (cuuint64_t)kC * 2 * d.nx, (cuuint64_t)kC * 2 * d.nx * d.ny,
                           (cuuint64_t)kC * 2 * d.nx * d.ny * d.nz};
  cuuint32_t box[5] = {(cuuint32_t)kC, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, 1};
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), gdim, gstride, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename K>
static int grid_for(K kernel, int threads, int smem) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return -1;
  return occupancy_blocks(kernel, threads, smem);
}

static int device_sms() {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return nsm > 0 ? nsm : 1;
}

template <int EPI>
static cudaError_t conv_epi(const void* x, const void* wpack, ConvArgs a, cudaStream_t s) {
  static int grid_cache = 0;
  if (!grid_cache) grid_cache = grid_for(k_conv<EPI>, kConvThreads, kConvSmem);
  if (grid_cache < 0) return cudaErrorInvalidValue;
  // z-runs: a run of c outputs costs c + 2 planes.  The tensor core's operand
  // reads bound an SM that has two or more runs in work (its runs' planes add
  // up: 0.36 us a plane on 256 x 128 x 128 voxels); a lone run is bound by its
  // own chain (0.68 us a plane on 64 x 64 x 256 in one and in two runs), so it
  // counts 1.7 of those planes; 1.5 to 1.9 give the same runs on all shapes
  // below.  Whole gn_conv3d calls, 44 us of each not the convolution, in
  // 1 / 2 / 4 / 6 / 8 / 16 runs: 8 x 64^3 (4 chosen) 98 / 96 / 89 / 96 / 95 / 96 us,
  // 256 x 128 x 128 (4) 157 / 144 / 134 / 145 / 133 / 134, 64^3 (8) 83 / 59 / 49 / 47 /
  // 46 / 46, 64 x 64 x 256 (9: 70) 219 / 132 / 82 / 82 / 69 / 69, 96 x 80 x 64 (5: 54)
  // 83 / 59 / 57 / 56 / 57 / 57, 3 x 100 x 60 x 40 (4) 71 / 66 / 58 / 59 / 60.
  const long long columns = (long long)a.tx * a.ty * a.nn;
  const long long nsm = device_sms();
  double best = -1.0;
  for (int runs = 1; runs <= (a.nz + 3) / 4; ++runs) {
    const int zc = (a.nz + runs - 1) / runs;
    const long long items = columns * ((a.nz + zc - 1) / zc);
    const double cost = std::max((double)((items + nsm - 1) / nsm), 1.7) * (zc + 2);
    if (best >= 0.0 && cost >= best) continue;
    best = cost;
    a.zc = zc;
    a.nzc = (a.nz + zc - 1) / zc;
    a.nitems = items;
  }
  const long long g = a.nitems < grid_cache ? a.nitems : grid_cache;
  k_conv<EPI><<<(unsigned)(g > 0 ? g : 1), kConvThreads, kConvSmem, s>>>((const unsigned char*)x,
                                                                          (const unsigned char*)wpack, a);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_conv(const void* x, const void* wpack, void* out, int epi, const void* mask, const float* scale,
                        const Dims& d, int* err, cudaStream_t s) {
  if (d.n <= 0 || d.vox() == 0) return cudaSuccess;
  if (((uintptr_t)x | (uintptr_t)wpack) & 15) return cudaErrorInvalidValue;
  ConvArgs a;
  a.nx = d.nx;
  a.ny = d.ny;
  a.nz = d.nz;
  a.nn = d.n;
  a.tx = (d.nx + kTX - 1) / kTX;
  a.ty = (d.ny + kTY - 1) / kTY;
  a.zc = a.nzc = 0;
  a.nitems = 0;
  a.out = out;
  a.mask = (const __nv_bfloat16*)mask;
  a.scale = scale;
  a.err = err;
  switch (epi) {
    case kEpiF32: return conv_epi<kEpiF32>(x, wpack, a, s);
    case kEpiRelu: return conv_epi<kEpiRelu>(x, wpack, a, s);
    case kEpiLin: return conv_epi<kEpiLin>(x, wpack, a, s);
    case kEpiMask: return conv_epi<kEpiMask>(x, wpack, a, s);
    case kEpiOut0: return conv_epi<kEpiOut0>(x, wpack, a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_wgrad(const void* x, const void* g, float* partials, int max_blocks, int* nblocks, const Dims& d,
                         int* err, cudaStream_t s) {
  static int grid_cache = 0;
  if (!grid_cache) grid_cache = grid_for(k_wgrad, kWgThreads, kWgSmem);
  if (grid_cache < 0) return cudaErrorInvalidValue;
  CUtensorMap xm, gm;
  if (!encode_act(&xm, x, d, kWTX + 2, kWTY + 2, kWTZ + 2) || !encode_act(&gm, g, d, kWTX, kWTY, kWTZ))
    return cudaErrorInvalidValue;
  WgArgs a;
  a.nx = d.nx;
  a.ny = d.ny;
  a.nz = d.nz;
  a.nn = d.n;
  a.tx = (d.nx + kWTX - 1) / kWTX;
  a.ty = (d.ny + kWTY - 1) / kWTY;
  a.tz = (d.nz + kWTZ - 1) / kWTZ;
  a.ntiles = (long long)a.tx * a.ty * a.tz * d.n;
  a.partials = partials;
  a.err = err;
  long long gsz = a.ntiles < grid_cache ? a.ntiles : grid_cache;
  if (gsz > max_blocks) gsz = max_blocks;
  if (gsz < 1) gsz = 1;
  *nblocks = (int)gsz;
  k_wgrad<<<(unsigned)gsz, kWgThreads, kWgSmem, s>>>(xm, gm, a);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_wgrad_reduce(const float* partials, int nblocks, float* dw, float scale, bool accumulate,
                                cudaStream_t s) {
  k_wgrad_reduce<<<kWElems / 32, 256, 0, s>>>(partials, nblocks, dw, scale, accumulate ? 1 : 0);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

static Lv lv_of(const Dims& d, int shift) { return Lv{d.nx >> shift, d.ny >> shift, d.nz >> shift}; }

cudaError_t launch_pool(const void* fine, void* coarse, const Dims& d, cudaStream_t s) {
  const size_t total = d.vox() / 8 * d.n * 2;
  GN_INDEXED(total, k_pool, grid_1d(total), 256, s, (const uint4*)fine, (uint4*)coarse, lv_of(d, 0), lv_of(d, 1), total);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_up_add(const void* coarse, const void* fine, void* out, const Dims& d, cudaStream_t s) {
  const size_t total = d.vox() * d.n * 2;
  GN_INDEXED(total, k_up_add, grid_1d(total), 256, s, (const uint4*)coarse, (const uint4*)fine, (uint4*)out, lv_of(d, 0),
                                          lv_of(d, 1), total);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_upbwd_mask(const void* gfine, const void* act_coarse, void* out_coarse, const Dims& d,
                              cudaStream_t s) {
  const size_t total = d.vox() / 8 * d.n * 2;
  GN_INDEXED(total, k_upbwd_mask, grid_1d(total), 256, s, (const uint4*)gfine, (const uint4*)act_coarse, (uint4*)out_coarse,
                                              lv_of(d, 0), lv_of(d, 1), total);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_poolbwd_add_mask(const void* gskip, const void* gcoarse, const void* act, void* out,
                                    const Dims& d, cudaStream_t s) {
  const size_t total = d.vox() * d.n * 2;
  GN_INDEXED(total, k_poolbwd_add_mask, grid_1d(total), 256, s, (const uint4*)gskip, (const uint4*)gcoarse, (const uint4*)act,
                                                    (uint4*)out, lv_of(d, 0), lv_of(d, 1), total);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_rms(const Fields& f, const Dims& d, bool pooled, float* partials, float* rms, float* inv_rms,
                       cudaStream_t s) {
  const int nblk = 64;
  k_sumsq<<<dim3(nblk, d.n, 2), 256, 0, s>>>(f, d.vox(), partials);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  k_rms_final<<<(2 * d.n + 127) / 128, 128, 0, s>>>(partials, nblk, d.vox(), d.n, pooled ? 1 : 0, rms, inv_rms);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_pack_input(const Fields& f, const float* inv_rms, void* x0, const Dims& d, cudaStream_t s) {
  GN_INDEXED(d.vox() * d.n, k_pack_input, grid_1d(d.vox() * d.n), 256, s, f, inv_rms, (uint4*)x0, d.vox(), d.n);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_loss_grad(const float* y, const Fields& f, const float* inv_rms, void* gy, double* partials,
                             double* loss, const Dims& d, cudaStream_t s) {
  const int g = grid_1d(d.vox() * d.n);
  GN_INDEXED(d.vox() * d.n, k_loss_grad, g, 256, s, y, f, inv_rms, (uint4*)gy, d.vox(), d.n, partials);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  k_sum_partials<<<1, 256, 0, s>>>(partials, g, 0.5 / ((double)d.vox() * d.n), loss);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_residual_loss_grad(const float* y, const Fields& f, const float* inv_rms, float inv_h2, float* r,
                                      void* gy, double* partials, double* loss, const Dims& d, cudaStream_t s) {
  const int g = grid_1d(d.vox() * d.n);
  GN_INDEXED(d.vox() * d.n, k_residual, g, 256, s, y, f, inv_rms, d.nx, d.ny, d.nz, d.n, inv_h2, r, partials);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  k_sum_partials<<<1, 256, 0, s>>>(partials, g, 0.5 / ((double)d.vox() * d.n), loss);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  GN_INDEXED(d.vox() * d.n, k_apply_crop, g, 256, s, r, f, d.nx, d.ny, d.nz, d.n, inv_h2, (uint4*)gy);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_adam_pack(float* w, float* m, float* v, const float* grad, bool update, AdamArgs a, void* wf,
                             void* wd, cudaStream_t s) {
  k_adam_pack<<<(kLayers * kWElems + 255) / 256, 256, 0, s>>>(w, m, v, grad, update ? 1 : 0, a,
                                                              (__nv_bfloat16*)wf, (__nv_bfloat16*)wd);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_crop(const float* b, const float* p_next, const float* dp, const uint8_t* solid,
                        const int64_t full[3], const int64_t crop[3], const int64_t origin[3], float* dst,
                        cudaStream_t s) {
  const size_t vox = (size_t)(crop[0] * crop[1] * crop[2]);
  k_crop<<<grid_1d(vox), 256, 0, s>>>(b, p_next, dp, solid, full[0], full[1], crop[0], crop[1], crop[2], origin[0],
                                      origin[1], origin[2], dst);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_pack_layer(const float* w, void* wf, void* wd, cudaStream_t s) {
  k_pack_layer<<<(kWElems + 255) / 256, 256, 0, s>>>(w, (__nv_bfloat16*)wf, (__nv_bfloat16*)wd);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace gn
}  // namespace npmg
