// Internal definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdio.h>

#include "../../include/npmg.h"

namespace npmg {

constexpr int kMaxLevels = 16;
constexpr int kMaxHalo = 3;            // max Jacobi sweeps fused per tile pass
constexpr int kThreads = 256;          // threads per tile block
constexpr int kHistory = 32;

// Cell byte of a masked level: bit 7 = fluid; bits 0-1, 2-3, 4-5 = number of
// links per axis (x, y, z) that enter the diagonal of A (a fluid neighbour
// inside the domain, or a Dirichlet domain face).  Solid cells hold 0.
constexpr uint8_t kFluidBit = 0x80;

// One grid level as the kernels see it (passed by value).
struct LevelDev {
  int nx, ny, nz;        // cells per axis (nz = 1 in 2D)
  float wx, wy, wz;      // operator weights: c / h_a^2 (c = h_0x^2)
  int bcD;               // bit f set when face f (x-,x+,y-,y+,z-,z+) is Dirichlet
  const uint8_t* cell;   // cell bytes, or nullptr when the level has no solid
};

// Device-resident control block of one solve.  Written by the "last block"
// of the reduction kernels, read by every kernel of the next phase.
struct SolveState {
  // parameters (set at solve start)
  double tol, inner_floor;
  int max_inner, max_outer, krylov, n_fluid;
  // refinement loop
  double bnorm2;         // ||b||^2
  double relres, relres0;
  double sigma;          // d = sigma * d' for the current inner solve
  double eta;            // relative tolerance of the current inner solve
  int outer, outer_done, status, stall;
  double hist[kHistory];
  // inner CG
  int inner_done, it, iters_total, first;
  double r0norm2, rz, rz_old, alpha, beta, rnorm2, pAp;
  // reduction counters (one per reducing kernel family)
  unsigned int counter[8];
  // device-side solve loop: the float-float buffer holding the iterate, and
  // the checks and bodies run by the loop's conditional nodes
  int cur;
  unsigned int loop_checks, loop_bodies, loop_outer;
};

enum Counter { kCntInit = 0, kCntOuter = 1, kCntRZ = 2, kCntPAP = 3, kCntRR = 4, kCntMisc = 5 };

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  The kernels of a solve's launch chain
// (level legs, coarse block, CG updates) are launched with a programmatic
// dependency on the previous one, so that their launch overlaps its drain;
// each first waits until the preceding grid has completed and its writes
// are visible (a no-op when it was launched without the dependency).
// Only constants of the handle (cell bytes, the dense coarse matrix) may be
// read before this call, and nothing written.  Most grids release their
// successor at exit: measured on GB300, successors parked on the SMs from the
// start of large grids made the 2D and 3D solves 5-8% slower, while the
// release at exit makes the 2D flow step about 1.5% faster.
__device__ __forceinline__ void chain_enter() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// Release the successor now, so that its blocks start, form what does not
// depend on this grid and wait for its end.  For the small 3D levels and the
// coarse matrix between them, whose grids leave room on the SMs and whose
// successors have work before their wait (geometry, diagonals, the matrix
// rows): 256x128x128 FE flow step 3.41 -> 3.27 ms, masked 96x80x64 cycle 30.1
// -> 27.7 us, 256^3 solve 9.85 -> 9.76 ms.  In 2D the same release measured
// 2-5% slower (448x576 1.01 -> 1.06 ms), so 2D grids keep the release at exit.
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// storage conversions
template <typename T> __device__ __forceinline__ float ld(const T* p, size_t i);
template <> __device__ __forceinline__ float ld<float>(const float* p, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float ld<__half>(const __half* p, size_t i) { return __half2float(p[i]); }
template <> __device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16* p, size_t i) { return __bfloat162float(p[i]); }

template <typename T> __device__ __forceinline__ T cvt(float v);
template <> __device__ __forceinline__ float cvt<float>(float v) { return v; }
template <> __device__ __forceinline__ __half cvt<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------
// Deterministic reductions: warp shuffles, then a fixed-order block tree;
// grid totals by the last block to finish (fixed-order sum of the partials).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block; the result is valid in thread 0.  `sh` holds >= 32
// doubles.  Every thread of the block must call it.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (lane < nw) ? sh[lane] : 0.0;
    v = warp_sum(v);
  }
  return v;
}

__device__ __forceinline__ unsigned linear_block() {
  return blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
}

// Float-float pair (hi + lo, about 48 significant bits) of a reduction:
// two_sum (Knuth) of the high parts, the low parts added to its error.
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float s = a.x + b.x, bb = s - a.x;
  const float e = ((a.x - (s - bb)) + (b.x - bb)) + (a.y + b.y);
  const float h = s + e;
  return make_float2(h, e - (h - s));
}

// Sum of the first `n` lanes' pairs, valid in lane 0 (lanes from n on add
// nothing; they may not exist).
__device__ __forceinline__ float2 warp_pair_sum(float2 v, int lane, int n) {
  const unsigned mask = n >= 32 ? 0xffffffffu : (1u << n) - 1u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float2 t = make_float2(__shfl_down_sync(mask, v.x, o), __shfl_down_sync(mask, v.y, o));
    if (lane + o < n) v = pair_add(v, t);
  }
  return v;
}

// Sum over the block, valid in thread 0; `sh` holds >= 32 pairs.
__device__ __forceinline__ float2 block_pair_sum(float2 v, float2* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  v = warp_pair_sum(v, lane, min(32, (int)blockDim.x - 32 * w));
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) v = warp_pair_sum(lane < nw ? sh[lane] : make_float2(0.f, 0.f), lane, min(32, (int)blockDim.x));
  return v;
}

// One more arrival at the counter: the block's writes before it are visible
// to the block that sees the last count (release), and that block's later
// reads are ordered after it (acquire; the other threads' by the barrier
// that follows).
__device__ __forceinline__ unsigned arrive(unsigned int* counter) {
  unsigned t;
  asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
  return t;
}

// Each block contributes `v`, a sum of float32 terms kept in float32 (or as a
// pair) by each thread; returns true in every thread of the last block to arrive, with the
// grid total in *total (valid in thread 0).  Latency-bound tail of every
// reducing kernel: the sums are float-float pairs (the terms themselves carry
// 2^-24), since one float64 warp instruction holds its sub-partition's pipe
// for 64 cycles on GB300 and a float64 tree is ten dependent ones per level,
// and the arrival is one acquire-release atomic instead of a fence on each
// side.  Against the float64 tree with fences: 448x576 solve 1.25 -> 1.23 ms,
// 128^3 2.38 -> 2.31 ms, 2048x1024 flow step 1.845 -> 1.820 ms.
__device__ __forceinline__ bool grid_sum_last(float2 v, double* partials, unsigned int* counter, double* total) {
  __shared__ float2 sh[32];
  __shared__ bool last;
  float2* part = reinterpret_cast<float2*>(partials);
  const float2 s = block_pair_sum(v, sh);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  if (threadIdx.x == 0) {
    part[linear_block()] = s;
    last = arrive(counter) == nb - 1;
  }
  __syncthreads();
  if (!last) return false;
  float2 acc = make_float2(0.f, 0.f);
  for (unsigned i = threadIdx.x; i < nb; i += blockDim.x) acc = pair_add(acc, __ldcg(part + i));
  const float2 r = block_pair_sum(acc, sh);
  if (threadIdx.x == 0) {
    *total = (double)r.x + (double)r.y;
    *counter = 0u;
  }
  return true;
}

// The same for a thread's float32 sum of CG (r', z or A' p with r' scaled to
// an rms near 1, but r' of a guess far from the solution is as much larger as
// its residual is): summed 2^32 times smaller, so that what fits float32 in a
// thread fits it over any grid.
__device__ __forceinline__ bool grid_sum_last(float v, double* partials, unsigned int* counter, double* total) {
  const bool last = grid_sum_last(make_float2(v * 0x1p-32f, 0.f), partials, counter, total);
  if (last && threadIdx.x == 0) *total *= 0x1p32;
  return last;
}

// The same for float64 contributions.
__device__ __forceinline__ bool grid_sum_last(double v, double* partials, unsigned int* counter, double* total) {
  __shared__ double sh[32];
  __shared__ bool last;
  const double s = block_sum(v, sh);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  if (threadIdx.x == 0) {
    partials[linear_block()] = s;
    last = arrive(counter) == nb - 1;
  }
  __syncthreads();
  if (!last) return false;
  double acc = 0.0;
  for (unsigned i = threadIdx.x; i < nb; i += blockDim.x) acc += __ldcg(partials + i);
  const double r = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    *total = r;
    *counter = 0u;
  }
  return true;
}

// ---------------------------------------------------------------------------
// Diagonal of the scaled operator at a cell.
__device__ __forceinline__ int axis_count(int g, int n, int bcD, int face_lo) {
  // links along one axis for an unmasked level: 2 inside, minus Neumann faces
  return 2 - ((g == 0) & !((bcD >> face_lo) & 1)) - ((g == n - 1) & !((bcD >> (face_lo + 1)) & 1));
}

template <int DIM, bool MASKED>
__device__ __forceinline__ float diag_at(const LevelDev& L, int gx, int gy, int gz, uint8_t m) {
  if (MASKED) {
    float d = L.wx * (float)(m & 3) + L.wy * (float)((m >> 2) & 3);
    if (DIM == 3) d += L.wz * (float)((m >> 4) & 3);
    return d;
  } else {
    float d = L.wx * (float)axis_count(gx, L.nx, L.bcD, 0) + L.wy * (float)axis_count(gy, L.ny, L.bcD, 2);
    if (DIM == 3) d += L.wz * (float)axis_count(gz, L.nz, L.bcD, 4);
    return d;
  }
}

// Host-side error helper.
void set_error(const char* fmt, ...);

#define NPMG_CUDA(call)                                                        \
  do {                                                                         \
    cudaError_t e_ = (call);                                                   \
    if (e_ != cudaSuccess) {                                                   \
      ::npmg::set_error("%s:%d %s: %s", __FILE__, __LINE__, #call,             \
                        cudaGetErrorString(e_));                               \
      return MG_ERR_CUDA;                                                      \
    }                                                                          \
  } while (0)

}  // namespace npmg
