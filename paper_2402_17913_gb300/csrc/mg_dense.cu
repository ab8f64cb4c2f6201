// The coarse cycle as a dense matrix.
//
// One cycle on the levels kc .. L-1 from a zero guess is a fixed linear map
// of level kc's right-hand side: sweeps, transfers and the exact coarsest
// solve have no data-dependent step.  For a level of at most a couple of
// thousand cells its matrix (n x n floats, n^2 * 4 <= 16 MB, resident in L2)
// is written once at create, a column per unit vector run through the
// single-block coarse cycle, and a cycle then costs one matrix-vector product
// over all SMs instead of a chain of some twenty block barriers on one SM
// and, on grids whose sides are not powers of two, a dense coarsest inverse
// of up to 1000^2 read by that SM.  Measured per cycle (launch included):
// 21 -> 6.3 us on 256^3 (coarse levels 16^3 .. 4^3), 19 -> 8.2 us on 2048x1024,
// 69 -> 7.2 us on 1600x960 (coarsest 25x15), 890 -> 6.9 us on 144x144x192
// (coarsest 9x9x12).
#include <type_traits>

#include "coarse.cuh"
#include "launch.h"

namespace npmg {

namespace {

// Column j of the matrix into row j of `Mt` (one block per column): the
// coarse cycle of unit vector j.  `E` holds four zero arrays of 2 npad + 4
// floats with a single 1 at npad + s in array s, so that E + s (2 npad + 4) +
// npad + s - j is unit vector j and, with s = j mod 4, 16-byte aligned.
template <int DIM>
__global__ void __launch_bounds__(1024) k_dense_columns(const __grid_constant__ CoarseArgs a,
                                                        const float* __restrict__ E, int npad, int ld,
                                                        float* __restrict__ Mt, SolveState* __restrict__ st,
                                                        int total_floats) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int j = blockIdx.x, s = j & 3;
  coarse_cycle<DIM, float>(a, E + (size_t)s * (2 * npad + 4) + npad + s - j, Mt + (size_t)j * ld, st,
                           reinterpret_cast<float*>(smem_raw), total_floats);
}

__global__ void k_unit_vectors(float* __restrict__ E, int npad) {
  const int len = 2 * npad + 4;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 4 * len; i += gridDim.x * blockDim.x)
    E[i] = (i % len) == npad + i / len ? 1.f : 0.f;
}

// In-place transposition of the n x n matrix (row stride ld): a block swaps
// one 32 x 32 tile with its mirror image.
__global__ void __launch_bounds__(256) k_transpose(float* __restrict__ M, int n, int ld) {
  if (blockIdx.x < blockIdx.y) return;
  __shared__ float a[32][33], b[32][33];
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
  for (int k = threadIdx.x; k < 1024; k += 256) {
    const int r = k >> 5, c = k & 31;
    a[r][c] = y0 + r < n && x0 + c < n ? M[(size_t)(y0 + r) * ld + x0 + c] : 0.f;
    b[r][c] = x0 + r < n && y0 + c < n ? M[(size_t)(x0 + r) * ld + y0 + c] : 0.f;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 1024; k += 256) {
    const int r = k >> 5, c = k & 31;
    if (y0 + r < n && x0 + c < n) M[(size_t)(y0 + r) * ld + x0 + c] = b[c][r];
    if (x0 + r < n && y0 + c < n) M[(size_t)(x0 + r) * ld + y0 + c] = a[c][r];
  }
}

template <typename T>
__device__ __forceinline__ float4 ldb4(const T* __restrict__ b, int i) {
  if constexpr (std::is_same<T, float>::value) {
    return *reinterpret_cast<const float4*>(b + i);
  } else if constexpr (std::is_same<T, __half>::value) {
    const uint2 v = *reinterpret_cast<const uint2*>(b + i);
    const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
    const float2 q = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
    return make_float4(p.x, p.y, q.x, q.y);
  } else {
    const uint2 v = *reinterpret_cast<const uint2*>(b + i);
    const float2 p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 q = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(p.x, p.y, q.x, q.y);
  }
}

constexpr int kRowWarps = 8;   // warps (rows) per block
constexpr int kAhead = 16;     // float4 of its row a lane holds before b is needed (2048 columns)

}  // namespace

// y = M b, a warp per row.  Latency-bound: a lane's share of its row
// (up to 16 float4, the whole row for n <= 2048) is in flight before the
// wait for the previous kernel, since the matrix never changes, and b (shared
// by all rows) comes from L1/L2.  b may be read up to the next multiple of
// four (the buffers are padded to 256 bytes and hold finite values there; M's
// padding columns are 0).
template <typename T>
__global__ void __launch_bounds__(32 * kRowWarps) k_dense(int n, int ld, const float* __restrict__ M,
                                                          const T* __restrict__ b, T* __restrict__ y,
                                                          const int* __restrict__ done, int release) {
  if (release) chain_release();
  const int row = blockIdx.x * kRowWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const float4* __restrict__ m = reinterpret_cast<const float4*>(M + (size_t)min(row, n - 1) * ld);
  const int n4 = ld / 4;
  float4 r[kAhead];
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    const int i = lane + 32 * k;
    r[k] = i < n4 ? __ldg(m + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  chain_enter();
  if (done && *done) return;
  if (row >= n) return;  // whole warps
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    const int i = lane + 32 * k;
    const float4 v = i < n4 ? ldb4(b, 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
    acc[k & 3] = fmaf(r[k].w, v.w, fmaf(r[k].z, v.z, fmaf(r[k].y, v.y, fmaf(r[k].x, v.x, acc[k & 3]))));
  }
  for (int i = lane + 32 * kAhead; i < n4; i += 32) {
    const float4 q = __ldg(m + i), v = ldb4(b, 4 * i);
    acc[0] = fmaf(q.w, v.w, fmaf(q.z, v.z, fmaf(q.y, v.y, fmaf(q.x, v.x, acc[0]))));
  }
  float t = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) y[row] = cvt<T>(t);
}

int dense_stride(int n) { return (n + 3) & ~3; }
size_t dense_bytes(int n) { return (size_t)n * dense_stride(n) * sizeof(float); }
size_t dense_scratch_bytes(int n) { return 4 * (size_t)(2 * dense_stride(n) + 4) * sizeof(float); }

cudaError_t launch_transpose(float* M, int n, cudaStream_t s) {
  const int t = (n + 31) / 32;
  k_transpose<<<dim3(t, t), 256, 0, s>>>(M, n, dense_stride(n));
  return cudaGetLastError();
}

cudaError_t launch_dense_matrix(const CoarseArgs& a, size_t smem_bytes, int n, float* M, float* scratch,
                                SolveState* st, cudaStream_t s) {
  const int ld = dense_stride(n);
  const auto k = a.dim == 3 ? k_dense_columns<3> : k_dense_columns<2>;
  cudaError_t e = cudaMemsetAsync(M, 0, dense_bytes(n), s);
  int dev = 0, optin = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
  if (e != cudaSuccess) return e;
  k_unit_vectors<<<32, 256, 0, s>>>(scratch, ld);
  k<<<n, 1024, smem_bytes, s>>>(a, scratch, ld, ld, M, st, (int)(smem_bytes / sizeof(float)));
  e = cudaGetLastError();
  return e == cudaSuccess ? launch_transpose(M, n, s) : e;
}

template <typename T>
cudaError_t launch_dense(int dim, int n, const float* M, const void* b, void* y, const int* done, cudaStream_t s) {
  return launch_chain(k_dense<T>, (n + kRowWarps - 1) / kRowWarps, 32 * kRowWarps, 0, s, n, dense_stride(n), M,
                      (const T*)b, (T*)y, done, dim == 3 ? 1 : 0);
}
template cudaError_t launch_dense<float>(int, int, const float*, const void*, void*, const int*, cudaStream_t);
template cudaError_t launch_dense<__half>(int, int, const float*, const void*, void*, const int*, cudaStream_t);
template cudaError_t launch_dense<__nv_bfloat16>(int, int, const float*, const void*, void*, const int*, cudaStream_t);

}  // namespace npmg
