// The coarse cycle as a dense matrix.
//
// One cycle on the levels kc .. L-1 from a zero guess is a fixed linear map
// of level kc's right-hand side: sweeps, transfers and the exact coarsest
// solve have no data-dependent step.  For a level of at most a couple of
// thousand cells its matrix (n x n floats, n^2 * 4 <= 16 MB, resident in L2)
// is written once at create, a column per unit vector run through the cycle
// in float-float, and a cycle then costs one matrix-vector product
// over all SMs instead of a chain of some twenty block barriers on one SM
// and, on grids whose sides are not powers of two, a dense coarsest inverse
// of up to 1000^2 read by that SM.  Measured per cycle (launch included):
// 21 -> 6.3 us on 256^3 (coarse levels 16^3 .. 4^3), 19 -> 8.2 us on 2048x1024,
// 69 -> 7.2 us on 1600x960 (coarsest 25x15), 890 -> 6.9 us on 144x144x192
// (coarsest 9x9x12).
#include <type_traits>

#include "coarse.cuh"
#include "launch.h"
#include "refine.cuh"

namespace npmg {

namespace {

constexpr int kColT = 256;  // threads of a column's block

// Arrays of one level in the block's shared memory: x, x', b (float-float,
// padded with a zero ring as in coarse.cuh) and the cell bytes (0 on the
// ring); d, 1 / d and omega / d by link counts (0 where there are none).
struct DLev {
  CGeo g;
  float wx, wy, wz;
  float2 *x, *y, *b;
  const float2 *d, *id, *w;
  uint8_t* m;
};
constexpr int kTabs = 3 * 64;  // pairs of a level's tables

__device__ __forceinline__ ff get(const float2* p, int i) { return {p[i].x, p[i].y}; }
__device__ __forceinline__ void put(float2* p, int i, ff v) { p[i] = make_float2(v.hi, v.lo); }
__device__ __forceinline__ ff to_ff(double v) {
  const float hi = (float)v;
  return {hi, (float)(v - (double)hi)};
}
__device__ __forceinline__ ff scale(ff a, float w) {
  const float p = a.hi * w;
  return quick_two_sum(p, fmaf(a.lo, w, fmaf(a.hi, w, -p)));
}

__device__ __forceinline__ DLev d_level(const CoarseArgs& a, int l, float2* tab, float2* arr, uint8_t* bytes) {
  DLev v;
  const LevelDev& L = a.lv[l];
  v.g = cgeo(L, a.off[l]);
  v.wx = L.wx;
  v.wy = L.wy;
  v.wz = L.wz;
  const int P = v.g.WH * (v.g.nz + (v.g.nz > 1 ? 2 : 0)), o = a.off[l] / 4;  // padded cells, and those before
  v.x = arr + 3 * o;
  v.y = v.x + P;
  v.b = v.y + P;
  v.d = tab + kTabs * l;
  v.id = v.d + 64;
  v.w = v.id + 64;
  v.m = bytes + o;
  return v;
}

template <int DIM>
__device__ __forceinline__ ff d_nb(const DLev& v, const float2* x, int p) {
  ff nb = ff_add(scale(ff_add(get(x, p - 1), get(x, p + 1)), v.wx),
                 scale(ff_add(get(x, p - v.g.W), get(x, p + v.g.W)), v.wy));
  if (DIM == 3) nb = ff_add(nb, scale(ff_add(get(x, p - v.g.WH), get(x, p + v.g.WH)), v.wz));
  return nb;
}

// f(i, p, entry of the tables or -1 off the fluid) on every cell, then a
// barrier.
template <typename F>
__device__ __forceinline__ void d_cells(const DLev& v, F&& f) {
  for (int i = threadIdx.x; i < v.g.n; i += kColT) {
    int x, y, z;
    v.g.xyz(i, x, y, z);
    const int p = v.g.pad(x, y, z), m = v.m[p];
    f(i, p, m ? m & 63 : -1, x, y, z);
  }
  __syncthreads();
}

__device__ __forceinline__ void d_swap(DLev& v) {
  float2* t = v.x;
  v.x = v.y;
  v.y = t;
}

template <int DIM>
__device__ __forceinline__ void d_sweep(DLev& v, ff keep) {
  d_cells(v, [&](int, int p, int q, int, int, int) {
    const ff zero = {0.f, 0.f};
    put(v.y, p, q < 0 ? zero : ff_add(ff_mul(get(v.x, p), keep),
                                      ff_mul(ff_add(get(v.b, p), d_nb<DIM>(v, v.x, p)), get(v.w, q))));
  });
  d_swap(v);
}

// Column j of the matrix into row j of `Mt` (one block per column): the
// coarse cycle (coarse_cycle's steps) of unit vector j in float-float with the
// float64 coarsest inverse, rounded to float32 once.  The columns of a float32
// cycle carried its roundings into every product: a cycle on 64^2 was 0.9e-7
// of its result off, 0.6e-7 with these (0.8e-7 to 1.4e-7 launch by launch).
// 48 bits are enough for that, and one float64 instruction holds its pipe as
// long as 64 float32 ones: creating a 64^2 handle takes 0.46 ms so, 0.58 with
// float64 columns, 0.49 with float32 ones.  256 threads, so that an SM works
// on several columns.
template <int DIM>
__global__ void __launch_bounds__(kColT) k_dense_columns(const __grid_constant__ CoarseArgs a,
                                                        const double* __restrict__ inv, double omega, double s,
                                                        float* __restrict__ Mt, int ld) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int j = blockIdx.x, last = a.nlev - 1, nc = a.ncoarse;
  const bool saw = a.pre < 0;
  float* __restrict__ out = Mt + (size_t)j * ld;
  if (last == 0 && !saw) {  // the inverse itself
    for (int i = threadIdx.x; i < nc; i += kColT) out[i] = (float)inv[(size_t)j * nc + i];
    return;
  }
  float2* tab = reinterpret_cast<float2*>(smem_raw);
  float2* arr = tab + kTabs * a.nlev;
  int cells = 0;
  for (int l = 0; l < a.nlev; ++l) {
    const CGeo g = cgeo(a.lv[l], 0);
    cells += g.WH * (g.nz + (g.nz > 1 ? 2 : 0));
  }
  uint8_t* bytes = reinterpret_cast<uint8_t*>(arr + 3 * cells);
  for (int i = threadIdx.x; i < 3 * cells; i += kColT) arr[i] = make_float2(0.f, 0.f);
  for (int i = threadIdx.x; i < cells; i += kColT) bytes[i] = 0;
  for (int i = threadIdx.x; i < 64 * a.nlev; i += kColT) {
    const LevelDev& L = a.lv[i >> 6];
    const double d = (double)L.wx * (i & 3) + (double)L.wy * ((i >> 2) & 3) + (double)L.wz * ((i >> 4) & 3);
    float2* t = tab + kTabs * (i >> 6) + (i & 63);
    put(t, 0, to_ff(d));
    put(t, 64, to_ff(d > 0.0 ? 1.0 / d : 0.0));
    put(t, 128, to_ff(d > 0.0 ? omega / d : 0.0));
  }
  __syncthreads();
  for (int l = 0; l < a.nlev; ++l) {
    const LevelDev& L = a.lv[l];
    const DLev v = d_level(a, l, tab, arr, bytes);
    for (int i = threadIdx.x; i < v.g.n; i += kColT) {
      int x, y, z;
      v.g.xyz(i, x, y, z);
      int m = kFluidBit | axis_count(x, L.nx, L.bcD, 0) | axis_count(y, L.ny, L.bcD, 2) << 2;
      if (DIM == 3) m |= axis_count(z, L.nz, L.bcD, 4) << 4;
      v.m[v.g.pad(x, y, z)] = L.cell ? L.cell[i] : (uint8_t)m;
      if (l == 0 && i == j) v.b[v.g.pad(x, y, z)] = make_float2(1.f, 0.f);
    }
  }
  __syncthreads();
  const ff keep = to_ff(1.0 - omega), sc = to_ff(s), zero = {0.f, 0.f};
  unsigned odd = 0u;  // bit l: level l's x and x' have changed places
  auto level = [&](int l) {
    DLev v = d_level(a, l, tab, arr, bytes);
    if ((odd >> l) & 1u) d_swap(v);
    return v;
  };
  // down legs: x from zero, the restricted residual (sawtooth: b's average)
  for (int l = 0; l < last; ++l) {
    DLev v = level(l);
    const DLev c = level(l + 1);
    d_cells(v, [&](int, int p, int q, int, int, int) {
      put(v.x, p, q < 0 || a.pre == 0 ? zero : ff_mul(get(v.b, p), get(saw ? v.id : v.w, q)));
    });
    for (int k = 2; k <= a.pre; ++k) d_sweep<DIM>(v, keep);
    if (a.pre > 1 && !(a.pre & 1)) odd |= 1u << l;
    d_cells(c, [&](int, int pc, int, int X, int Y, int Z) {
      ff sum = zero;
      for (int k = 0; k < (DIM == 3 ? 8 : 4); ++k) {
        const int p = v.g.pad(2 * X + (k & 1), 2 * Y + ((k >> 1) & 1), 2 * Z + (k >> 2)), m = v.m[p];
        if (!m) continue;
        ff r = get(v.b, p);
        if (!saw) r = ff_add(r, ff_add(d_nb<DIM>(v, v.x, p), ff_neg(ff_mul(get(v.x, p), get(v.d, m & 63)))));
        sum = ff_add(sum, r);
      }
      put(c.b, pc, scale(sum, DIM == 3 ? 0.125f : 0.25f));
    });
  }
  // coarsest: A^-1 b in float64 (sawtooth: a Jacobi step and the sweeps)
  {
    DLev v = level(last);
    if (saw) {
      d_cells(v, [&](int, int p, int q, int, int, int) {
        put(v.x, p, q < 0 ? zero : ff_mul(get(v.b, p), get(v.id, q)));
      });
      for (int k = 1; k <= a.post; ++k) d_sweep<DIM>(v, keep);
      if (a.post & 1) odd |= 1u << last;
    } else {
      // a unit vector reaches a few coarsest cells only: their list (in order,
      // so that the sums are the same every time) in the array x' has no use
      // for, then a row per thread
      __shared__ int count;
      int* list = reinterpret_cast<int*>(v.y);
      if (threadIdx.x < 32) {
        int have = 0;
        for (int k0 = 0; k0 < nc; k0 += 32) {
          const int k = k0 + (int)threadIdx.x;
          bool on = false;
          if (k < nc) {
            int x, y, z;
            v.g.xyz(k, x, y, z);
            on = v.b[v.g.pad(x, y, z)].x != 0.f;
          }
          const unsigned mask = __ballot_sync(0xffffffffu, on);
          if (on) list[have + __popc(mask & ((1u << threadIdx.x) - 1u))] = k;
          have += __popc(mask);
        }
        if (threadIdx.x == 0) count = have;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < nc; i += kColT) {
        double acc = 0.0;
        int x, y, z;
        for (int q = 0; q < count; ++q) {
          const int k = list[q];
          v.g.xyz(k, x, y, z);
          const float2 b = v.b[v.g.pad(x, y, z)];
          acc = fma(__ldg(inv + (size_t)k * nc + i), (double)b.x + (double)b.y, acc);
        }
        v.g.xyz(i, x, y, z);
        put(v.x, v.g.pad(x, y, z), to_ff(acc));
      }
      __syncthreads();
    }
  }
  // up legs: x + s P e, the sweeps
  for (int l = last - 1; l >= 0; --l) {
    DLev v = level(l);
    const DLev c = level(l + 1);
    d_cells(v, [&](int, int p, int q, int X, int Y, int Z) {
      if (q >= 0) put(v.x, p, ff_add(get(v.x, p), ff_mul(get(c.x, c.g.pad(X >> 1, Y >> 1, Z >> 1)), sc)));
    });
    for (int k = 1; k <= a.post; ++k) d_sweep<DIM>(v, keep);
    if (a.post & 1) odd ^= 1u << l;
  }
  const DLev v = level(0);
  d_cells(v, [&](int i, int p, int, int, int, int) { out[i] = v.x[p].x + v.x[p].y; });
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

cudaError_t launch_transpose(float* M, int n, cudaStream_t s) {
  const int t = (n + 31) / 32;
  k_transpose<<<dim3(t, t), 256, 0, s>>>(M, n, dense_stride(n));
  return cudaGetLastError();
}

// Shared memory of a column's block: the tables, three float-float arrays and
// the cell bytes (`bytes`: what coarse_layout asks, 16 per padded cell).
size_t dense_smem(size_t bytes, int nlev) { return (size_t)nlev * kTabs * 8 + bytes / 16 * 25; }

cudaError_t launch_dense_matrix(const CoarseArgs& a, size_t layout_bytes, int n, const double* inv, double omega,
                                double scale, float* M, cudaStream_t s) {
  const int ld = dense_stride(n);
  const auto k = a.dim == 3 ? k_dense_columns<3> : k_dense_columns<2>;
  cudaError_t e = cudaMemsetAsync(M, 0, dense_bytes(n), s);
  int dev = 0, optin = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
  if (e != cudaSuccess) return e;
  k<<<n, kColT, dense_smem(layout_bytes, a.nlev), s>>>(a, inv, omega, scale, M, ld);
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
