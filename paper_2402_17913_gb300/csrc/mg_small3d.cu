// 3D level kernels with two Jacobi sweeps for levels too small to fill the
// GPU with streamed columns.
//
// Such a level is bound by the latency of one block (load, two or three
// barrier-separated phases, store), not by bytes: a streamed column walks
// its planes one after another at a few hundred nanoseconds each, and the
// 32 x 8 x 8 tiles of k_down / k_up leave most SMs idle while each block
// works through twenty cells per thread and phase.  Here a block of 256
// threads owns a 16 x 4 x 4 tile (region with the two-cell halo 20 x 8 x 8:
// five cells per thread, all loads in flight at once; one output cell per
// thread), so that even an 8192-cell level spreads over 32 SMs and a phase is
// a few cells per thread.  Geometry, link counts and diagonals do not depend
// on the previous kernel and are formed before the wait for it.
//
// Same arithmetic as the streamed kernels (Eq. Jacobi-1-relax, the average
// restriction and copy prolongation of App. B / Sec. 2.2).
#include <stdlib.h>

#include <type_traits>

#include "launch.h"
#include "mg_kernels.cuh"

namespace npmg {

namespace {

constexpr int TX = 16, TY = 4, TZ = 4, TN = TX * TY * TZ;  // tile
constexpr int RX = TX + 4, RY = TY + 4, RZ = TZ + 4, RN = RX * RY * RZ, RXY = RX * RY;
constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + 2, SN = SX * SY * SZ;  // tile and one cell around it
constexpr int NT = 256;
constexpr int KA = (RN + NT - 1) / NT, KB = (SN + NT - 1) / NT;
static_assert(TN == NT && RN % NT == 0, "one output cell per thread, whole passes over the region");

// Per-thread region cells: global offsets (-1 off the fluid) and diagonals.
struct Cells {
  int off[KA];
  float d[KA];
};

template <bool MASKED>
__device__ __forceinline__ void region_cells(const LevelDev& L, Cells& c, int* gxyz) {
  const int ox = blockIdx.x * TX - 2, oy = blockIdx.y * TY - 2, oz = blockIdx.z * TZ - 2;
#pragma unroll
  for (int k = 0; k < KA; ++k) {
    const int i = threadIdx.x + k * NT;
    const int gx = ox + i % RX, gy = oy + (i / RX) % RY, gz = oz + i / RXY;
    const bool in = inside<3>(L, gx, gy, gz);
    c.off[k] = in ? (gz * L.ny + gy) * L.nx + gx : -1;
    c.d[k] = 0.f;
    if (in) {
      const uint8_t m = MASKED ? L.cell[c.off[k]] : kFluidBit;
      if (m) c.d[k] = diag_at<3, MASKED>(L, gx, gy, gz, m);
      else c.off[k] = -1;
    }
    if (gxyz) gxyz[k] = in ? ((gz >> 1) * (L.ny >> 1) + (gy >> 1)) * (L.nx >> 1) + (gx >> 1) : 0;
  }
}

__device__ __forceinline__ float nb7(const LevelDev& L, const float* x, int i) {
  return L.wx * (x[i - 1] + x[i + 1]) + L.wy * (x[i - RX] + x[i + RX]) + L.wz * (x[i - RXY] + x[i + RXY]);
}

// One sweep of the cells of the tile and its one-cell ring.
__device__ __forceinline__ void sweep_ring(const LevelDev& L, const float* xin, float* xout, const float* sB,
                                           const float* sD, float omega) {
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int i = threadIdx.x + k * NT;
    if (i < SN) {
      const int li = (i / (SX * SY) + 1) * RXY + ((i / SX) % SY + 1) * RX + i % SX + 1;
      const float d = sD[li];
      xout[li] = d > 0.f ? fmaf(1.f - omega, xin[li], __fdividef(omega, d) * (sB[li] + nb7(L, xin, li))) : 0.f;
    }
  }
}

}  // namespace

// Down leg: x = two sweeps from zero, bcoarse = R (b - A' x).
template <typename T, bool MASKED, typename TB>
__global__ void __launch_bounds__(NT) k_down_c3(LevelDev L, const TB* __restrict__ b, T* __restrict__ x,
                                                T* __restrict__ bcoarse, float omega,
                                                const SolveState* __restrict__ st) {
  __shared__ float sB[RN], sD[RN], s1[RN], s2[RN], sR[TN];
  Cells c;
  region_cells<MASKED>(L, c, nullptr);
  chain_enter();
  if (st && st->inner_done) return;
  float v[KA];
#pragma unroll
  for (int k = 0; k < KA; ++k) v[k] = c.off[k] >= 0 ? ld(b, c.off[k]) : 0.f;
#pragma unroll
  for (int k = 0; k < KA; ++k) {
    const int i = threadIdx.x + k * NT;
    sB[i] = v[k];
    sD[i] = c.d[k];
    s1[i] = c.d[k] > 0.f ? __fdividef(omega, c.d[k]) * v[k] : 0.f;
  }
  __syncthreads();
  sweep_ring(L, s1, s2, sB, sD, omega);
  __syncthreads();
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX % TY, tz = threadIdx.x / (TX * TY);
  const int li = (tz + 2) * RXY + (ty + 2) * RX + tx + 2;
  {
    const float d = sD[li], xc = s2[li];
    const int gx = blockIdx.x * TX + tx, gy = blockIdx.y * TY + ty, gz = blockIdx.z * TZ + tz;
    sR[threadIdx.x] = d > 0.f ? sB[li] - (d * xc - nb7(L, s2, li)) : 0.f;
    if (inside<3>(L, gx, gy, gz)) x[(gz * L.ny + gy) * L.nx + gx] = cvt<T>(xc);
  }
  __syncthreads();
  if (threadIdx.x < TN / 8) {
    const int cx = threadIdx.x % (TX / 2), cy = threadIdx.x / (TX / 2) % (TY / 2), cz = threadIdx.x / (TX * TY / 4);
    const int gx = blockIdx.x * (TX / 2) + cx, gy = blockIdx.y * (TY / 2) + cy, gz = blockIdx.z * (TZ / 2) + cz;
    if (gx < L.nx / 2 && gy < L.ny / 2 && gz < L.nz / 2) {
      float sum = 0.f;
#pragma unroll
      for (int az = 0; az < 2; ++az)
#pragma unroll
        for (int ay = 0; ay < 2; ++ay) {
          const float* r = sR + (2 * cz + az) * (TX * TY) + (2 * cy + ay) * TX + 2 * cx;
          sum += r[0] + r[1];
        }
      bcoarse[(gz * (L.ny / 2) + gy) * (L.nx / 2) + gx] = cvt<T>(sum * 0.125f);
    }
  }
}

// Up leg: xout = two sweeps from x + s P e; on the finest level (r, z) and
// CG's beta.
template <typename T, bool MASKED, bool FINEST, typename TB>
__global__ void __launch_bounds__(NT) k_up_c3(LevelDev L, const TB* __restrict__ b, const T* __restrict__ xin,
                                              TB* __restrict__ xout, const T* __restrict__ e, float omega, float s,
                                              SolveState* __restrict__ st, double* __restrict__ partials) {
  __shared__ float sB[RN], sD[RN], s0[RN], s1[RN];
  Cells c;
  int co[KA];
  region_cells<MASKED>(L, c, co);
  chain_enter();
  if (st && st->inner_done) return;
  float v[KA], w[KA], q[KA];
#pragma unroll
  for (int k = 0; k < KA; ++k) {
    const bool on = c.off[k] >= 0;
    v[k] = on ? ld(xin, c.off[k]) : 0.f;
    w[k] = on ? ld(b, c.off[k]) : 0.f;
    q[k] = on ? ld(e, co[k]) : 0.f;
  }
#pragma unroll
  for (int k = 0; k < KA; ++k) {
    const int i = threadIdx.x + k * NT;
    sB[i] = w[k];
    sD[i] = c.d[k];
    s0[i] = fmaf(s, q[k], v[k]);
  }
  __syncthreads();
  sweep_ring(L, s0, s1, sB, sD, omega);
  __syncthreads();
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX % TY, tz = threadIdx.x / (TX * TY);
  const int li = (tz + 2) * RXY + (ty + 2) * RX + tx + 2;
  const int gx = blockIdx.x * TX + tx, gy = blockIdx.y * TY + ty, gz = blockIdx.z * TZ + tz;
  float acc = 0.f;
  if (inside<3>(L, gx, gy, gz)) {
    const float d = sD[li];
    const float z =
        d > 0.f ? fmaf(1.f - omega, s1[li], __fdividef(omega, d) * (sB[li] + nb7(L, s1, li))) : 0.f;
    const TB zt = cvt<TB>(z);
    xout[(gz * L.ny + gy) * L.nx + gx] = zt;
    if (FINEST) acc = sB[li] * ld(&zt, 0);
  }
  if (FINEST) {
    double tot;
    if (grid_sum_last((double)acc, partials, &st->counter[kCntRZ], &tot)) {
      if (threadIdx.x == 0) {
        st->rz = tot;
        st->beta = (st->first || !st->krylov) ? 0.0 : tot / st->rz_old;
        st->rz_old = tot;
      }
    }
  }
}

static dim3 c3_grid(const LevelDev& L) {
  return dim3((L.nx + TX - 1) / TX, (L.ny + TY - 1) / TY, (L.nz + TZ - 1) / TZ);
}

// Levels of at most 200,000 cells (or NPMG_SMALL3D_MAX): measured on both
// legs of a level together, the tiles are faster than the streamed columns
// by 7.8 us on 40 x 36 x 40, 4.0 us on 48 x 40 x 32, 2.5 us on 64 x 32 x 32
// and 3.0 us on 80 x 48 x 40 (153,600 cells), and 1.9 us slower on 64^3
// (262,144).  160 x 96 x 80 FP16 solve 3.57 -> 3.09 ms, 256^3 10.50 -> 10.29.
// A smallest level set for the streamed kernels (NPMG_TMA3D_MIN,
// NPMG_ROWS3D_MIN) keeps the levels with them.
bool small3d_eligible(int dim, int pre, int post, const LevelDev& L) {
  const char* e = getenv("NPMG_SMALL3D_MAX");
  const long most = e ? atol(e) : 200000;
  if (!e && (getenv("NPMG_TMA3D_MIN") || getenv("NPMG_ROWS3D_MIN"))) return false;
  const dim3 g = c3_grid(L);
  return dim == 3 && pre == 2 && post == 2 && (long)L.nx * L.ny * L.nz <= most &&
         (size_t)g.x * g.y * g.z <= 65536;
}

template <typename T, bool MASKED, typename TB>
cudaError_t launch_down_c3(const LevelDev& L, const void* b, void* x, void* bcoarse, float omega,
                           const SolveState* st, cudaStream_t s) {
  return launch_chain(k_down_c3<T, MASKED, TB>, c3_grid(L), NT, 0, s, L, (const TB*)b, (T*)x, (T*)bcoarse, omega, st);
}

template <typename T, bool MASKED, bool FINEST, typename TB>
cudaError_t launch_up_c3(const LevelDev& L, const void* b, const void* xin, void* xout, const void* e, float omega,
                         float sc, SolveState* st, double* partials, cudaStream_t s) {
  return launch_chain(k_up_c3<T, MASKED, FINEST, TB>, c3_grid(L), NT, 0, s, L, (const TB*)b, (const T*)xin,
                      (TB*)xout, (const T*)e, omega, sc, st, partials);
}

#define NPMG_INST_C3(T, M, TB)                                                                                    \
  template cudaError_t launch_down_c3<T, M, TB>(const LevelDev&, const void*, void*, void*, float,                \
                                                const SolveState*, cudaStream_t);                                 \
  template cudaError_t launch_up_c3<T, M, false, TB>(const LevelDev&, const void*, const void*, void*,            \
                                                     const void*, float, float, SolveState*, double*,             \
                                                     cudaStream_t);                                               \
  template cudaError_t launch_up_c3<T, M, true, TB>(const LevelDev&, const void*, const void*, void*,             \
                                                    const void*, float, float, SolveState*, double*, cudaStream_t);
NPMG_INST_C3(float, false, float)
NPMG_INST_C3(float, true, float)
NPMG_INST_C3(__half, false, __half)
NPMG_INST_C3(__half, true, __half)
NPMG_INST_C3(__half, false, float)
NPMG_INST_C3(__half, true, float)
NPMG_INST_C3(__nv_bfloat16, false, __nv_bfloat16)
NPMG_INST_C3(__nv_bfloat16, true, __nv_bfloat16)
NPMG_INST_C3(__nv_bfloat16, false, float)
NPMG_INST_C3(__nv_bfloat16, true, float)

}  // namespace npmg
