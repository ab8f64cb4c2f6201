// Level kernels with two Jacobi sweeps for levels too small to fill the GPU
// with streamed columns or large tiles.
//
// Such a level is bound by the latency of one block (load, two or three
// barrier-separated phases, store), not by bytes: a streamed column walks
// its planes one after another at a few hundred nanoseconds each, and the
// 32 x 8 x 8 (3D) and 64 x 16 (2D) tiles of the other kernels leave SMs idle
// while each block works through six to twenty cells per thread and phase.
// Here a block of 256 threads owns 16 x 4 x 4 or 32 x 8 cells (regions with
// the two-cell halo of 20 x 8 x 8 and 36 x 12: five and two cells per thread,
// all loads in flight at once; one output cell per thread), so that even an
// 8192-cell level spreads over 32 SMs and a phase is a few cells per thread.
// Geometry, link counts and diagonals do not depend on the previous kernel
// and are formed before the wait for it.
//
// Same arithmetic as the streamed kernels (Eq. Jacobi-1-relax, the average
// restriction and copy prolongation of App. B / Sec. 2.2).
#include <stdlib.h>

#include <type_traits>

#include "launch.h"
#include "mg_kernels.cuh"

namespace npmg {

namespace {

constexpr int NT = 256;

// Tile of a block, the region with its two-cell halo and the tile with a
// one-cell ring.
template <int DIM>
struct Tl {
  static constexpr int TX = DIM == 3 ? 16 : 32, TY = DIM == 3 ? 4 : 8, TZ = DIM == 3 ? 4 : 1, TN = TX * TY * TZ;
  static constexpr int HZ = DIM == 3 ? 2 : 0;
  static constexpr int RX = TX + 4, RY = TY + 4, RZ = TZ + 2 * HZ, RN = RX * RY * RZ, RXY = RX * RY;
  static constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + HZ, SN = SX * SY * SZ;
  static constexpr int KA = (RN + NT - 1) / NT, KB = (SN + NT - 1) / NT;
  static_assert(TN == NT, "one output cell per thread");
};

// Per-thread region cells: global offsets (-1 off the fluid), the offsets of
// their coarse parents, and diagonals.
template <int DIM, bool MASKED>
__device__ __forceinline__ void region_cells(const LevelDev& L, int (&off)[Tl<DIM>::KA], float (&d)[Tl<DIM>::KA],
                                             int* parent) {
  using W = Tl<DIM>;
  const int ox = blockIdx.x * W::TX - 2, oy = blockIdx.y * W::TY - 2, oz = blockIdx.z * W::TZ - W::HZ;
#pragma unroll
  for (int k = 0; k < W::KA; ++k) {
    const int i = threadIdx.x + k * NT;
    const int gx = ox + i % W::RX, gy = oy + (i / W::RX) % W::RY, gz = oz + i / W::RXY;
    const bool in = i < W::RN && inside<DIM>(L, gx, gy, gz);
    off[k] = in ? (gz * L.ny + gy) * L.nx + gx : -1;
    d[k] = 0.f;
    if (in) {
      const uint8_t m = MASKED ? L.cell[off[k]] : kFluidBit;
      if (m) d[k] = diag_at<DIM, MASKED>(L, gx, gy, gz, m);
      else off[k] = -1;
    }
    if (parent) parent[k] = in ? ((gz >> 1) * (L.ny >> 1) + (gy >> 1)) * (L.nx >> 1) + (gx >> 1) : 0;
  }
}

template <int DIM>
__device__ __forceinline__ float nbsum(const LevelDev& L, const float* x, int i) {
  using W = Tl<DIM>;
  float nb = L.wx * (x[i - 1] + x[i + 1]) + L.wy * (x[i - W::RX] + x[i + W::RX]);
  if (DIM == 3) nb += L.wz * (x[i - W::RXY] + x[i + W::RXY]);
  return nb;
}

// One sweep of a cell, x + (omega / d)(b + nb - d x).  The error of omega / d
// then scales with the residual; in (1 - omega) x + (omega / d)(b + nb) it
// scales with x, the same in every interior cell, and is a bias of the whole
// cycle: on 48 x 64 x 56 against 64 bits 1.5e-7, 0.64e-7 so (1.0e-7 with the
// streamed columns and their rounded quotient; that one here, formed before
// the wait, gave 1.2e-7).  Formed in every cell and selected at the end: with
// the formula behind the test of d its loads wait for d (96 x 80 x 64 cycle
// 27.8 us, 26.9 so, 27.0 in the biased form).
template <int DIM>
__device__ __forceinline__ float sweep_cell(const LevelDev& L, const float* x, const float* sB, float d, float omega,
                                            int i) {
  const float xc = x[i], nb = nbsum<DIM>(L, x, i);
  const float v = fmaf(__fdividef(omega, d), nb + fmaf(-d, xc, sB[i]), xc);
  return d > 0.f ? v : 0.f;
}

// One sweep of the cells of the tile and its one-cell ring.
template <int DIM>
__device__ __forceinline__ void sweep_ring(const LevelDev& L, const float* xin, float* xout, const float* sB,
                                           const float* sD, float omega) {
  using W = Tl<DIM>;
#pragma unroll
  for (int k = 0; k < W::KB; ++k) {
    const int i = threadIdx.x + k * NT;
    if (i < W::SN) {
      const int lz = DIM == 3 ? i / (W::SX * W::SY) + 1 : 0;
      const int li = lz * W::RXY + ((i / W::SX) % W::SY + 1) * W::RX + i % W::SX + 1;
      xout[li] = sweep_cell<DIM>(L, xin, sB, sD[li], omega, li);
    }
  }
}

// This thread's output cell: region index and global coordinates.
template <int DIM>
__device__ __forceinline__ int out_cell(int& gx, int& gy, int& gz) {
  using W = Tl<DIM>;
  const int tx = threadIdx.x % W::TX, ty = threadIdx.x / W::TX % W::TY, tz = threadIdx.x / (W::TX * W::TY);
  gx = blockIdx.x * W::TX + tx;
  gy = blockIdx.y * W::TY + ty;
  gz = blockIdx.z * W::TZ + tz;
  return (tz + W::HZ) * W::RXY + (ty + 2) * W::RX + tx + 2;
}

}  // namespace

// Down leg: x = two sweeps from zero, bcoarse = R (b - A' x).
template <int DIM, typename T, bool MASKED, typename TB>
__global__ void __launch_bounds__(NT) k_down_c(LevelDev L, const TB* __restrict__ b, T* __restrict__ x,
                                               T* __restrict__ bcoarse, float omega,
                                               const SolveState* __restrict__ st) {
  using W = Tl<DIM>;
  __shared__ float sB[W::RN], sD[W::RN], s1[W::RN], s2[W::RN], sR[W::TN];
  int off[W::KA];
  float d[W::KA], v[W::KA];
  if (DIM == 3) chain_release();
  region_cells<DIM, MASKED>(L, off, d, nullptr);
  chain_enter();
  if (st && st->inner_done) return;
#pragma unroll
  for (int k = 0; k < W::KA; ++k) v[k] = off[k] >= 0 ? ld(b, off[k]) : 0.f;
#pragma unroll
  for (int k = 0; k < W::KA; ++k) {
    const int i = threadIdx.x + k * NT;
    if (W::RN % NT == 0 || i < W::RN) {
      sB[i] = v[k];
      sD[i] = d[k];
      s1[i] = d[k] > 0.f ? __fdividef(omega, d[k]) * v[k] : 0.f;
    }
  }
  __syncthreads();
  sweep_ring<DIM>(L, s1, s2, sB, sD, omega);
  __syncthreads();
  {
    int gx, gy, gz;
    const int li = out_cell<DIM>(gx, gy, gz);
    const float dc = sD[li], xc = s2[li];
    sR[threadIdx.x] = dc > 0.f ? sB[li] - (dc * xc - nbsum<DIM>(L, s2, li)) : 0.f;
    if (inside<DIM>(L, gx, gy, gz)) x[(gz * L.ny + gy) * L.nx + gx] = cvt<T>(xc);
  }
  __syncthreads();
  constexpr int CX = W::TX / 2, CY = W::TY / 2, CZ = DIM == 3 ? W::TZ / 2 : 1;
  if (threadIdx.x < CX * CY * CZ) {
    const int cx = threadIdx.x % CX, cy = threadIdx.x / CX % CY, cz = threadIdx.x / (CX * CY);
    const int gx = blockIdx.x * CX + cx, gy = blockIdx.y * CY + cy, gz = blockIdx.z * CZ + cz;
    if (gx < L.nx / 2 && gy < L.ny / 2 && (DIM == 2 || gz < L.nz / 2)) {
      float sum = 0.f;
#pragma unroll
      for (int az = 0; az < (DIM == 3 ? 2 : 1); ++az)
#pragma unroll
        for (int ay = 0; ay < 2; ++ay) {
          const float* r = sR + (2 * cz + az) * (W::TX * W::TY) + (2 * cy + ay) * W::TX + 2 * cx;
          sum += r[0] + r[1];
        }
      bcoarse[(gz * (L.ny / 2) + gy) * (L.nx / 2) + gx] = cvt<T>(sum * (DIM == 3 ? 0.125f : 0.25f));
    }
  }
}

// Up leg: xout = two sweeps from x + s P e; on the finest level (r, z) and
// CG's beta.
template <int DIM, typename T, bool MASKED, bool FINEST, typename TB>
__global__ void __launch_bounds__(NT) k_up_c(LevelDev L, const TB* __restrict__ b, const T* __restrict__ xin,
                                             TB* __restrict__ xout, const T* __restrict__ e, float omega, float s,
                                             SolveState* __restrict__ st, double* __restrict__ partials) {
  using W = Tl<DIM>;
  __shared__ float sB[W::RN], sD[W::RN], s0[W::RN], s1[W::RN];
  int off[W::KA], parent[W::KA];
  float d[W::KA], v[W::KA], w[W::KA], q[W::KA];
  if (DIM == 3) chain_release();
  region_cells<DIM, MASKED>(L, off, d, parent);
  chain_enter();
  if (st && st->inner_done) return;
#pragma unroll
  for (int k = 0; k < W::KA; ++k) {
    const bool on = off[k] >= 0;
    v[k] = on ? ld(xin, off[k]) : 0.f;
    w[k] = on ? ld(b, off[k]) : 0.f;
    q[k] = on ? ld(e, parent[k]) : 0.f;
  }
#pragma unroll
  for (int k = 0; k < W::KA; ++k) {
    const int i = threadIdx.x + k * NT;
    if (W::RN % NT == 0 || i < W::RN) {
      sB[i] = w[k];
      sD[i] = d[k];
      s0[i] = fmaf(s, q[k], v[k]);
    }
  }
  __syncthreads();
  sweep_ring<DIM>(L, s0, s1, sB, sD, omega);
  __syncthreads();
  int gx, gy, gz;
  const int li = out_cell<DIM>(gx, gy, gz);
  float acc = 0.f;
  if (inside<DIM>(L, gx, gy, gz)) {
    const TB zt = cvt<TB>(sweep_cell<DIM>(L, s1, sB, sD[li], omega, li));
    xout[(gz * L.ny + gy) * L.nx + gx] = zt;
    if (FINEST) acc = sB[li] * ld(&zt, 0);
  }
  if (FINEST) {
    double tot;
    if (grid_sum_last(acc, partials, &st->counter[kCntRZ], &tot)) {
      if (threadIdx.x == 0) {
        st->rz = tot;
        st->beta = (st->first || !st->krylov) ? 0.0 : tot / st->rz_old;
        st->rz_old = tot;
      }
    }
  }
}

static dim3 c_grid(int dim, const LevelDev& L) {
  if (dim == 3)
    return dim3((L.nx + Tl<3>::TX - 1) / Tl<3>::TX, (L.ny + Tl<3>::TY - 1) / Tl<3>::TY,
                (L.nz + Tl<3>::TZ - 1) / Tl<3>::TZ);
  return dim3((L.nx + Tl<2>::TX - 1) / Tl<2>::TX, (L.ny + Tl<2>::TY - 1) / Tl<2>::TY);
}

// Levels of at most 200,000 cells (or NPMG_SMALL3D_MAX, NPMG_SMALL2D_MAX).
// 3D, measured on both legs of a level together: faster than the streamed
// columns by 7.8 us on 40 x 36 x 40, 4.0 us on 48 x 40 x 32, 2.5 us on
// 64 x 32 x 32 and 3.0 us on 80 x 48 x 40 (153,600 cells), and 1.9 us slower on
// 64^3 (262,144).  160 x 96 x 80 FP16 solve 3.57 -> 3.09 ms, 256^3 10.50 -> 10.29.
// 2D, with levels up to 0 / 40,000 / 140,000 / 300,000 cells here: 1600x960
// solve 2.19 / 1.91 / 1.95 / 1.98 ms, 2048x1024 flow step 1.82 / 1.77 / 1.72 /
// 1.76, 960x800 solve 1.57 / 1.52 / 1.30 / 1.26 (its 480 x 400 level), 448x576
// (258,048 cells) 1.23 / 1.05 / 1.01 / 1.06.
// A smallest level set for the streamed kernels (NPMG_TMA3D_MIN,
// NPMG_ROWS3D_MIN, NPMG_STREAM2D_MIN) keeps the levels with them.
bool small_level_eligible(int dim, int pre, int post, const LevelDev& L) {
  const char* e = getenv(dim == 3 ? "NPMG_SMALL3D_MAX" : "NPMG_SMALL2D_MAX");
  const long most = e ? atol(e) : 200000;
  if (dim == 3 && !e && (getenv("NPMG_TMA3D_MIN") || getenv("NPMG_ROWS3D_MIN"))) return false;
  if (dim == 2 && !e && getenv("NPMG_STREAM2D_MIN")) return false;
  const dim3 g = c_grid(dim, L);
  return pre == 2 && post == 2 && (long)L.nx * L.ny * L.nz <= most && (size_t)g.x * g.y * g.z <= 65536;
}

template <int DIM, typename T, bool MASKED, typename TB>
cudaError_t launch_down_c(const LevelDev& L, const void* b, void* x, void* bcoarse, float omega,
                          const SolveState* st, cudaStream_t s) {
  return launch_chain(k_down_c<DIM, T, MASKED, TB>, c_grid(DIM, L), NT, 0, s, L, (const TB*)b, (T*)x, (T*)bcoarse,
                      omega, st);
}

template <int DIM, typename T, bool MASKED, bool FINEST, typename TB>
cudaError_t launch_up_c(const LevelDev& L, const void* b, const void* xin, void* xout, const void* e, float omega,
                        float sc, SolveState* st, double* partials, cudaStream_t s) {
  return launch_chain(k_up_c<DIM, T, MASKED, FINEST, TB>, c_grid(DIM, L), NT, 0, s, L, (const TB*)b, (const T*)xin,
                      (TB*)xout, (const T*)e, omega, sc, st, partials);
}

#define NPMG_INST_C_D(DIM, T, M, TB)                                                                            \
  template cudaError_t launch_down_c<DIM, T, M, TB>(const LevelDev&, const void*, void*, void*, float,          \
                                                    const SolveState*, cudaStream_t);                           \
  template cudaError_t launch_up_c<DIM, T, M, false, TB>(const LevelDev&, const void*, const void*, void*,      \
                                                         const void*, float, float, SolveState*, double*,       \
                                                         cudaStream_t);                                         \
  template cudaError_t launch_up_c<DIM, T, M, true, TB>(const LevelDev&, const void*, const void*, void*,       \
                                                        const void*, float, float, SolveState*, double*,        \
                                                        cudaStream_t);
#define NPMG_INST_C(T, M, TB) NPMG_INST_C_D(2, T, M, TB) NPMG_INST_C_D(3, T, M, TB)
NPMG_INST_C(float, false, float)
NPMG_INST_C(float, true, float)
NPMG_INST_C(__half, false, __half)
NPMG_INST_C(__half, true, __half)
NPMG_INST_C(__half, false, float)
NPMG_INST_C(__half, true, float)
NPMG_INST_C(__nv_bfloat16, false, __nv_bfloat16)
NPMG_INST_C(__nv_bfloat16, true, __nv_bfloat16)
NPMG_INST_C(__nv_bfloat16, false, float)
NPMG_INST_C(__nv_bfloat16, true, float)

}  // namespace npmg
