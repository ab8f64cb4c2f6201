// Batched solver: the level legs and the direction update of one strip of
// rows, streamed along y by a single warp with no barrier of any kind.
//
// A warp holds 32 consecutive groups of four cells of a row (one float4 per
// lane) and walks a run of rows.  With H sweeps, when row p arrives its input
// is formed there, sweep k on row p - k and (down) the residual on row p - H:
// three-row rings in registers, neighbours in x from the adjacent lanes by
// shuffles, rows by asynchronous copies kSD rows ahead into a ring of
// shared-memory slots of which every lane reads back only its own bytes.  At
// a strip's inner edge one group beyond it is a halo lane: a sweep spoils one
// more of its cells from the outside, at most three of four, and the fourth
// is all the strip's own cells need.
//
// What bounds it: issue slots and memory about equally (140 to 160
// instructions per row of 128 cells against 0.6 to 1.8 KB).  The block tiles
// it replaced staged a 72 x 38 region for 64 x 32 cells behind seven block
// barriers, 6 us a tile at four blocks per SM: 256 instances of sides 64 to
// 512, three sweeps, 28.1 -> 21.0 ms a solve.
#pragma once

#include "npmg_internal.cuh"

namespace npmg {

constexpr int kSD = 5;          // rows in flight ahead of the row in use
constexpr int kSSlots = kSD + 1;
constexpr int kSRowDown = 32 * 16 + 32 * 4;                     // b, cell bytes
constexpr int kSRowUp = 2 * 32 * 16 + 32 * 8 + 32 * 4;          // x (or z), b (or p), e, cell bytes
constexpr int kSRing = kSSlots * kSRowUp;                       // bytes of one warp's ring
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void s_copy16(uint32_t dst, const void* src, bool full) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(full ? 16 : 0) : "memory");
}
template <int N>
__device__ __forceinline__ void s_copy(uint32_t dst, const void* src, bool full) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src), "n"(N), "r"(full ? N : 0)
               : "memory");
}
__device__ __forceinline__ void s_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void s_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(kSD - 1) : "memory"); }

// The lane's group of a strip [u0, u1) of the level's groups, and the level's
// diagonal by link counts (an entry per lane, read by shuffles).
struct SLane {
  int lane, gx, go;
  bool in, own;
  unsigned mx;       // no solid: fluid bits and x link counts of the four cells
  float tabd, tabw;  // entry (kx + 4 ky) of d and omega / d; 0 without links
};

__device__ __forceinline__ SLane s_lane(const LevelDev& L, int u0, int u1, float omega) {
  SLane c;
  c.lane = threadIdx.x & 31;
  const int g = (u0 > 0 ? u0 - 1 : 0) + c.lane;
  c.gx = 4 * g;
  c.in = g <= u1 && c.gx < L.nx;  // up to one group beyond the strip
  c.own = g >= u0 && g < u1;
  c.go = c.in ? c.gx : 0;  // copies that only fill with zeros keep a source in bounds
  c.mx = 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (c.in) c.mx |= (unsigned)(kFluidBit | axis_count(c.gx + j, L.nx, L.bcD, 0)) << (8 * j);
  const float d = c.lane < 16 ? L.wx * (float)(c.lane & 3) + L.wy * (float)(c.lane >> 2) : 0.f;
  c.tabd = d;
  c.tabw = d > 0.f ? __fdividef(omega, d) : 0.f;
  return c;
}

// cell bytes of the lane's group on row p: the copied word, or from the
// position on a level without solid
__device__ __forceinline__ unsigned s_cells(const LevelDev& L, const SLane& c, int p, const unsigned char* slot) {
  if (L.cell) return *reinterpret_cast<const unsigned*>(slot + c.lane * 4);
  if (p < 0 || p >= L.ny || !c.in) return 0u;
  return c.mx | ((unsigned)axis_count(p, L.ny, L.bcD, 2) * 0x04040404u);
}
__device__ __forceinline__ unsigned s_byte(unsigned m, int j) { return (m >> (8 * j)) & 0xffu; }

// values beside the lane's first and last cell: 0 beyond the warp, which is
// the level's edge or the spoilt side of a halo lane
__device__ __forceinline__ void s_edges(const SLane& c, const float (&a)[4], float& left, float& right) {
  left = __shfl_up_sync(kFull, a[3], 1);
  right = __shfl_down_sync(kFull, a[0], 1);
  if (c.lane == 0) left = 0.f;
  if (c.lane == 31) right = 0.f;
}

// one sweep on row a between rows dn and up
__device__ __forceinline__ void s_sweep(const LevelDev& L, const SLane& c, float keep, const float (&dn)[4],
                                        const float (&a)[4], const float (&up)[4], const float (&b)[4],
                                        const float (&w)[4], float (&out)[4]) {
  float left, right;
  s_edges(c, a, left, right);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float l = j == 0 ? left : a[j - 1], r = j == 3 ? right : a[j + 1];
    const float nb = L.wx * (l + r) + L.wy * (dn[j] + up[j]);
    out[j] = keep * a[j] + w[j] * (b[j] + nb);
  }
}

__device__ __forceinline__ void s_put(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void s_get(const unsigned char* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <int N>
__device__ __forceinline__ void s_shift(float (&a)[N][4]) {
#pragma unroll
  for (int k = 0; k + 1 < N; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) a[k][j] = a[k + 1][j];
}
template <int N>
__device__ __forceinline__ void s_zero(float (&a)[N][4]) {
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) a[k][j] = 0.f;
}

// Walks rows p = y0 - halo .. y1 + halo - 1 (an even count): issue(p, slot)
// starts a row's copies, step(p, slot) uses it.  Unrolled by six: the period
// of the three-row rings and of the restriction's row pairs.
template <int BYTES, typename I, typename S>
__device__ __forceinline__ void s_walk(int p0, int n, unsigned char* ring, I&& issue, S&& step) {
#pragma unroll
  for (int i = 0; i < kSD; ++i) {
    if (i < n) issue(p0 + i, ring + i * BYTES);
    s_commit();
  }
  static_assert(kSSlots == 6, "the unrolled body names its slots");
#pragma unroll 1
  for (int i = 0; i < n; i += 6) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (i + j < n) {
        s_wait();
        step(p0 + i + j, ring + j * BYTES);
        if (i + j + kSD < n) issue(p0 + i + j + kSD, ring + ((j + kSD) % kSSlots) * BYTES);
        s_commit();
      }
    }
  }
}

// down leg: H sweeps from zero, x, restricted residual
template <int H>
__device__ __forceinline__ void s_down(const LevelDev& L, int u0, int u1, int y0, int y1, const float* __restrict__ b,
                                       float* __restrict__ x, float* __restrict__ bc, float omega,
                                       unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, omega);
  const float keep = 1.f - omega;
  const int cnx = L.nx >> 1;
  // index H (or 2) is the newest row; xs[k] holds the rows after sweep k + 1
  float bq[H + 1][4], wq[H + 1][4], xs[H][3][4];
  unsigned mq[H + 1];
  float rp0 = 0.f, rp1 = 0.f;
  s_zero(bq);
  s_zero(wq);
#pragma unroll
  for (int k = 0; k < H; ++k) s_zero(xs[k]);
#pragma unroll
  for (int k = 0; k <= H; ++k) mq[k] = 0u;
  s_walk<kSRowDown>(
      y0 - H, y1 - y0 + 2 * H, ring,
      [&](int p, unsigned char* slot) {
        const bool f = c.in && p >= 0 && p < L.ny;
        const int at = f ? p * L.nx + c.go : 0;
        s_copy16(s_addr(slot) + c.lane * 16, b + at, f);
        if (L.cell) s_copy<4>(s_addr(slot) + 512 + c.lane * 4, L.cell + at, f);
      },
      [&](int p, const unsigned char* slot) {
        s_shift(bq);
        s_shift(wq);
#pragma unroll
        for (int k = 0; k < H; ++k) s_shift(xs[k]);
#pragma unroll
        for (int k = 0; k < H; ++k) mq[k] = mq[k + 1];
        s_get(slot + c.lane * 16, bq[H]);
        mq[H] = s_cells(L, c, p, slot + 512);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          wq[H][j] = __shfl_sync(kFull, c.tabw, (int)(s_byte(mq[H], j) & 15u));
          xs[0][2][j] = wq[H][j] * bq[H][j];
        }
#pragma unroll
        for (int k = 1; k < H; ++k)
          s_sweep(L, c, keep, xs[k - 1][0], xs[k - 1][1], xs[k - 1][2], bq[H - k], wq[H - k], xs[k][2]);
        // row o: x and its residual, pairs of cells summed; the coarse cells
        // are written on the odd row
        const int o = p - H;
        const float(&v)[3][4] = xs[H - 1];
        float left, right, r[4];
        s_edges(c, v[1], left, right);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float l = j == 0 ? left : v[1][j - 1], rr = j == 3 ? right : v[1][j + 1];
          const float d = __shfl_sync(kFull, c.tabd, (int)(s_byte(mq[0], j) & 15u));
          const float nb = L.wx * (l + rr) + L.wy * (v[0][j] + v[2][j]);
          r[j] = s_byte(mq[0], j) ? bq[0][j] - (d * v[1][j] - nb) : 0.f;
        }
        if (o >= y0 && c.own) s_put(x + o * L.nx + c.gx, v[1]);
        if (o & 1) {
          if (o >= y0 && c.own)
            *reinterpret_cast<float2*>(bc + (o >> 1) * cnx + (c.gx >> 1)) =
                make_float2(0.25f * (rp0 + (r[0] + r[1])), 0.25f * (rp1 + (r[2] + r[3])));
        } else {
          rp0 = r[0] + r[1];
          rp1 = r[2] + r[3];
        }
      });
}

// up leg: x + s P e, H sweeps, output; returns the lane's share of (b, out)
template <int H>
__device__ __forceinline__ float s_up(const LevelDev& L, int u0, int u1, int y0, int y1, const float* __restrict__ b,
                                      const float* __restrict__ xin, float* __restrict__ xout,
                                      const float* __restrict__ e, float omega, float s, unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, omega);
  const float keep = 1.f - omega;
  const int cnx = L.nx >> 1;
  // xs[k] holds the rows after sweep k (0: the corrected input)
  float bq[H + 1][4], wq[H + 1][4], xs[H][3][4];
  float acc = 0.f;
  s_zero(bq);
  s_zero(wq);
#pragma unroll
  for (int k = 0; k < H; ++k) s_zero(xs[k]);
  s_walk<kSRowUp>(
      y0 - H, y1 - y0 + 2 * H, ring,
      [&](int p, unsigned char* slot) {
        const bool f = c.in && p >= 0 && p < L.ny;
        const int at = f ? p * L.nx + c.go : 0;
        const uint32_t sl = s_addr(slot);
        s_copy16(sl + c.lane * 16, xin + at, f);
        s_copy16(sl + 512 + c.lane * 16, b + at, f);
        s_copy<8>(sl + 1024 + c.lane * 8, e + (f ? (p >> 1) * cnx + (c.go >> 1) : 0), f);
        if (L.cell) s_copy<4>(sl + 1280 + c.lane * 4, L.cell + at, f);
      },
      [&](int p, const unsigned char* slot) {
        s_shift(bq);
        s_shift(wq);
#pragma unroll
        for (int k = 0; k < H; ++k) s_shift(xs[k]);
        float xv[4];
        s_get(slot + c.lane * 16, xv);
        s_get(slot + 512 + c.lane * 16, bq[H]);
        const float2 ev = *reinterpret_cast<const float2*>(slot + 1024 + c.lane * 8);
        const unsigned m = s_cells(L, c, p, slot + 1280);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          wq[H][j] = __shfl_sync(kFull, c.tabw, (int)(s_byte(m, j) & 15u));
          xs[0][2][j] = s_byte(m, j) ? xv[j] + s * (j < 2 ? ev.x : ev.y) : 0.f;
        }
        float z[4];
#pragma unroll
        for (int k = 1; k <= H; ++k)
          s_sweep(L, c, keep, xs[k - 1][0], xs[k - 1][1], xs[k - 1][2], bq[H - k], wq[H - k],
                  *(k < H ? &xs[k < H ? k : 0][2] : &z));
        const int o = p - H;
        if (o >= y0 && c.own) {
          s_put(xout + o * L.nx + c.gx, z);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc = fmaf(wq[0][j] > 0.f ? bq[0][j] : 0.f, z[j], acc);
        }
      });
  return acc;
}

// p = z + beta p_old, Ap; returns the lane's share of (p, Ap)
__device__ __forceinline__ float s_pupdate(const LevelDev& L, int u0, int u1, int y0, int y1,
                                           const float* __restrict__ z, const float* __restrict__ pold,
                                           float* __restrict__ pnew, float* __restrict__ Ap, float beta, bool first,
                                           unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, 1.f);
  float ps[3][4];
  unsigned mp = 0u;
  float acc = 0.f;
  s_zero(ps);
  s_walk<kSRowUp>(
      y0 - 1, y1 - y0 + 2, ring,
      [&](int p, unsigned char* slot) {
        const bool f = c.in && p >= 0 && p < L.ny;
        const int at = f ? p * L.nx + c.go : 0;
        const uint32_t sl = s_addr(slot);
        s_copy16(sl + c.lane * 16, z + at, f);
        if (!first) s_copy16(sl + 512 + c.lane * 16, pold + at, f);
        if (L.cell) s_copy<4>(sl + 1280 + c.lane * 4, L.cell + at, f);
      },
      [&](int p, const unsigned char* slot) {
        s_shift(ps);
        float zv[4], pv[4] = {0.f, 0.f, 0.f, 0.f};
        s_get(slot + c.lane * 16, zv);
        if (!first) s_get(slot + 512 + c.lane * 16, pv);
        const unsigned m = s_cells(L, c, p, slot + 1280);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          ps[2][j] = s_byte(m, j) ? (first ? zv[j] : fmaf(beta, pv[j], zv[j])) : 0.f;
        const int o = p - 1;
        float left, right, ap[4];
        s_edges(c, ps[1], left, right);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float l = j == 0 ? left : ps[1][j - 1], r = j == 3 ? right : ps[1][j + 1];
          const float d = __shfl_sync(kFull, c.tabd, (int)(s_byte(mp, j) & 15u));
          float nb = 0.f;
          nb += L.wx * l;
          nb += L.wx * r;
          nb += L.wy * ps[0][j];
          nb += L.wy * ps[2][j];
          ap[j] = s_byte(mp, j) ? d * ps[1][j] - nb : 0.f;
        }
        mp = m;
        if (o >= y0 && c.own) {
          s_put(pnew + o * L.nx + c.gx, ps[1]);
          s_put(Ap + o * L.nx + c.gx, ap);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc = fmaf(ps[1][j], ap[j], acc);
        }
      });
  return acc;
}

}  // namespace npmg
