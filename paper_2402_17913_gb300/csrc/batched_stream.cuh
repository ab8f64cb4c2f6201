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
// What bounds it: 256 instances of sides 64 to 512, three sweeps: the p and
// x / r updates run at the copy rate, the two finest legs at 0.6 of it (four
// warps per scheduler at 128 registers, about seven cycles an issue; three
// blocks per SM at 80 registers spill: 36 ms).  The block tiles before staged
// 72 x 38 cells for 64 x 32 behind seven block barriers, 6 us a tile at four
// blocks per SM: 28.1 -> 21.0 ms a solve, -> 19.7 with paired arithmetic and
// with the phases walking the list up and down in turn, -> 18.8 with Ap
// formed again instead of stored, -> 18.2 with cheaper barriers and sums, ->
// 17.5 with the refinement residual on strips too.
#pragma once

#include "npmg_internal.cuh"
#include "refine.cuh"

namespace npmg {

constexpr int kSD = 5;          // rows in flight ahead of the row in use
constexpr int kSSlots = kSD + 1;
constexpr int kSRowDown = 32 * 16 + 32 * 4;                     // b, cell bytes
constexpr int kSRowUp = 2 * 32 * 16 + 32 * 8 + 32 * 4;          // x (or z), b (or p), e, cell bytes
constexpr int kSRowXr = 3 * 32 * 16 + 32 * 4;                  // p, d, r, cell bytes
constexpr int kSRowRes = 4 * 32 * 16 + 32 * 4;                 // iterate (hi, lo), d, b, cell bytes
constexpr int kSRing = kSSlots * kSRowRes;                      // bytes of one warp's ring
static_assert(kSRowRes >= kSRowXr && kSRowXr >= kSRowUp && kSRowUp >= kSRowDown, "the ring holds the longest rows");
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

// The four cells of a lane as two pairs: a pair's multiply-add is one
// instruction (fma.rn.f32x2), and issue slots are what the sweeps run out of.
struct Quad {
  float2 a, b;
  __device__ __forceinline__ float2 pair(int q) const { return q ? b : a; }
  __device__ __forceinline__ float get(int j) const { return j == 0 ? a.x : j == 1 ? a.y : j == 2 ? b.x : b.y; }
  __device__ __forceinline__ void set(int j, float v) {
    if (j == 0) a.x = v;
    else if (j == 1) a.y = v;
    else if (j == 2) b.x = v;
    else b.y = v;
  }
};
__device__ __forceinline__ float2 s_dup(float v) { return make_float2(v, v); }

// sums of the two neighbours in x of each cell of a row: 0 beyond the warp,
// which is the level's edge or the spoilt side of a halo lane
__device__ __forceinline__ Quad s_xsum(const SLane& c, const Quad& v) {
  float left = __shfl_up_sync(kFull, v.b.y, 1);
  float right = __shfl_down_sync(kFull, v.a.x, 1);
  if (c.lane == 0) left = 0.f;
  if (c.lane == 31) right = 0.f;
  Quad o;
  o.a = make_float2(left + v.a.y, v.a.x + v.b.x);
  o.b = make_float2(v.a.y + v.b.y, v.b.x + right);
  return o;
}

// f + wx (left + right) + wy (below + above)
__device__ __forceinline__ Quad s_stencil(const SLane& c, float2 wx, float2 wy, const Quad& f, const Quad& dn,
                                          const Quad& v, const Quad& up) {
  const Quad x = s_xsum(c, v);
  Quad o;
  o.a = __ffma2_rn(wx, x.a, __ffma2_rn(wy, __fadd2_rn(dn.a, up.a), f.a));
  o.b = __ffma2_rn(wx, x.b, __ffma2_rn(wy, __fadd2_rn(dn.b, up.b), f.b));
  return o;
}

// one sweep on row v between rows dn and up
__device__ __forceinline__ Quad s_sweep(const SLane& c, float2 wx, float2 wy, float2 keep, const Quad& dn,
                                        const Quad& v, const Quad& up, const Quad& b, const Quad& w) {
  const Quad t = s_stencil(c, wx, wy, b, dn, v, up);
  Quad o;
  o.a = __ffma2_rn(w.a, t.a, __fmul2_rn(keep, v.a));
  o.b = __ffma2_rn(w.b, t.b, __fmul2_rn(keep, v.b));
  return o;
}

__device__ __forceinline__ void s_put(float* p, const Quad& v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
}
__device__ __forceinline__ Quad s_get(const unsigned char* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  return Quad{make_float2(q.x, q.y), make_float2(q.z, q.w)};
}
__device__ __forceinline__ Quad s_table(const SLane& c, float entry, unsigned m) {
  Quad o;
#pragma unroll
  for (int j = 0; j < 4; ++j) o.set(j, __shfl_sync(kFull, entry, (int)(s_byte(m, j) & 15u)));
  return o;
}
template <int N>
__device__ __forceinline__ void s_shift(Quad (&a)[N]) {
#pragma unroll
  for (int k = 0; k + 1 < N; ++k) a[k] = a[k + 1];
}
template <int N>
__device__ __forceinline__ void s_zero(Quad (&a)[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) a[k].a = a[k].b = make_float2(0.f, 0.f);
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
  const float2 wx = s_dup(L.wx), wy = s_dup(L.wy), keep = s_dup(1.f - omega);
  const int cnx = L.nx >> 1;
  // index H (or 2) is the newest row; xs[k] holds the rows after sweep k + 1
  Quad bq[H + 1], wq[H + 1], xs[H][3];
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
        bq[H] = s_get(slot + c.lane * 16);
        mq[H] = s_cells(L, c, p, slot + 512);
        wq[H] = s_table(c, c.tabw, mq[H]);
        xs[0][2].a = __fmul2_rn(wq[H].a, bq[H].a);
        xs[0][2].b = __fmul2_rn(wq[H].b, bq[H].b);
#pragma unroll
        for (int k = 1; k < H; ++k)
          xs[k][2] = s_sweep(c, wx, wy, keep, xs[k - 1][0], xs[k - 1][1], xs[k - 1][2], bq[H - k], wq[H - k]);
        // row o: x and its residual b + nb - d x, pairs of cells summed; the
        // coarse cells are written on the odd row
        const int o = p - H;
        const Quad(&v)[3] = xs[H - 1];
        const Quad d = s_table(c, c.tabd, mq[0]), t = s_stencil(c, wx, wy, bq[0], v[0], v[1], v[2]);
        float r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) r[j] = s_byte(mq[0], j) ? fmaf(-d.get(j), v[1].get(j), t.get(j)) : 0.f;
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
  const float2 wx = s_dup(L.wx), wy = s_dup(L.wy), keep = s_dup(1.f - omega);
  const int cnx = L.nx >> 1;
  // xs[k] holds the rows after sweep k (0: the corrected input, H: the output)
  Quad bq[H + 1], wq[H + 1], xs[H + 1][3];
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
        const Quad xv = s_get(slot + c.lane * 16);
        bq[H] = s_get(slot + 512 + c.lane * 16);
        const float2 ev = *reinterpret_cast<const float2*>(slot + 1024 + c.lane * 8);
        const unsigned m = s_cells(L, c, p, slot + 1280);
        wq[H] = s_table(c, c.tabw, m);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          xs[0][2].set(j, s_byte(m, j) ? fmaf(s, j < 2 ? ev.x : ev.y, xv.get(j)) : 0.f);
#pragma unroll
        for (int k = 1; k <= H; ++k)
          xs[k][2] = s_sweep(c, wx, wy, keep, xs[k - 1][0], xs[k - 1][1], xs[k - 1][2], bq[H - k], wq[H - k]);
        const int o = p - H;
        if (o >= y0 && c.own) {
          const Quad& z = xs[H][2];
          s_put(xout + o * L.nx + c.gx, z);
          // b off the fluid stays out of the sum
#pragma unroll
          for (int j = 0; j < 4; ++j) acc = fmaf(wq[0].get(j) > 0.f ? bq[0].get(j) : 0.f, z.get(j), acc);
        }
      });
  return acc;
}

// A p of row v between rows dn and up (0 off the fluid)
__device__ __forceinline__ Quad s_apply(const SLane& c, float2 nwx, float2 nwy, unsigned m, const Quad& dn,
                                        const Quad& v, const Quad& up) {
  Quad t = s_table(c, c.tabd, m);
  t.a = __fmul2_rn(t.a, v.a);
  t.b = __fmul2_rn(t.b, v.b);
  t = s_stencil(c, nwx, nwy, t, dn, v, up);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (!s_byte(m, j)) t.set(j, 0.f);
  return t;
}

// p = z + beta p_old and the lane's share of (p, Ap)
__device__ __forceinline__ float s_pupdate(const LevelDev& L, int u0, int u1, int y0, int y1,
                                           const float* __restrict__ z, const float* __restrict__ pold,
                                           float* __restrict__ pnew, float beta, bool first, unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, 1.f);
  const float2 wx = s_dup(-L.wx), wy = s_dup(-L.wy), bt = s_dup(beta);
  Quad ps[3];
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
        Quad v = s_get(slot + c.lane * 16);
        const unsigned m = s_cells(L, c, p, slot + 1280);
        if (!first) {
          const Quad pv = s_get(slot + 512 + c.lane * 16);
          v.a = __ffma2_rn(bt, pv.a, v.a);
          v.b = __ffma2_rn(bt, pv.b, v.b);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) ps[2].set(j, s_byte(m, j) ? v.get(j) : 0.f);
        const int o = p - 1;
        const Quad ap = s_apply(c, wx, wy, mp, ps[0], ps[1], ps[2]);
        mp = m;
        if (o >= y0 && c.own) {
          s_put(pnew + o * L.nx + c.gx, ps[1]);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc = fmaf(ps[1].get(j), ap.get(j), acc);
        }
      });
  return acc;
}

// d += alpha p (d = alpha p on the first iteration), r -= alpha Ap with Ap
// formed again from p, the values (p, Ap) was summed from: both updates run
// at the copy rate, and Ap stored and read back was 8 of their 41 bytes per
// cell (256 instances: the two phases 6.25 -> 4.86 ms of a solve).  Returns
// the lane's share of ||r||^2.
__device__ __forceinline__ float s_xrupdate(const LevelDev& L, int u0, int u1, int y0, int y1,
                                            const float* __restrict__ pv, float* __restrict__ dv,
                                            float* __restrict__ rv, float alpha, bool first, unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, 1.f);
  const float2 wx = s_dup(-L.wx), wy = s_dup(-L.wy), al = s_dup(alpha), na = s_dup(-alpha);
  Quad ps[3];
  unsigned mp = 0u;
  float acc = 0.f;
  s_zero(ps);
  s_walk<kSRowXr>(
      y0 - 1, y1 - y0 + 2, ring,
      [&](int p, unsigned char* slot) {
        // row p of p and of the cell bytes, row p - 1 of d and r
        const bool f = c.in && p >= 0 && p < L.ny, fo = c.own && p > y0;
        const int at = f ? p * L.nx + c.go : 0, ao = fo ? (p - 1) * L.nx + c.go : 0;
        const uint32_t sl = s_addr(slot);
        s_copy16(sl + c.lane * 16, pv + at, f);
        if (!first) s_copy16(sl + 512 + c.lane * 16, dv + ao, fo);
        s_copy16(sl + 1024 + c.lane * 16, rv + ao, fo);
        if (L.cell) s_copy<4>(sl + 1536 + c.lane * 4, L.cell + at, f);
      },
      [&](int p, const unsigned char* slot) {
        s_shift(ps);
        ps[2] = s_get(slot + c.lane * 16);
        const unsigned m = s_cells(L, c, p, slot + 1536);
        const Quad ap = s_apply(c, wx, wy, mp, ps[0], ps[1], ps[2]);
        mp = m;
        const int o = p - 1;
        if (o >= y0 && c.own) {
          Quad d, r = s_get(slot + 1024 + c.lane * 16);
          if (first) {
            d.a = __fmul2_rn(al, ps[1].a);
            d.b = __fmul2_rn(al, ps[1].b);
          } else {
            d = s_get(slot + 512 + c.lane * 16);
            d.a = __ffma2_rn(al, ps[1].a, d.a);
            d.b = __ffma2_rn(al, ps[1].b, d.b);
          }
          r.a = __ffma2_rn(na, ap.a, r.a);
          r.b = __ffma2_rn(na, ap.b, r.b);
          s_put(dv + o * L.nx + c.gx, d);
          s_put(rv + o * L.nx + c.gx, r);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc = fmaf(r.get(j), r.get(j), acc);
        }
      });
  return acc;
}

// Refinement residual of the float-float iterate after x += sigma_old d (when
// `update`), r = (c b - A' x) inv_sig in float-float on the fluid cells.  As
// block tiles between two barriers it ran at a fifth of the copy rate (256
// instances: 18.2 -> 17.5 ms a solve); returns the lane's share of ||r||^2 (before inv_sig).
// kx, ky: link counts; the iterate and d hold 0 off the fluid.
__device__ __forceinline__ float s_resid(const LevelDev& L, int u0, int u1, int y0, int y1,
                                         const float* __restrict__ b, const float2* __restrict__ xin,
                                         float2* __restrict__ xo, const float* __restrict__ dv,
                                         float* __restrict__ rv, ff wx, ff wy, ff cff, bool update, float sig_old,
                                         float inv_sig, unsigned char* ring) {
  const SLane c = s_lane(L, u0, u1, 1.f);
  float hi[3][4], lo[3][4];
  unsigned mp = 0u;
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) hi[k][j] = lo[k][j] = 0.f;
  s_walk<kSRowRes>(
      y0 - 1, y1 - y0 + 2, ring,
      [&](int p, unsigned char* slot) {
        // row p of the iterate, d and the cell bytes, row p - 1 of b
        const bool f = c.in && p >= 0 && p < L.ny, fo = c.own && p > y0;
        const int at = f ? p * L.nx + c.go : 0, ao = fo ? (p - 1) * L.nx + c.go : 0;
        const uint32_t sl = s_addr(slot);
        s_copy16(sl + c.lane * 32, xin + at, f);
        s_copy16(sl + c.lane * 32 + 16, xin + at + 2, f);
        if (update) s_copy16(sl + 1024 + c.lane * 16, dv + at, f);
        s_copy16(sl + 1536 + c.lane * 16, b + ao, fo);
        if (L.cell) s_copy<4>(sl + 2048 + c.lane * 4, L.cell + at, f);
      },
      [&](int p, const unsigned char* slot) {
        const Quad q0 = s_get(slot + c.lane * 32), q1 = s_get(slot + c.lane * 32 + 16);
        const float xh[4] = {q0.a.x, q0.b.x, q1.a.x, q1.b.x}, xl[4] = {q0.a.y, q0.b.y, q1.a.y, q1.b.y};
        Quad d;
        d.a = d.b = make_float2(0.f, 0.f);
        if (update) d = s_get(slot + 1024 + c.lane * 16);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          hi[0][j] = hi[1][j];
          lo[0][j] = lo[1][j];
          hi[1][j] = hi[2][j];
          lo[1][j] = lo[2][j];
          ff v = {xh[j], xl[j]};
          if (update) {
            const ff s2 = two_sum(xh[j], sig_old * d.get(j));
            v = quick_two_sum(s2.hi, s2.lo + xl[j]);
          }
          hi[2][j] = v.hi;
          lo[2][j] = v.lo;
        }
        const unsigned m = s_cells(L, c, p, slot + 2048);
        float lh = __shfl_up_sync(kFull, hi[1][3], 1), ll = __shfl_up_sync(kFull, lo[1][3], 1);
        float rh = __shfl_down_sync(kFull, hi[1][0], 1), rl = __shfl_down_sync(kFull, lo[1][0], 1);
        if (c.lane == 0) lh = ll = 0.f;
        if (c.lane == 31) rh = rl = 0.f;
        const int o = p - 1;
        if (o >= y0 && c.own) {
          const Quad bb = s_get(slot + 1536 + c.lane * 16);
          Quad r;
          float oh[4], ol[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const unsigned mj = s_byte(mp, j);
            const ff xc = {hi[1][j], lo[1][j]};
            const ff xw = {j == 0 ? lh : hi[1][j - 1], j == 0 ? ll : lo[1][j - 1]};
            const ff xe = {j == 3 ? rh : hi[1][j + 1], j == 3 ? rl : lo[1][j + 1]};
            const ff xd = {hi[0][j], lo[0][j]}, xu = {hi[2][j], lo[2][j]};
            ff ax = ff_mul(ff_add(ff_mul(xc, ff{(float)(mj & 3u), 0.f}), ff_neg(ff_add(xw, xe))), wx);
            ax = ff_add(ax, ff_mul(ff_add(ff_mul(xc, ff{(float)((mj >> 2) & 3u), 0.f}), ff_neg(ff_add(xd, xu))), wy));
            const ff rr = ff_add(ff_mul(ff{bb.get(j), 0.f}, cff), ff_neg(ax));
            const float rs = mj ? rr.hi + rr.lo : 0.f;
            r.set(j, rs * inv_sig);
            acc = fmaf(rs, rs, acc);
            oh[j] = mj ? xc.hi : 0.f;
            ol[j] = mj ? xc.lo : 0.f;
          }
          s_put(rv + o * L.nx + c.gx, r);
          if (update) {
            float4* out = reinterpret_cast<float4*>(xo + o * L.nx + c.gx);
            out[0] = make_float4(oh[0], ol[0], oh[1], ol[1]);
            out[1] = make_float4(oh[2], ol[2], oh[3], ol[3]);
          }
        }
        mp = m;
      });
  return acc;
}

}  // namespace npmg
