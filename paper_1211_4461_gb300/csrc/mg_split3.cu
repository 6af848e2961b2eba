// 3D V(1,1) red-black Gauss-Seidel cycles on colour-split arrays (Sec. 4).
//
// Bound by memory traffic: a half sweep reads the other colour of u, its own
// colour of b and 1/d and writes its own colour of u.  With the colours
// interleaved every one of those streams moves whole cache lines, both colours
// of each array; split by colour a half sweep moves half as much.
//
// Layout: row (iy, iz) of a colour holds its points in order, x = 2 j + o in
// slot j with o the row's parity of the colour (red: (iy + iz + 1) mod 2, black
// the other), HP slots a row (a multiple of four; slots outside the domain are
// zero).  The six neighbours of slot j lie in the other colour's array: slots
// j + o - 1 and j + o of the same row, slot j of the rows above, below, before
// and behind.  A thread takes two slots of a row (one 16-byte access).
//
// A cycle has four passes per level instead of eight:
//  - the red half sweep from zero, u = d^{-1} b, is folded into the full
//    weighting that forms b;
//  - no residual array: after the black half sweep every black equation holds
//    and the red residual is r = c sum_nbr delta, delta the change of the black
//    values since the red half sweep (their values themselves when the iterate
//    entered as zero), because the red half sweep left d u = b + c sum_nbr u_old.
//    Full weighting of r (centre 1/8, the twelve red edge points 1/32) then is
//    one 38-point sum over delta: 1/4 at the 6 points at distance (1,0,0), 3/32
//    at the 8 at (1,1,1), 1/32 at the 24 at (2,1,0), times c;
//  - the prolongation is needed at the black points only, as neighbours of the
//    red half sweep (the black half sweep overwrites them): the red half sweep
//    adds the interpolated correction's neighbour sum, formed from the coarse
//    values directly;
//  - the last black half sweep writes both colours in natural order.
// 257^3 FP32 cycle through the public call (natural order in and out): 358 us,
// 670 with interleaved colours.  Passes of 255^3 from a cold L2 (share of DRAM's
// peak): half sweep 42 us (75 %), with the black change 55 (82 %), prolonging 64
// (52 %), into natural order 57 (66 %); the 38-point full weighting 37 (28 %: load
// latency).  Interleaved: 80 a half sweep, 125 with the prolongation's pass, 123 for
// residual and full weighting.
#include "csff_internal.h"

#include <cmath>

namespace csff {
namespace {

struct Pair { float2 a, b; };
__device__ __forceinline__ float2 zc() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ Pair ld2(const float2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return Pair{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void st2(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
// a + b c for complex values, a chain of fused multiply-adds
template <typename C> __device__ __forceinline__ C cfma(C a, C b, C c) {
  return mk<C>(fma(b.x, c.x, fma(-b.y, c.y, a.x)), fma(b.x, c.y, fma(b.y, c.x, a.y)));
}

// d^{-1} t.  d^{-1} is held as d0 + dv, d0 the level's FP32 value without the
// potential and dv the FP32 difference: rounding d^{-1} itself shifts every
// equation by the same 2^-25 |d|, which the folded residual (no explicit b - A u)
// would pass to the coarse levels as a residual.  dv's products come first: added
// to a rounded d0 t, terms below half its last place would be lost at every point
// alike and leave two thirds of that shift (a cycle from an iterate that cycles
// left, 65^3, k = 1, no potential: 20.1 units of 2^-24 off on a box of 5, 5.8 on one
// of 15; in this order 3.0 and 1.9; per-level passes 2.1 and 1.7).
__device__ __forceinline__ float2 dinv_mul(float2 d0, float2 dv, float2 t) {
  return make_float2(fmaf(d0.x, t.x, fmaf(-d0.y, t.y, fmaf(dv.x, t.x, -(dv.y * t.y)))),
                     fmaf(d0.x, t.y, fmaf(d0.y, t.x, fmaf(dv.x, t.y, dv.y * t.x))));
}

// Launches of at most one CTA an SM (the small levels) let their dependent be set
// up as soon as they have passed their own wait; a sweep's and a full weighting's
// 1/d, which no pass writes, is loaded before that wait.
__device__ __forceinline__ void wait_and_trigger() {
  pdl_prologue();
  if (gridDim.x * gridDim.y * gridDim.z <= 152u) pdl_trigger();
}

// coordinates of a thread: slot pair, row, plane
struct At { int j, iy, iz; long long row; };
__device__ __forceinline__ bool at(int m, int HP, At& p) {
  p.j = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
  p.iy = blockIdx.y * blockDim.y + threadIdx.y;
  p.iz = blockIdx.z;
  p.row = (long long)p.iz * m + p.iy;
  return p.j < HP && p.iy < m;
}

// Natural order in: b by colour and the red half sweep, from zero (u = d^{-1} b,
// NAT_U false) or from a natural iterate, whose black points go to ub.
template <bool NAT_U>
__global__ void k3s_first(const float2* __restrict__ b_nat, const float2* __restrict__ u_nat,
                          const float2* __restrict__ dr, float2 c, float2 d0, int m, int HP, float2* __restrict__ br,
                          float2* __restrict__ bb, float2* __restrict__ ub, float2* __restrict__ ur) {
  using C = float2;
  wait_and_trigger();
  At p;
  if (!at(m, HP, p)) return;
  const int o = (p.iy + p.iz + 1) & 1;                 // red parity of the row
  const C* row = b_nat + p.row * m;
  const int x = 2 * p.j, x0 = x + o, x1 = x0 + 2;
  C v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = x + k < m ? row[x + k] : zc();
  const long long s = p.row * HP + p.j;
  const Pair d = ld2(dr + s);
  C s0 = zc(), s1 = zc();
  if constexpr (NAT_U) {
    const C* u = u_nat + p.row * m;
    const long long pl = (long long)m * m;
    const bool i0 = x0 < m, i1 = x1 < m;
    const C xl = (x0 > 0 && x0 - 1 < m) ? u[x0 - 1] : zc(), xm = x0 + 1 < m ? u[x0 + 1] : zc(),
            xr = x1 + 1 < m ? u[x1 + 1] : zc();
    auto at_row = [&](bool in, long long off, C& q0, C& q1) {
      q0 = in && i0 ? u[x0 + off] : zc();
      q1 = in && i1 ? u[x1 + off] : zc();
    };
    C yl0, yl1, yr0, yr1, zl0, zl1, zr0, zr1;
    at_row(p.iy > 0, -m, yl0, yl1);
    at_row(p.iy < m - 1, m, yr0, yr1);
    at_row(p.iz > 0, -pl, zl0, zl1);
    at_row(p.iz < m - 1, pl, zr0, zr1);
    s0 = cadd(cadd(cadd(xl, xm), cadd(yl0, yr0)), cadd(zl0, zr0));
    s1 = cadd(cadd(cadd(xm, xr), cadd(yl1, yr1)), cadd(zl1, zr1));
    // black slots: x = 2 j + 1 - o
    st2(ub + s, o ? xl : xm, o ? xm : xr);
  }
  const C r0 = o ? v[1] : v[0], r1 = o ? v[3] : v[2];
  st2(br + s, r0, r1);
  st2(bb + s, o ? v[0] : v[1], o ? v[2] : v[3]);
  st2(ur + s, x0 < m ? dinv_mul(d0, d.a, NAT_U ? cfma(r0, c, s0) : r0) : zc(),
      x1 < m ? dinv_mul(d0, d.b, NAT_U ? cfma(r1, c, s1) : r1) : zc());
}

// a level's d^{-1} by colour: FP64 as stored; FP32 as the difference to d0 of
// 1 / (6 c - q) with c the FP32 value that the sweeps multiply by, to first
// order in dc, six times the rounding of c (relative 2^-25: its square and the
// rounding of this term lie far below the result's)
__global__ void k3s_split(const double2* __restrict__ dinv, float2 dc, float2 d0, int m, int HP,
                          float2* __restrict__ red, float2* __restrict__ black) {
  using C = float2;
  At p;
  if (!at(m, HP, p)) return;
  const int o = (p.iy + p.iz + 1) & 1, x = 2 * p.j;
  C v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = zc();
    if (x + k < m) {
      const double2 di = dinv[p.row * m + x + k];
      const float2 f = make_float2((float)di.x, (float)di.y), t = cmul(cmul(f, f), dc);
      v[k] = make_float2((float)(di.x - (double)d0.x) - t.x, (float)(di.y - (double)d0.y) - t.y);
    }
  }
  const long long s = p.row * HP + p.j;
  st2(red + s, o ? v[1] : v[0], o ? v[3] : v[2]);
  st2(black + s, o ? v[0] : v[1], o ? v[2] : v[3]);
}

// largest |6 c / d| of a level (as bits; a d of zero gives infinity or NaN)
__global__ void k3s_worst(const float2* __restrict__ dinv, float c6, long long N, unsigned* __restrict__ worst) {
  unsigned w = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const float2 d = make_float2(c6 * dinv[i].x, c6 * dinv[i].y);
    w = max(w, __float_as_uint(sqrtf(fmaf(d.x, d.x, d.y * d.y))));
  }
  w = __reduce_max_sync(0xffffffffu, w);
  if ((threadIdx.x & 31) == 0) atomicMax(worst, w);
}

// The coarse correction e is kept with a ring of zeros: node (X, Y, Z), X, Y, Z
// in [0, mc + 1], at (Z (mc + 2) + Y) pe + X + 1, so that the columns X = j + 1,
// j + 2 of an even slot j are one aligned access and no load is tested.
//
// Neighbour sum of the interpolated correction P e at the red slots j, j + 1 of
// row (iy, iz).  Node indices: a red node has an even number of odd indices.
// All even (a coarse node K): 3 e_K + 1/2 sum of its six coarse neighbours.
// Two odd: with S4 the sum of the four coarse corners around the point in the
// plane of its odd axes, 5/4 S4 + 1/8 (S4 one coarse plane up and one down the
// even axis).
__device__ __forceinline__ Pair prolong_nbr(const float2* __restrict__ e, int pe, int mc, int j, int iy, int iz) {
  using C = float2;
  const bool oy = !(iy & 1), oz = !(iz & 1);           // odd node indices
  const int Y = (iy + 1) >> 1, Z = (iz + 1) >> 1;      // coarse node at or below
  const long long pz = (long long)(mc + 2) * pe;
  const C* r = e + Z * pz + (long long)Y * pe + j;     // r[k]: column X = j - 1 + k
  Pair out;
  if (oy == oz) {                                      // x even: coarse columns j + 1 and j + 2
    if (!oy) {
      const C e0 = r[1], e3 = r[4];
      const Pair m = ld2(r + 2), a = ld2(r + 2 - pe), b = ld2(r + 2 + pe), f = ld2(r + 2 - pz), g = ld2(r + 2 + pz);
      const C s0 = cadd(cadd(e0, m.b), cadd(cadd(a.a, b.a), cadd(f.a, g.a)));
      const C s1 = cadd(cadd(m.a, e3), cadd(cadd(a.b, b.b), cadd(f.b, g.b)));
      out.a = cadd(cscale(m.a, 3.f), cscale(s0, 0.5f));
      out.b = cadd(cscale(m.b, 3.f), cscale(s1, 0.5f));
    } else {
      C s[4];
      const C *r2 = r + pe, *r3 = r + pz, *r4 = r3 + pe;
      const Pair m1 = ld2(r + 2), m2 = ld2(r2 + 2), m3 = ld2(r3 + 2), m4 = ld2(r4 + 2);
      s[0] = cadd(cadd(r[1], r2[1]), cadd(r3[1], r4[1]));
      s[1] = cadd(cadd(m1.a, m2.a), cadd(m3.a, m4.a));
      s[2] = cadd(cadd(m1.b, m2.b), cadd(m3.b, m4.b));
      s[3] = cadd(cadd(r[4], r2[4]), cadd(r3[4], r4[4]));
      out.a = cadd(cscale(s[1], 1.25f), cscale(cadd(s[0], s[2]), 0.125f));
      out.b = cadd(cscale(s[2], 1.25f), cscale(cadd(s[1], s[3]), 0.125f));
    }
  } else {                                             // x odd: between coarse columns j and j + 1 (j + 1 and j + 2)
    C t0[3], t1[3];                                    // S4 at the even axis' plane below, at, above
    const long long step = oy ? pz : pe, pair = oy ? pe : pz;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const C* q = r + (k - 1) * step;
      const Pair a = ld2(q + 2), b = ld2(q + pair + 2);
      const C c0 = cadd(q[1], q[pair + 1]), c1 = cadd(a.a, b.a), c2 = cadd(a.b, b.b);
      t0[k] = cadd(c0, c1);
      t1[k] = cadd(c1, c2);
    }
    out.a = cadd(cscale(t0[1], 1.25f), cscale(cadd(t0[0], t0[2]), 0.125f));
    out.b = cadd(cscale(t1[1], 1.25f), cscale(cadd(t1[0], t1[2]), 0.125f));
  }
  return out;
}

// One colour of a sweep: u <- d^{-1} (b + c sum_nbr u), uo the other colour.
//  PLAIN: u
//  PROLONG (red): the neighbours are u + P e
//  DELTA (black): also delta = u_new - u_old
//  NAT (black): both colours to nat in natural order
//  RING (black): both colours to nat as the ringed correction, rows nat_pitch apart
// PLAIN: 32 registers, so that an SM holds its 64 warps (255^3: 38.7 us, 42.6 at 34)
enum Mode { PLAIN, PROLONG, DELTA, NAT, RING };
template <int COLOUR, int MODE>
__global__ void __launch_bounds__(256, MODE == PLAIN ? 8 : 4) k3s_sweep(const float2* __restrict__ uo, const float2* __restrict__ b, const float2* __restrict__ dinv,
                          float2 c, float2 d0, int m, int HP, float2* u, float2* __restrict__ delta,
                          const float2* __restrict__ e, int pe, int mc, float2* __restrict__ nat, int nat_pitch) {
  using C = float2;
  At p;
  if (!at(m, HP, p)) return;
  const int o = (p.iy + p.iz + 1 + COLOUR) & 1;
  const long long s = p.row * HP + p.j;
  const Pair dv = ld2(dinv + s);
  wait_and_trigger();
  const long long plane = (long long)m * HP;
  const Pair zero{zc(), zc()};
  const Pair mid = ld2(uo + s);
  const int je = o ? p.j + 2 : p.j - 1;                 // the row's third neighbour slot
  const C edge = (je >= 0 && je < HP) ? uo[s + (je - p.j)] : zc();
  const Pair yl = p.iy > 0 ? ld2(uo + s - HP) : zero, yr = p.iy < m - 1 ? ld2(uo + s + HP) : zero;
  const Pair zl = p.iz > 0 ? ld2(uo + s - plane) : zero, zr = p.iz < m - 1 ? ld2(uo + s + plane) : zero;
  const Pair bv = ld2(b + s);
  Pair old = zero;
  if constexpr (MODE == DELTA) old = ld2(u + s);
  // x - 1 and x + 1 of both slots
  const C a0 = o ? mid.a : edge, a1 = o ? mid.b : mid.a, b0 = o ? mid.b : mid.a, b1 = o ? edge : mid.b;
  // pairs first: fewer roundings of large partial sums
  C s0 = cadd(cadd(cadd(a0, a1), cadd(yl.a, yr.a)), cadd(zl.a, zr.a));
  C s1 = cadd(cadd(cadd(b0, b1), cadd(yl.b, yr.b)), cadd(zl.b, zr.b));
  if constexpr (MODE == PROLONG) {
    const Pair q = prolong_nbr(e, pe, mc, p.j, p.iy, p.iz);
    s0 = cadd(s0, q.a);
    s1 = cadd(s1, q.b);
  }
  const int x0 = 2 * p.j + o, x1 = x0 + 2;
  const C v0 = x0 < m ? dinv_mul(d0, dv.a, cfma(bv.a, c, s0)) : zc();
  const C v1 = x1 < m ? dinv_mul(d0, dv.b, cfma(bv.b, c, s1)) : zc();
  if constexpr (MODE != NAT && MODE != RING) st2(u + s, v0, v1);
  if constexpr (MODE == DELTA) st2(delta + s, csub(v0, old.a), csub(v1, old.b));
  if constexpr (MODE == RING) {
    // slots outside the domain are zero, as the ring has to stay
    C* n = nat + ((long long)(p.iz + 1) * (m + 2) + p.iy + 1) * nat_pitch + 2 * p.j + 2;
    st2(n, o ? mid.a : v0, o ? v0 : mid.a);
    if (2 * p.j + 2 < m) st2(n + 2, o ? mid.b : v1, o ? v1 : mid.b);
  }
  if constexpr (MODE == NAT) {
    C* n = nat + p.row * m + 2 * p.j;
    const C w[4] = {o ? mid.a : v0, o ? v0 : mid.a, o ? mid.b : v1, o ? v1 : mid.b};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (2 * p.j + k < m) n[k] = w[k];
  }
}

// Full weighting of the red residual c sum_nbr delta into the coarse level:
// its b in both colours and the red half sweep u = d^{-1} b from zero, or (the
// coarsest level, nat) b in natural order.  A thread takes the coarse points
// P, P + 1 (P even) of a row: one of them red.
__global__ void k3s_restrict(const float2* __restrict__ delta, int m, int HP, float2 c, int mc, int HPc,
                             float2* __restrict__ br, float2* __restrict__ bb, const float2* __restrict__ dr,
                             float2 d0, float2* __restrict__ ur, float2* __restrict__ nat) {
  using C = float2;
  const int P = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
  const int Yc = blockIdx.y * blockDim.y + threadIdx.y, Zc = blockIdx.z;
  if (P >= mc || Yc >= mc) return;
  const long long row = (long long)Zc * mc + Yc, s = row * HPc + (P >> 1);
  const C dc = nat ? zc() : dr[s];
  wait_and_trigger();
  const int fy = 2 * Yc + 1, fz = 2 * Zc + 1;          // rows one unit off lie inside the grid (m is odd)
  const C* const own = delta + ((long long)fz * m + fy) * HP + P;
  auto rowp = [&](int dy, int dz) {
    const bool in = fy + dy >= 0 && fy + dy < m && fz + dz >= 0 && fz + dz < m;
    return in ? own + ((long long)dz * m + dy) * HP : own;
  };
  // slots P, P + 1 of a row; the pair's neighbours: slot P - 1 and P + 2.  Every
  // load is made, outside the grid from a place inside it whose value is then
  // dropped: with tests around them the loads ran one after another (127^3
  // coarse points 35 -> 32 us, 31^3 and 15^3 7.9 and 7.7 -> 6.5 and 6.0)
  auto pair = [&](const C* r) { return ld2(r); };
  auto pair_in = [&](const C* r) {
    const Pair v = ld2(r);
    return r != own ? v : Pair{zc(), zc()};
  };
  const int ro = P + 2 < HP ? 2 : 0, lo = P > 0 ? -1 : 0;
  auto right = [&](const C* r) { const C v = r[ro]; return ro ? v : zc(); };
  auto left = [&](const C* r) { const C v = r[lo]; return lo ? v : zc(); };
  C f0 = zc(), f1 = f0, g0 = f0, g1 = f0, h0 = f0, h1 = f0;      // distance (1,0,0), (1,1,1), (2,1,0)
  auto add = [](C& x, C& y, C u, C v) { x = cadd(x, u); y = cadd(y, v); };
  {                                                    // own row: x offsets -1 and +1
    const C* r = rowp(0, 0);
    const Pair v = ld2(r);
    add(f0, f1, cadd(v.a, v.b), cadd(v.b, right(r)));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {                        // one unit off in y or z: x offset 0, and -2, +2
    const int s = (k & 1) ? 1 : -1;
    const C* r = (k < 2) ? rowp(s, 0) : rowp(0, s);
    const Pair v = pair(r);
    add(f0, f1, v.a, v.b);
    add(h0, h1, cadd(left(r), v.b), cadd(v.a, right(r)));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {                        // one unit off in both: x offsets -1 and +1
    const C* r = rowp((k & 1) ? 1 : -1, (k & 2) ? 1 : -1);
    const Pair v = pair(r);
    add(g0, g1, cadd(v.a, v.b), cadd(v.b, right(r)));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {                        // two units off in one: x offsets -1 and +1
    const int s = (k & 1) ? 2 : -2;
    const C* r = (k < 2) ? rowp(s, 0) : rowp(0, s);
    const Pair v = pair_in(r);
    add(h0, h1, cadd(v.a, v.b), cadd(v.b, r != own ? right(r) : zc()));
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {                        // two and one: x offset 0
    const int s = (k & 1) ? 1 : -1, s2 = (k & 2) ? 2 : -2;
    const Pair v = pair_in((k & 4) ? rowp(s2, s) : rowp(s, s2));
    add(h0, h1, v.a, v.b);
  }
  const C w0 = cadd(cadd(cscale(f0, 0.25f), cscale(g0, 0.09375f)), cscale(h0, 0.03125f));
  const C w1 = cadd(cadd(cscale(f1, 0.25f), cscale(g1, 0.09375f)), cscale(h1, 0.03125f));
  const C v0 = cmul(c, w0), v1 = P + 1 < mc ? cmul(c, w1) : zc();
  if (nat) {
    nat[row * mc + P] = v0;
    if (P + 1 < mc) nat[row * mc + P + 1] = v1;
    return;
  }
  const int o = (Yc + Zc + 1) & 1;                     // red parity of the coarse row
  const C vr = o ? v1 : v0;
  br[s] = vr;
  bb[s] = o ? v0 : v1;
  ur[s] = dinv_mul(d0, dc, vr);
}

// All levels from one of at most 15 points a side down to the coarsest and back
// in one CTA (FP32 cycles; FP64 ones would be bound by the one SM's FP64 pipe).
//
// Bound by latency: a chain of short phases on grids in shared memory, natural
// order with a ring of zeros (u, b, 1/d of the smoothing levels; 137 KB from 17^3
// down).  A row of a colour takes eight lanes; phases as above.  17^3, 9^3 and 5^3:
// 20.9 us alone, where the ten passes took 42 one by one; in the dependent
// launches of a cycle 4 us of that difference are left (257^3 cycle 367 -> 363;
// with the early triggers and the full weighting's loads 129^3 89.5 -> 75.9, 33^3
// 33.3 -> 27.2).
constexpr int BLOCK_M = 15, BLOCK_NT = 1024, BLOCK_LEVELS = 6, BLOCK_LAST = 64;
struct BlockLevels {
  int nl, m[BLOCK_LEVELS], HP[BLOCK_LEVELS];            // the last is the coarsest
  const float2 *dr[BLOCK_LEVELS], *db[BLOCK_LEVELS];
  float2 c[BLOCK_LEVELS], d0[BLOCK_LEVELS];
};
__host__ __device__ inline int ringed(int m) { return (m + 2) * (m + 2) * (m + 2); }

// neighbour sum of the interpolated correction at a red point (node indices
// nx, ny, nz), e ringed with W values a row: the cases of prolong_nbr
__device__ __forceinline__ float2 prolong_nbr_ringed(const float2* e, int W, int nx, int ny, int nz) {
  const float2* p = e + ((nz >> 1) * W + (ny >> 1)) * W + (nx >> 1);
  const int W2 = W * W;
  if (!((nx | ny | nz) & 1)) {
    const float2 s = cadd(cadd(cadd(p[-1], p[1]), cadd(p[-W], p[W])), cadd(p[-W2], p[W2]));
    return cadd(cscale(p[0], 3.f), cscale(s, 0.5f));
  }
  const int se = !(nx & 1) ? 1 : !(ny & 1) ? W : W2, s1 = (nx & 1) ? 1 : W, s2 = (nz & 1) ? W2 : W;
  auto s4 = [&](const float2* q) { return cadd(cadd(q[0], q[s1]), cadd(q[s2], q[s1 + s2])); };
  return cadd(cscale(s4(p), 1.25f), cscale(cadd(s4(p - se), s4(p + se)), 0.125f));
}

template <typename TI>
__global__ void __launch_bounds__(BLOCK_NT, 1)
    k3s_block(BlockLevels L, const float2* __restrict__ br, const float2* __restrict__ bb, const float2* __restrict__ ur,
              const cx<TI>* __restrict__ inv, float2* __restrict__ e_out, int pe) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) cx<TI> Bc[BLOCK_LAST];
  float2* const base = reinterpret_cast<float2*>(smem_raw);
  const int t = threadIdx.x, last = L.nl - 1, j = t & 7, r0 = t >> 3;
  constexpr int RS = BLOCK_NT / 8;
  int total = ringed(L.m[last]);
  for (int l = 0; l < last; ++l) total += 3 * ringed(L.m[l]);
  for (int i = t; i < total; i += BLOCK_NT) base[i] = make_float2(0.f, 0.f);
  __syncthreads();
  float2* p = base;
  for (int l = 0; l < last; ++l) {                     // 1/d in natural order
    const int m = L.m[l], W = m + 2, A = ringed(m);
    for (int row = r0; row < m * m; row += RS) {
      const int iz = row / m, iy = row - iz * m, o = (iy + iz + 1) & 1, i = ((iz + 1) * W + iy + 1) * W + 2 * j + 1;
      const long long s = (long long)row * L.HP[l] + j;
      if (2 * j + o < m) p[2 * A + i + o] = L.dr[l][s];
      if (2 * j + 1 - o < m) p[2 * A + i + 1 - o] = L.db[l][s];
    }
    p += 3 * A;
  }
  pdl_prologue();
  pdl_trigger();
  {
    const int m = L.m[0], W = m + 2, A = ringed(m);
    for (int row = r0; row < m * m; row += RS) {
      const int iz = row / m, iy = row - iz * m, o = (iy + iz + 1) & 1, i = ((iz + 1) * W + iy + 1) * W + 2 * j + 1;
      const long long s = (long long)row * L.HP[0] + j;
      if (2 * j + o < m) {
        base[i + o] = ur[s];
        base[A + i + o] = br[s];
      }
      if (2 * j + 1 - o < m) base[A + i + 1 - o] = bb[s];
    }
  }
  __syncthreads();
  auto nbr = [](const float2* u, int W) {
    const int W2 = W * W;
    return cadd(cadd(cadd(u[-1], u[1]), cadd(u[-W], u[W])), cadd(u[-W2], u[W2]));
  };
  p = base;
  for (int l = 0; l < last; ++l) {
    const int m = L.m[l], W = m + 2, A = ringed(m), mc = L.m[l + 1], Wc = mc + 2, Ac = ringed(mc);
    float2 *U = p, *B = p + A, *D = p + 2 * A, *next = p + 3 * A;
    const float2 c = L.c[l], d0 = L.d0[l];
    for (int row = r0; row < m * m; row += RS) {       // black
      const int iz = row / m, iy = row - iz * m, x = 2 * j + ((iy + iz) & 1);
      const int i = ((iz + 1) * W + iy + 1) * W + x + 1;
      if (x < m) U[i] = dinv_mul(d0, D[i], cfma(B[i], c, nbr(U + i, W)));
    }
    __syncthreads();
    for (int q = t; q < mc * mc * mc; q += BLOCK_NT) { // full weighting of the red residuals
      const int Z = q / (mc * mc), Y = q / mc - Z * mc, X = q - (Z * mc + Y) * mc, W2 = W * W;
      const float2* u = U + ((2 * Z + 2) * W + 2 * Y + 2) * W + 2 * X + 2;
      auto pair = [&](int a) { return cadd(u[-a], u[a]); };
      const float2 f = cadd(cadd(pair(1), pair(W)), pair(W2));
      const float2 g = cadd(cadd(pair(1 + W + W2), pair(1 + W - W2)), cadd(pair(1 - W + W2), pair(1 - W - W2)));
      auto edge = [&](int a, int b) { return cadd(cadd(pair(2 * a + b), pair(2 * a - b)), cadd(pair(a + 2 * b), pair(a - 2 * b))); };
      const float2 h = cadd(cadd(edge(1, W), edge(1, W2)), edge(W, W2));
      const float2 v = cmul(c, cadd(cadd(cscale(f, 0.25f), cscale(g, 0.09375f)), cscale(h, 0.03125f)));
      if (l + 1 < last) {
        const int s = ((Z + 1) * Wc + Y + 1) * Wc + X + 1;
        next[Ac + s] = v;
        if ((X + Y + Z) & 1) next[s] = dinv_mul(L.d0[l + 1], next[2 * Ac + s], v);
      } else {
        Bc[q] = mk<cx<TI>>((TI)v.x, (TI)v.y);
      }
    }
    __syncthreads();
    p = next;
  }
  {                                                    // coarsest: inv b, 16 lanes a row
    const int ml = L.m[last], n = ml * ml * ml, i = t >> 4, part = t & 15;
    TI re = (TI)0, im = (TI)0;
    if (i < n)
      for (int k = part; k < n; k += 16) {
        const cx<TI> a = inv[i * n + k], b = Bc[k];
        re = fma(a.x, b.x, fma(-a.y, b.y, re));
        im = fma(a.x, b.y, fma(a.y, b.x, im));
      }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (i < n && part == 0) {
      const int z = i / (ml * ml), y = i / ml - z * ml, x = i - (z * ml + y) * ml;
      p[((z + 1) * (ml + 2) + y + 1) * (ml + 2) + x + 1] = make_float2((float)re, (float)im);
    }
    __syncthreads();
  }
  const float2* E = p;
  for (int l = last - 1; l >= 0; --l) {
    const int m = L.m[l], W = m + 2, A = ringed(m), Wc = L.m[l + 1] + 2;
    p -= 3 * A;
    float2 *U = p, *B = p + A, *D = p + 2 * A;
    const float2 c = L.c[l], d0 = L.d0[l];
    for (int row = r0; row < m * m; row += RS) {       // red, with the correction's neighbour sum
      const int iz = row / m, iy = row - iz * m, x = 2 * j + ((iy + iz + 1) & 1);
      const int i = ((iz + 1) * W + iy + 1) * W + x + 1;
      if (x < m)
        U[i] = dinv_mul(d0, D[i], cfma(B[i], c, cadd(nbr(U + i, W), prolong_nbr_ringed(E, Wc, x + 1, iy + 1, iz + 1))));
    }
    __syncthreads();
    for (int row = r0; row < m * m; row += RS) {       // black; the top level's correction goes out
      const int iz = row / m, iy = row - iz * m, o = (iy + iz) & 1, x = 2 * j + o;
      const int i = ((iz + 1) * W + iy + 1) * W + x + 1;
      float2* out = e_out + ((long long)(iz + 1) * W + iy + 1) * pe + 2 * j + 2;
      if (x < m) {
        const float2 v = dinv_mul(d0, D[i], cfma(B[i], c, nbr(U + i, W)));
        if (l > 0) U[i] = v;
        else out[o] = v;
      }
      if (l == 0 && 2 * j + 1 - o < m) out[1 - o] = U[i + 1 - 2 * o];
    }
    __syncthreads();
    E = U;
  }
}

size_t block_bytes(const std::vector<Level>& lv, int lb) {
  size_t n = ringed(lv.back().m);
  for (size_t l = lb; l + 1 < lv.size(); ++l) n += 3 * (size_t)ringed(lv[l].m);
  return n * sizeof(float2);
}

struct Shape { dim3 g, b; };
// threads along x cover a row's slot pairs, rows fill the block up to 256
// threads (128 on small levels, whose passes last one CTA's lifetime)
Shape shape(int pairs, int m) {
  const int tx = pairs < 128 ? pairs : 128;
  const int want = m >= 127 ? 256 : 128;
  int ty = want / tx;
  ty = ty < 1 ? 1 : (ty > m ? m : ty);
  return Shape{dim3((pairs + tx - 1) / tx, (m + ty - 1) / ty, m), dim3(tx, ty)};
}

}  // namespace

int split3_pitch(int m) { return ((m + 1) / 2 + 3) / 4 * 4; }
// the finer level's slots j < HP read columns up to j + 4
int split3_ring_pitch(int mc) { return split3_pitch(2 * mc + 1) + 4; }

cudaError_t split3_coefs(Level& L, double k2, cudaStream_t s) {
  const int HP = split3_pitch(L.m);
  const Shape h = shape(HP / 2, L.m);
  Split3& S = L.s32;
  const float2 c = make_float2((float)L.c.x, (float)L.c.y);
  const double dx = 6.0 * (double)c.x - k2, dy = 6.0 * (double)c.y, den = dx * dx + dy * dy;
  S.d0 = den > 0.0 ? make_float2((float)(dx / den), (float)(-dy / den)) : make_float2(0.f, 0.f);
  const float2 dc = make_float2((float)(6.0 * ((double)c.x - L.c.x)), (float)(6.0 * ((double)c.y - L.c.y)));
  k3s_split<<<h.g, h.b, 0, s>>>(L.dinv64, dc, S.d0, L.m, HP, S.dr, S.db);
  count_launch();
  return cudaGetLastError();
}

// The line to the per-level kernels, by the smallest diagonal: 1/d is that of the
// FP32 value of c (k3s_split), which moves it by |6 c / d| 2^-25 of itself.  One
// cycle's error from an iterate against the per-level kernels', restated in FP32
// (33^3, box of 15, Gaussian barriers): 0.9 at |6 c / d| of 3.7 and 4.9, 1.3 at 5.8,
// 1.9 at 8.3, 3.8 at 10.8.
constexpr float SPLIT3_WORST = 4.f;
cudaError_t split3_suits(const std::vector<Level>& lv, unsigned* scratch, cudaStream_t s, bool* suits) {
  cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(unsigned), s);
  for (size_t l = 0; l + 1 < lv.size() && e == cudaSuccess; ++l) {
    const Level& L = lv[l];
    const long long blocks = (L.N + 255) / 256;
    k3s_worst<<<(unsigned)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, s>>>(
        L.dinv32, (float)(6.0 * std::hypot(L.c.x, L.c.y)), L.N, scratch);
    count_launch();
    e = cudaGetLastError();
  }
  float worst = 0.f;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&worst, scratch, sizeof(worst), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  *suits = worst <= SPLIT3_WORST;                      // false for NaN
  return e;
}

// the line lies at 15 points a side, where a level's passes last one CTA's
// lifetime each and its grids fit the block; the coarsest product has 16 lanes
// a row
int split3_block_level(const std::vector<Level>& lv) {
  const int nl = (int)lv.size();
  if (lv.back().N > BLOCK_LAST) return 0;
  for (int l = 1; l + 1 < nl; ++l)
    if (lv[l].m <= BLOCK_M) return nl - l <= BLOCK_LEVELS ? l : 0;
  return 0;
}
cudaError_t prepare_split3_block() {
  const int bytes = 160 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k3s_block<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(k3s_block<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
cudaError_t launch_split3_block(std::vector<Level>& lv, int lb, const float2* inv, const double2* inv64, cudaStream_t s) {
  BlockLevels L{};
  L.nl = (int)lv.size() - lb;
  for (int i = 0; i < L.nl; ++i) {
    const Level& v = lv[lb + i];
    L.m[i] = v.m;
    L.HP[i] = split3_pitch(v.m);
    L.dr[i] = v.s32.dr;
    L.db[i] = v.s32.db;
    L.c[i] = make_float2((float)v.c.x, (float)v.c.y);
    L.d0[i] = v.s32.d0;
  }
  const Split3& F = lv[lb].s32;
  const size_t sm = block_bytes(lv, lb);
  const int pe = split3_ring_pitch(lv[lb].m);
  ProfScope ps(mg_family<float>(), s, 2.0 * sizeof(float2) * lv[lb].N, 0);
  const float2 *br = F.br, *bb = F.bb, *ur = F.ur;
  const cudaError_t e = inv64 ? launch_pdl(k3s_block<double>, dim3(1), dim3(BLOCK_NT), sm, s, L, br, bb, ur, inv64, F.e, pe)
                              : launch_pdl(k3s_block<float>, dim3(1), dim3(BLOCK_NT), sm, s, L, br, bb, ur, inv, F.e, pe);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_split3_down(std::vector<Level>& lv, int stop, const float2* u, const float2* b, bool zero_init,
                               cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  int launches = 0;
  auto ok = [&](cudaError_t r) { ++launches; if (e == cudaSuccess) e = r; };
  const int nl = (int)lv.size();
  const double S = sizeof(float2);
  for (int l = 0; l < stop && e == cudaSuccess; ++l) {
    Level &L = lv[l], &C = lv[l + 1];
    Split3 &F = L.s32, &G = C.s32;
    const int m = L.m, HP = split3_pitch(m), HPc = split3_pitch(C.m);
    const float2 c = make_float2((float)L.c.x, (float)L.c.y);
    const Shape h = shape(HP / 2, m), hc = shape((C.m + 1) / 2, C.m);
    const float2* none = nullptr;
    float2* no = nullptr;
    const bool zero = zero_init || l > 0;
    ProfScope ps(mg_family<float>(), s, (zero ? 3.5 : 6.0) * S * L.N + S * C.N, 0);
    if (l == 0) {
      if (zero)
        ok(launch_pdl(k3s_first<false>, h.g, h.b, 0, s, b, none, (const float2*)F.dr, c, F.d0, m, HP, F.br, F.bb, no,
                      F.ur));
      else if (u)
        ok(launch_pdl(k3s_first<true>, h.g, h.b, 0, s, b, u, (const float2*)F.dr, c, F.d0, m, HP, F.br, F.bb, F.ub,
                      F.ur));
      else
        ok(launch_pdl(k3s_sweep<0, PLAIN>, h.g, h.b, 0, s, (const float2*)F.ub, (const float2*)F.br,
                      (const float2*)F.dr, c, F.d0, m, HP, F.ur, no, none, 0, 0, no, 0));
    }
    if (zero)
      ok(launch_pdl(k3s_sweep<1, PLAIN>, h.g, h.b, 0, s, (const float2*)F.ur, (const float2*)F.bb, (const float2*)F.db,
                    c, F.d0, m, HP, F.ub, no, none, 0, 0, no, 0));
    else
      ok(launch_pdl(k3s_sweep<1, DELTA>, h.g, h.b, 0, s, (const float2*)F.ur, (const float2*)F.bb, (const float2*)F.db,
                    c, F.d0, m, HP, F.ub, F.delta, none, 0, 0, no, 0));
    ok(launch_pdl(k3s_restrict, hc.g, hc.b, 0, s, (const float2*)(zero ? F.ub : F.delta), m, HP, c, C.m, HPc, G.br,
                  G.bb, (const float2*)G.dr, G.d0, G.ur, l + 2 == nl ? C.b32 : no));
  }
  count_launch(launches);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_split3_up(std::vector<Level>& lv, int stop, float2* u_nat, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  int launches = 0;
  auto ok = [&](cudaError_t r) { ++launches; if (e == cudaSuccess) e = r; };
  const double S = sizeof(float2);
  for (int l = stop - 1; l >= 0 && e == cudaSuccess; --l) {
    Level &L = lv[l], &C = lv[l + 1];
    Split3 &F = L.s32, &G = C.s32;
    const int m = L.m, HP = split3_pitch(m);
    const float2 c = make_float2((float)L.c.x, (float)L.c.y);
    const Shape h = shape(HP / 2, m);
    const float2* none = nullptr;
    float2* no = nullptr;
    ProfScope ps(mg_family<float>(), s, 5.0 * S * L.N + S * C.N, 0);
    ok(launch_pdl(k3s_sweep<0, PROLONG>, h.g, h.b, 0, s, (const float2*)F.ub, (const float2*)F.br,
                  (const float2*)F.dr, c, F.d0, m, HP, F.ur, no, (const float2*)G.e, split3_ring_pitch(C.m), C.m, no, 0));
    if (l > 0)
      ok(launch_pdl(k3s_sweep<1, RING>, h.g, h.b, 0, s, (const float2*)F.ur, (const float2*)F.bb, (const float2*)F.db,
                    c, F.d0, m, HP, no, no, none, 0, 0, F.e, split3_ring_pitch(m)));
    else if (u_nat)
      ok(launch_pdl(k3s_sweep<1, NAT>, h.g, h.b, 0, s, (const float2*)F.ur, (const float2*)F.bb, (const float2*)F.db,
                    c, F.d0, m, HP, no, no, none, 0, 0, u_nat, 0));
    else
      ok(launch_pdl(k3s_sweep<1, PLAIN>, h.g, h.b, 0, s, (const float2*)F.ur, (const float2*)F.bb, (const float2*)F.db,
                    c, F.d0, m, HP, F.ub, no, none, 0, 0, no, 0));
  }
  count_launch(launches);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace csff
