// Multigrid kernels on the rotated grid (Sec. 3.2 eq. (csg) with the Sec. 5.2
// stencil; Sec. 4 V-cycle components).  Templated on the real type (double for
// the plain and refinement path, float for the inner cycles of the mixed
// path) and on the dimension.
//
// Layout: m^d interior unknowns, x fastest, interleaved complex.  Boundary
// nodes are not stored (homogeneous Dirichlet).  Grid mapping: block (32, 8)
// over (x, y), blockIdx.z = z plane in 3D; (32, 2) on levels of few blocks,
// whose passes last one block's FP64 work (a warp instruction in 19 clocks an
// SM, in 65 from one warp).  Together with dependent launches, sweeps from zero,
// the norm of the residual without storing it and the operation counts below,
// the 65^2 FP64 map (17 Jacobi V(2,2) cycles) went from 1910 to 1180 us.
#include "csff_internal.h"
#include "df_bits.cuh"

namespace csff {
namespace {

constexpr int BX = 32, BY = 8, BY_SMALL = 2;

// wait for the predecessor; a grid of at most one block an SM lets its
// successor be set up at once
__device__ __forceinline__ void pdl_start() {
  pdl_prologue();
  if (gridDim.x * gridDim.y * gridDim.z <= 152u) pdl_trigger();
}

template <int D>
__device__ __forceinline__ bool thread_point(int m, int& ix, int& iy, int& iz, long long& idx) {
  ix = blockIdx.x * BX + threadIdx.x;
  iy = blockIdx.y * blockDim.y + threadIdx.y;
  iz = (D == 3) ? (int)blockIdx.z : 0;
  if (ix >= m || iy >= m) return false;
  idx = ((long long)iz * m + iy) * m + ix;
  return true;
}

// r_j = b_j - c (2d u_j - sum_nbr u) + q_j u_j ; neighbours outside the
// interior are zero, summed by pairs; the products as one chain of fused
// multiply-adds (FP64 runs at 1/61 of the FP32 rate: 20 operations a point in
// 3D, 28 with separate products, sums and a zero start).
template <typename T, int D>
__device__ __forceinline__ cx<T> residual_point(const cx<T>* __restrict__ u, cx<T> uj, cx<T> bj, cx<T> qj, cx<T> c,
                                                int m, int ix, int iy, int iz, long long idx) {
  using C = cx<T>;
  const C z = mk<C>((T)0, (T)0);
  C s = cadd(ix > 0 ? u[idx - 1] : z, ix < m - 1 ? u[idx + 1] : z);
  s = cadd(s, cadd(iy > 0 ? u[idx - m] : z, iy < m - 1 ? u[idx + m] : z));
  if (D == 3) {
    const long long p = (long long)m * m;
    s = cadd(s, cadd(iz > 0 ? u[idx - p] : z, iz < m - 1 ? u[idx + p] : z));
  }
  const T d = (T)(2 * D), tx = fma(d, uj.x, -s.x), ty = fma(d, uj.y, -s.y);
  return mk<C>(fma(-c.x, tx, fma(c.y, ty, fma(qj.x, uj.x, fma(-qj.y, uj.y, bj.x)))),
               fma(-c.x, ty, fma(-c.y, tx, fma(qj.x, uj.y, fma(qj.y, uj.x, bj.y)))));
}

template <typename T, int D>
__global__ void k_residual(const cx<T>* __restrict__ u, const cx<T>* __restrict__ b,
                           const cx<T>* __restrict__ q, cx<T> c, int m, cx<T>* __restrict__ r) {
  pdl_start();
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(m, ix, iy, iz, idx)) return;
  r[idx] = residual_point<T, D>(u, u[idx], b[idx], q[idx], c, m, ix, iy, iz, idx);
}

// u_out = u + omega d^{-1} (b - A u) = (1 - omega) u + omega d^{-1} (b + c
// sum_nbr u), since A u = d u - c sum_nbr u: 18 FP64 operations a point in 2D,
// 26 by way of the residual, and no read of q.  ZERO: from u = 0, omega d^{-1} b.
template <typename T, int D, bool ZERO>
__global__ void k_jacobi(const cx<T>* __restrict__ u, const cx<T>* __restrict__ b, const cx<T>* __restrict__ dinv,
                         cx<T> c, T omega, int m, cx<T>* __restrict__ u_out) {
  pdl_start();
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(m, ix, iy, iz, idx)) return;
  using C = cx<T>;
  const C di = dinv[idx];
  C v = b[idx];
  if constexpr (!ZERO) {
    const C z = mk<C>((T)0, (T)0);
    C s = cadd(ix > 0 ? u[idx - 1] : z, ix < m - 1 ? u[idx + 1] : z);
    s = cadd(s, cadd(iy > 0 ? u[idx - m] : z, iy < m - 1 ? u[idx + m] : z));
    if (D == 3) {
      const long long p = (long long)m * m;
      s = cadd(s, cadd(iz > 0 ? u[idx - p] : z, iz < m - 1 ? u[idx + p] : z));
    }
    v = mk<C>(fma(c.x, s.x, fma(-c.y, s.y, v.x)), fma(c.x, s.y, fma(c.y, s.x, v.y)));
  }
  C r = mk<C>(omega * fma(di.x, v.x, -di.y * v.y), omega * fma(di.x, v.y, di.y * v.x));
  if constexpr (!ZERO) {
    const C uj = u[idx];
    r = mk<C>(fma((T)1 - omega, uj.x, r.x), fma((T)1 - omega, uj.y, r.y));
  }
  u_out[idx] = r;
}

// One colour of red-black Gauss-Seidel, in place.  colour 0 (red) = even sum
// of node indices (interior index + 1 per axis).  One thread per point of the
// colour: x thread t of a row takes ix = 2 t + (colour + iy + iz + D) mod 2.
// With d = 2 D c - q the point's equation (A u)_j = d u_j - c sum_nbr u = b_j
// solved for u_j: u_j <- d^{-1} (b_j + c sum_nbr u), which reads neither q nor
// the point's old value.
template <typename T, int D>
__global__ void k_rbgs(cx<T>* u, const cx<T>* __restrict__ b, const cx<T>* __restrict__ dinv, cx<T> c, int m,
                       int colour) {
  pdl_start();
  const int iy = blockIdx.y * blockDim.y + threadIdx.y;
  const int iz = (D == 3) ? (int)blockIdx.z : 0;
  const int ix = 2 * (int)(blockIdx.x * BX + threadIdx.x) + ((colour + iy + iz + D) & 1);
  if (ix >= m || iy >= m) return;
  const long long idx = ((long long)iz * m + iy) * m + ix;
  using C = cx<T>;
  C s = mk<C>(0, 0);
  if (ix > 0) s = cadd(s, u[idx - 1]);
  if (ix < m - 1) s = cadd(s, u[idx + 1]);
  if (iy > 0) s = cadd(s, u[idx - m]);
  if (iy < m - 1) s = cadd(s, u[idx + m]);
  if (D == 3) {
    const long long p = (long long)m * m;
    if (iz > 0) s = cadd(s, u[idx - p]);
    if (iz < m - 1) s = cadd(s, u[idx + p]);
  }
  u[idx] = cmul(dinv[idx], cadd(b[idx], cmul(c, s)));
}

// Full weighting: coarse interior P <- sum over offsets o in {-1,0,1}^d of
// prod(1/2 if o = 0 else 1/4) * r_f[2P + 1 + o], axis by axis as
// ((left + right)/2 + middle)/2: in 3D 54 operations a point, 144 with a
// product and a sum for every offset.
template <typename C, typename T> __device__ __forceinline__ C weigh(C l, C mid, C r) {
  const T h = (T)0.5;
  return mk<C>(fma(l.x + r.x, h, mid.x), fma(l.y + r.y, h, mid.y));
}
template <typename T, int D, typename R>
__device__ __forceinline__ cx<T> full_weight(R r) {
  using C = cx<T>;
  C plane[3];
#pragma unroll
  for (int oz = (D == 3 ? -1 : 0); oz <= (D == 3 ? 1 : 0); ++oz) {
    C row[3];
#pragma unroll
    for (int oy = -1; oy <= 1; ++oy) row[oy + 1] = weigh<C, T>(r(-1, oy, oz), r(0, oy, oz), r(1, oy, oz));
    plane[oz + 1] = weigh<C, T>(row[0], row[1], row[2]);
  }
  if (D == 2) return cscale(plane[1], (T)0.25);
  return cscale(weigh<C, T>(plane[0], plane[1], plane[2]), (T)0.125);
}

template <typename T, int D>
__global__ void k_restrict(const cx<T>* __restrict__ rf, int mf, cx<T>* __restrict__ bc, int mc) {
  pdl_start();
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(mc, ix, iy, iz, idx)) return;
  const long long f = ((long long)(D == 3 ? 2 * iz + 1 : 0) * mf + 2 * iy + 1) * mf + 2 * ix + 1;
  const long long p = (long long)mf * mf;
  bc[idx] = full_weight<T, D>([&](int ox, int oy, int oz) { return rf[f + ox + (long long)oy * mf + oz * p]; });
}

// u_f += P e by coarse cells: cell (Nx, Ny, Nz), N in [0, mc] per axis, spans
// coarse nodes N and N + 1 (node 0 and mc + 1 on the boundary, value zero)
// and holds the fine nodes 2N + 1 (the midpoint: weight 1/2 on each end) and
// 2N + 2 (coarse node N + 1: weight 1), interior indices 2N and 2N + 1 (the
// latter only for N < mc).  The bilinear/trilinear weights are products of
// these per axis, applied axis by axis; one thread per cell, its two x points
// adjacent in memory.
template <typename T, int D>
__global__ void k_prolong_cells(const cx<T>* __restrict__ ec, int mc, cx<T>* __restrict__ uf, int mf) {
  using C = cx<T>;
  pdl_start();
  const int Nx = blockIdx.x * BX + threadIdx.x, Ny = blockIdx.y * blockDim.y + threadIdx.y;
  const int Nz = (D == 3) ? (int)blockIdx.z : 0;
  if (Nx > mc || Ny > mc) return;
  const T h = (T)0.5;
  // coarse values at the cell's corners: node K -> e[K - 1] inside [1, mc]
  auto ev = [&](int kx, int ky, int kz) -> C {
    const int X = Nx + kx, Y = Ny + ky, Z = Nz + kz;
    if (X < 1 || X > mc || Y < 1 || Y > mc || (D == 3 && (Z < 1 || Z > mc))) return mk<C>(0, 0);
    return ec[((long long)(D == 3 ? Z - 1 : 0) * mc + (Y - 1)) * mc + (X - 1)];
  };
  // along x for each (y, z) corner: mid and coincident values
  C xm[2][2], xc[2][2];
#pragma unroll
  for (int kz = 0; kz < (D == 3 ? 2 : 1); ++kz)
#pragma unroll
    for (int ky = 0; ky < 2; ++ky) {
      const C a = ev(0, ky, kz), b = ev(1, ky, kz);
      xm[kz][ky] = cscale(cadd(a, b), h);
      xc[kz][ky] = b;
    }
  const bool x1 = Nx < mc, y1 = Ny < mc, z1 = (D == 3) ? Nz < mc : false;
  const long long f0 = ((long long)(D == 3 ? 2 * Nz : 0) * mf + 2 * Ny) * mf + 2 * Nx;
  // the cell's fine values first, all in flight together (a load after a
  // store through the same pointer would wait for it)
  C u0[2][2], u1[2][2];
#pragma unroll
  for (int sz = 0; sz < (D == 3 ? 2 : 1); ++sz)
#pragma unroll
    for (int sy = 0; sy < 2; ++sy) {
      const bool in = (sz == 0 || z1) && (sy == 0 || y1);
      const long long f = f0 + ((long long)sz * mf + sy) * mf;
      u0[sz][sy] = in ? uf[f] : mk<C>(0, 0);
      u1[sz][sy] = (in && x1) ? uf[f + 1] : mk<C>(0, 0);
    }
#pragma unroll
  for (int sz = 0; sz < (D == 3 ? 2 : 1); ++sz) {        // fine z: 0 mid, 1 coincident
    if (sz == 1 && !z1) continue;
#pragma unroll
    for (int sy = 0; sy < 2; ++sy) {                      // fine y: 0 mid, 1 coincident
      if (sy == 1 && !y1) continue;
      // along z, then y
      C vm, vc;
      if (D == 3) {
        C ym_m = sz ? xm[1][0] : cscale(cadd(xm[0][0], xm[1][0]), h);
        C ym_c = sz ? xc[1][0] : cscale(cadd(xc[0][0], xc[1][0]), h);
        C yc_m = sz ? xm[1][1] : cscale(cadd(xm[0][1], xm[1][1]), h);
        C yc_c = sz ? xc[1][1] : cscale(cadd(xc[0][1], xc[1][1]), h);
        vm = sy ? yc_m : cscale(cadd(ym_m, yc_m), h);
        vc = sy ? yc_c : cscale(cadd(ym_c, yc_c), h);
      } else {
        vm = sy ? xm[0][1] : cscale(cadd(xm[0][0], xm[0][1]), h);
        vc = sy ? xc[0][1] : cscale(cadd(xc[0][0], xc[0][1]), h);
      }
      const long long f = f0 + ((long long)sz * mf + sy) * mf;
      uf[f] = cadd(u0[sz][sy], vm);
      if (x1) uf[f + 1] = cadd(u1[sz][sy], vc);
    }
  }
}

// Coarsest level: u = inv b, the inverse from FP64 Gauss-Jordan, in TI
// arithmetic, rounded once to T.  LPR lanes a row (4, or 32 for large N), chains
// of fused multiply-adds joined by shuffles: FP64 work is scarce on this part.  Above
// 32 unknowns four lanes keep NA = 8 chains each where the product is in the vectors'
// own precision (121 unknowns: 1.2 units of rounding off, 2.1 with one chain, 1.5
// with 32 lanes).
template <typename T, typename TI, int LPR, int NA>
__global__ void __launch_bounds__(256) k_coarse_solve(const cx<TI>* __restrict__ inv, int N,
                                                      const cx<T>* __restrict__ b, cx<T>* __restrict__ u, int ring_m,
                                                      int ring_pitch) {
  pdl_start();
  const int t = blockIdx.x * 256 + threadIdx.x, i = t / LPR, part = t % LPR;
  TI rc[NA], ic[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) rc[a] = ic[a] = (TI)0;
  if (i < N) {
    const cx<TI>* row = inv + (long long)i * N;
#pragma unroll(NA == 1 ? 8 : 1)
    for (int j0 = part; j0 < N; j0 += LPR * NA) {
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        const int j = j0 + LPR * c;
        if (j >= N) continue;
        const cx<TI> a = row[j];
        const cx<T> bj = b[j];
        const TI bx = (TI)bj.x, by = (TI)bj.y;
        rc[c] = fma(a.x, bx, fma(-a.y, by, rc[c]));
        ic[c] = fma(a.x, by, fma(a.y, bx, ic[c]));
      }
    }
  }
#pragma unroll
  for (int h = NA / 2; h > 0; h >>= 1)
#pragma unroll
    for (int c = 0; c < h; ++c) {
      rc[c] += rc[c + h];
      ic[c] += ic[c + h];
    }
  TI re = rc[0], im = ic[0];
#pragma unroll
  for (int o = 1; o < LPR; o <<= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if (i < N && part == 0) {
    long long o = i;
    if (ring_m > 0) {
      const int r = i / ring_m, y = r % ring_m, z = r / ring_m;
      o = ((long long)(z + 1) * (ring_m + 2) + y + 1) * ring_pitch + (i - r * ring_m) + 2;
    }
    u[o] = mk<cx<T>>((T)re, (T)im);
  }
}

// ---- reductions ------------------------------------------------------------
// Block-wide reduction; the result is valid in thread 0.
template <typename V, typename Op>
__device__ __forceinline__ V block_reduce(V v, Op op, V* sh, V identity) {
  for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  int nw = blockDim.x >> 5;
  if (w == 0) {
    v = (l < nw) ? sh[l] : identity;
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

struct AddOp { __device__ double operator()(double a, double b) const { return a + b; } };
struct MaxIOp { __device__ int operator()(int a, int b) const { return a > b ? a : b; } };

constexpr int RED_THREADS = 256;

template <typename T>
__global__ void k_norm_partial(const cx<T>* __restrict__ v, long long N, double scale,
                               double* __restrict__ partial) {
  pdl_prologue();
  __shared__ double sh[32];
  double acc = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x) {
    double a = (double)v[i].x, b = (double)v[i].y;
    if (scale != 1.0) {
      a *= scale;
      b *= scale;
    }
    acc = fma(a, a, fma(b, b, acc));
  }
  acc = block_reduce(acc, AddOp(), sh, 0.0);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// the same for a solve's right-hand side, with its rounding r32 = 2^-s v to FP32,
// the first right-hand side of the cycles from zero
__global__ void k_first_residual(const double2* __restrict__ v, int N, double scale, int s, float2* __restrict__ r32,
                                 double* __restrict__ partial) {
  pdl_prologue();
  __shared__ double sh[32];
  double acc = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    double2 x = v[i];
    r32[i] = make_float2(bits::narrow(x.x, s), bits::narrow(x.y, s));
    if (scale != 1.0) x = cscale(x, scale);
    acc = fma(x.x, x.x, fma(x.y, x.y, acc));
  }
  acc = block_reduce(acc, AddOp(), sh, 0.0);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

__global__ void k_norm_finish(const double* __restrict__ partial, int nblk, double inv_scale,
                              double* __restrict__ out) {
  pdl_prologue();
  __shared__ double sh[32];
  double acc = 0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += partial[i];
  acc = block_reduce(acc, AddOp(), sh, 0.0);
  if (threadIdx.x == 0) *out = sqrt(acc) * inv_scale;
}

// per-block sums of |2^-e (b - A u)|^2 in FP64, the residual not stored; a
// block walks grid rows
template <int D>
__global__ void __launch_bounds__(RED_THREADS) k_resid_norm(const double2* __restrict__ u,
                                                            const double2* __restrict__ b,
                                                            const double2* __restrict__ q, double2 c, int m, int tx,
                                                            double scale, double* __restrict__ partial) {
  pdl_start();
  __shared__ double sh[32];
  const int nrows = (D == 3) ? m * m : m, ty = RED_THREADS / tx, y = threadIdx.x / tx;
  double acc = 0;
  for (int row = blockIdx.x * ty + y; row < nrows; row += gridDim.x * ty) {
    const int iz = (D == 3) ? row / m : 0, iy = (D == 3) ? row - iz * m : row;
    for (int ix = threadIdx.x - y * tx; ix < m; ix += tx) {
      const long long i = (long long)row * m + ix;
      const double2 r = residual_point<double, D>(u, u[i], b[i], q[i], c, m, ix, iy, iz, i);
      const double rx = r.x * scale, ry = r.y * scale;
      acc = fma(rx, rx, fma(ry, ry, acc));
    }
  }
  acc = block_reduce(acc, AddOp(), sh, 0.0);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// frexp's exponent of max(|re|, |im|) from the IEEE fields: -2000 for zero, 4000
// when a component is not finite
__device__ __forceinline__ int max_exp(double2 x) {
  const int Ex = bits::exp_field(x.x), Ey = bits::exp_field(x.y);
  if (Ex == 0x7ff || Ey == 0x7ff) return 4000;
  const bool nzx = ((unsigned long long)__double_as_longlong(x.x) & bits::ABS_MASK) != 0;
  const bool nzy = ((unsigned long long)__double_as_longlong(x.y) & bits::ABS_MASK) != 0;
  return max(nzx ? bits::frexp_exp(x.x) : -2000, nzy ? bits::frexp_exp(x.y) : -2000);
}

__global__ void k_max_exp(const double2* __restrict__ v, long long N, int* __restrict__ out) {
  __shared__ int sh[32];
  int mx = -2000;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x) {
    mx = max(mx, max_exp(v[i]));
  }
  mx = block_reduce(mx, MaxIOp(), sh, -2000);
  if (threadIdx.x == 0) atomicMax(out, mx);
}

__global__ void k_set_int(int* p, int v) { *p = v; }

// ---- coefficients and right-hand side ----------------------------------------
template <int D>
__device__ __forceinline__ double2 chi_point(const double2* const* tabs, int n_gauss, int m, int ix,
                                             int iy, int iz) {
  double2 chi = make_double2(0, 0);
  for (int g = 0; g < n_gauss; ++g) {
    const double2* t = tabs[g];
    double2 v = cmul(t[ix], t[m + iy]);
    if (D == 3) v = cmul(v, t[2 * m + iz]);
    chi = cadd(chi, v);
  }
  return chi;
}

struct TabPtrs { const double2* p[8]; };

template <int D>
__global__ void k_coefs(TabPtrs tabs, int n_gauss, int m, double k2, double2 c, double2* q64,
                        double2* dinv64, float2* q32, float2* dinv32) {
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(m, ix, iy, iz, idx)) return;
  double2 chi = chi_point<D>(tabs.p, n_gauss, m, ix, iy, iz);
  double2 q = make_double2(k2 * (1.0 + chi.x), k2 * chi.y);
  double2 dg = make_double2(2 * D * c.x - q.x, 2 * D * c.y - q.y);
  double den = dg.x * dg.x + dg.y * dg.y;
  double2 di = make_double2(dg.x / den, -dg.y / den);
  q64[idx] = q;
  dinv64[idx] = di;
  q32[idx] = make_float2((float)q.x, (float)q.y);
  dinv32[idx] = make_float2((float)di.x, (float)di.y);
}

// coarse q at the coarse nodes, which are fine nodes 2 I + 1 per axis
template <int D>
__global__ void k_inject_q(const double2* __restrict__ qf, int mf, double2* __restrict__ qc, int mc) {
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(mc, ix, iy, iz, idx)) return;
  const long long f = ((long long)(D == 3 ? 2 * iz + 1 : 0) * mf + 2 * iy + 1) * mf + 2 * ix + 1;
  qc[idx] = qf[f];
}

// 1/d = 1/(2d c - q) and the FP32 copies from a level's q64
template <int D>
__global__ void k_coefs_from_q(const double2* __restrict__ q64, int m, double2 c, double2* dinv64, float2* q32,
                               float2* dinv32) {
  int ix, iy, iz; long long idx;
  if (!thread_point<D>(m, ix, iy, iz, idx)) return;
  const double2 q = q64[idx];
  const double2 dg = make_double2(2 * D * c.x - q.x, 2 * D * c.y - q.y);
  const double den = dg.x * dg.x + dg.y * dg.y;
  const double2 di = make_double2(dg.x / den, -dg.y / den);
  dinv64[idx] = di;
  q32[idx] = make_float2((float)q.x, (float)q.y);
  dinv32[idx] = make_float2((float)di.x, (float)di.y);
}

// The incident wave's tables, on the device: the 2 x 1023 exponentials of a
// 1025^2 map took the host longer than a V-cycle takes the GPU, before the first
// kernel of a solve and again of a far field.
__global__ void k_incident(double2* __restrict__ tab, int m, double lo, double h, double k, double eta0, double eta1,
                           double eta2, double cg, double sg) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
  if (i >= m) return;
  const double eta = c == 0 ? eta0 : c == 1 ? eta1 : eta2;
  const double x = __dadd_rn(lo, __dmul_rn((double)(i + 1), h));
  tab[(long long)c * m + i] = incident(__dmul_rn(__dmul_rn(k, eta), x), cg, sg);
}

template <int D>
__global__ void k_rhs(TabPtrs tabs, int n_gauss, const double2* __restrict__ uinc, int m, double k2,
                      double2* __restrict__ b, int* __restrict__ emax) {
  // chi u_in = sum_g prod_c (E_{g,c} U_c): each axis' Gaussian factor is paired
  // with its incident-wave factor first, so no partial product leaves the
  // FP64 range when chi u_in itself does not.  The pairs for the block's 32
  // columns and 8 rows are formed once per block (in 3D for its 8 planes), the row
  // factors k^2 (E_y U_y)(E_z U_z) once per plane: a node costs one complex
  // product per Gaussian (this pass runs on the FP64 pipe, 1/61 of the FP32 rate
  // here).  257^3 with the exponent 238 us; one plane a block 290, or 213 and a pass of
  // its own for the exponent, 70.
  __shared__ double2 px[8][BX], py[8][BY], pyz[2][8][BY];
  __shared__ int wmax;
  const int t = threadIdx.y * BX + threadIdx.x;
  if (t == 0) wmax = -2000;
  for (int i = t; i < n_gauss * (BX + BY); i += BX * BY) {
    const int g = i / (BX + BY), r = i % (BX + BY);
    const double2* E = tabs.p[g];
    if (r < BX) {
      const int x = blockIdx.x * BX + r;
      px[g][r] = x < m ? cmul(E[x], uinc[x]) : make_double2(0, 0);
    } else {
      const int y = blockIdx.y * BY + (r - BX);
      py[g][r - BX] = y < m ? cmul(E[m + y], uinc[m + y]) : make_double2(0, 0);
    }
  }
  __syncthreads();
  const int ix = blockIdx.x * BX + threadIdx.x, iy = blockIdx.y * BY + threadIdx.y;
  const int z0 = (D == 3) ? 8 * (int)blockIdx.z : 0, z1 = (D == 3) ? min(z0 + 8, m) : 1;
  int e = -2000;
  for (int iz = z0; iz < z1; ++iz) {
    const int buf = iz & 1;              // the other one may still be read
    for (int i = t; i < n_gauss * BY; i += BX * BY) {
      const int g = i / BY, r = i % BY;
      const double2 v = (D == 3) ? cmul(py[g][r], cmul(tabs.p[g][2 * m + iz], uinc[2 * m + iz])) : py[g][r];
      pyz[buf][g][r] = cscale(v, k2);
    }
    __syncthreads();
    if (ix >= m || iy >= m) continue;
    double2 acc = n_gauss > 0 ? cmul(px[0][threadIdx.x], pyz[buf][0][threadIdx.y]) : make_double2(0, 0);
    for (int g = 1; g < n_gauss; ++g) acc = cadd(acc, cmul(px[g][threadIdx.x], pyz[buf][g][threadIdx.y]));
    b[((long long)iz * m + iy) * m + ix] = acc;
    // a solve's exponent of max |b|, while the values are at hand
    if (emax) e = max(e, max_exp(acc));
  }
  if (!emax) return;
  e = __reduce_max_sync(0xffffffffu, e);
  if ((t & 31) == 0) atomicMax(&wmax, e);
  __syncthreads();
  if (t == 0 && wmax > *(volatile int*)emax) atomicMax(emax, wmax);
}

// ---- FP64 refinement of the mixed solve (option refine_fp64) -------------------
// One pass of the FP64 refinement step (option refine_fp64): the residual
// r = b - A u in FP64 as a chain of fused multiply-adds,
//   r = b - c (2d u - sum_nbr u) + q u,
// its rounding r32 = 2^-s r to FP32 (the right-hand side of the next FP32
// cycles: an exact FP64 scaling and one conversion), and per-block sums of
// |r32|^2 for the norm (within 2^-24 relative of ||2^-s r||, far inside what
// the stopping test resolves).  s is fixed for a solve (the exponent of
// max |b|), so the FP32 values stay below 1 in magnitude.  The kernel is
// bound by the FP64 pipe (a warp instruction in 19 clocks an SM), so the scaling
// and the rounding to FP32 work on the bit fields and each CTA walks grid rows
// (no index division per point).  20 FP64 operations a point in 3D, 24 with
// the scaling and the conversion in FP64: 257^3 750 -> 631 us, 1025^2 46 -> 38 us.
template <int D>
__global__ void k_refine_residual(const double2* __restrict__ u, const double2* __restrict__ b,
                                  const double2* __restrict__ q, double2 c, int m, int s_exp,
                                  float2* __restrict__ r32, double* __restrict__ partial) {
  pdl_prologue();
  __shared__ double sh[32];
  float acc = 0.f;
  const int nrows = (D == 3) ? m * m : m;
  const int ix = blockIdx.x * blockDim.x + threadIdx.x;
  const double2 z = make_double2(0.0, 0.0);
  if (ix < m) {
    for (int row = blockIdx.y; row < nrows; row += gridDim.y) {
      const int iz = (D == 3) ? row / m : 0;
      const int iy = (D == 3) ? row - iz * m : row;
      const long long i = (long long)row * m + ix;
      const double2 uj = u[i];
      const double2 xl = ix > 0 ? u[i - 1] : z, xr = ix < m - 1 ? u[i + 1] : z;
      const double2 yl = iy > 0 ? u[i - m] : z, yr = iy < m - 1 ? u[i + m] : z;
      double sx = (xl.x + xr.x) + (yl.x + yr.x), sy = (xl.y + xr.y) + (yl.y + yr.y);
      if (D == 3) {
        const long long mm = (long long)m * m;
        const double2 zl = iz > 0 ? u[i - mm] : z, zr = iz < m - 1 ? u[i + mm] : z;
        sx += zl.x + zr.x;
        sy += zl.y + zr.y;
      }
      const double tx = fma((double)(2 * D), uj.x, -sx), ty = fma((double)(2 * D), uj.y, -sy);
      const double2 bj = b[i], qj = q[i];
      const double rx = fma(-c.x, tx, fma(c.y, ty, fma(qj.x, uj.x, fma(-qj.y, uj.y, bj.x))));
      const double ry = fma(-c.x, ty, fma(-c.y, tx, fma(qj.x, uj.y, fma(qj.y, uj.x, bj.y))));
      const float fx = bits::narrow(rx, s_exp), fy = bits::narrow(ry, s_exp);
      r32[i] = make_float2(fx, fy);
      acc = __fmaf_rn(fx, fx, __fmaf_rn(fy, fy, acc));
    }
  }
  const double tot = block_reduce((double)acc, AddOp(), sh, 0.0);
  if (threadIdx.x == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = tot;
}

// u += 2^s e.  NEAR: the FP32 correction is widened on the bit fields, which
// leaves two FP64 additions a point and the pass bound by memory (257^3: 128 ->
// 94 us, 665 MB); else (scales near the ends of the FP64 range) by conversions
// and multiply-adds.
template <bool NEAR>
__global__ void k_update64_fixed(double2* __restrict__ u, const float2* __restrict__ e, int N, int s, double p2) {
  pdl_prologue();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const float2 c = e[i];
    double2 v = u[i];
    if constexpr (NEAR) {
      v.x += bits::widen_near(c.x, s);
      v.y += bits::widen_near(c.y, s);
    } else {
      v.x = fma((double)c.x, p2, v.x);
      v.y = fma((double)c.y, p2, v.y);
    }
    u[i] = v;
  }
}

template <typename T>
__global__ void k_zero(cx<T>* v, long long N) {
  pdl_start();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x)
    v[i] = mk<cx<T>>(0, 0);
}

inline dim3 grid_of(int dim, int m) {
  return dim3((m + BX - 1) / BX, (m + BY - 1) / BY, dim == 3 ? m : 1);
}
// grid and block for passes over wx x wy (x wz) threads: small blocks where the
// large ones would leave SMs without one
struct Shape { dim3 g, b; };
inline Shape shape_of(int wx, int wy, int wz) {
  const long long big = (long long)((wx + BX - 1) / BX) * ((wy + BY - 1) / BY) * wz;
  const int by = big < 152 ? BY_SMALL : BY;
  return Shape{dim3((wx + BX - 1) / BX, (wy + by - 1) / by, wz), dim3(BX, by)};
}
inline Shape shape_of(int dim, int m) { return shape_of(m, m, dim == 3 ? m : 1); }
inline int flat_blocks(long long N) {
  long long b = (N + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T> static const cx<T>* qtab(const Level& L);
template <> const double2* qtab<double>(const Level& L) { return L.q64; }
template <> const float2* qtab<float>(const Level& L) { return L.q32; }
template <typename T> static const cx<T>* dtab(const Level& L);
template <> const double2* dtab<double>(const Level& L) { return L.dinv64; }
template <> const float2* dtab<float>(const Level& L) { return L.dinv32; }

template <typename T>
cudaError_t launch_residual(int dim, const Level& L, const cx<T>* u, const cx<T>* b, cx<T>* r,
                            cudaStream_t s) {
  const Shape h = shape_of(dim, L.m);
  cx<T> c = mk<cx<T>>((T)L.c.x, (T)L.c.y);
  ProfScope ps(mg_family<T>(), s, 3.0 * sizeof(cx<T>) * L.N, 0);
  cudaError_t e = (dim == 2) ? launch_pdl(k_residual<T, 2>, h.g, h.b, 0, s, u, b, qtab<T>(L), c, L.m, r)
                             : launch_pdl(k_residual<T, 3>, h.g, h.b, 0, s, u, b, qtab<T>(L), c, L.m, r);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_jacobi(int dim, const Level& L, double omega, const cx<T>* u, const cx<T>* b,
                          cx<T>* u_out, cudaStream_t s) {
  const Shape h = shape_of(dim, L.m);
  cx<T> c = mk<cx<T>>((T)L.c.x, (T)L.c.y);
  const cx<T>* d = dtab<T>(L);
  ProfScope ps(mg_family<T>(), s, (u ? 3.0 : 2.0) * sizeof(cx<T>) * L.N, 0);
  cudaError_t e;
  if (u)
    e = dim == 2 ? launch_pdl(k_jacobi<T, 2, false>, h.g, h.b, 0, s, u, b, d, c, (T)omega, L.m, u_out)
                 : launch_pdl(k_jacobi<T, 3, false>, h.g, h.b, 0, s, u, b, d, c, (T)omega, L.m, u_out);
  else
    e = dim == 2 ? launch_pdl(k_jacobi<T, 2, true>, h.g, h.b, 0, s, u, b, d, c, (T)omega, L.m, u_out)
                 : launch_pdl(k_jacobi<T, 3, true>, h.g, h.b, 0, s, u, b, d, c, (T)omega, L.m, u_out);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_rbgs(int dim, const Level& L, cx<T>* u, const cx<T>* b, cudaStream_t s) {
  // one thread per point of a colour along x
  const Shape h = shape_of((L.m + 1) / 2, L.m, dim == 3 ? L.m : 1);
  cx<T> c = mk<cx<T>>((T)L.c.x, (T)L.c.y);
  ProfScope ps(mg_family<T>(), s, 3.0 * sizeof(cx<T>) * L.N, 0);
  cudaError_t e = cudaSuccess;
  for (int colour = 0; colour < 2 && e == cudaSuccess; ++colour)
    e = dim == 2 ? launch_pdl(k_rbgs<T, 2>, h.g, h.b, 0, s, u, b, dtab<T>(L), c, L.m, colour)
                 : launch_pdl(k_rbgs<T, 3>, h.g, h.b, 0, s, u, b, dtab<T>(L), c, L.m, colour);
  count_launch(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_restrict(int dim, const Level& F, const Level& C, const cx<T>* r, cx<T>* bc,
                            cudaStream_t s) {
  const Shape h = shape_of(dim, C.m);
  ProfScope ps(mg_family<T>(), s, (double)sizeof(cx<T>) * (F.N + C.N), 0);
  cudaError_t e = dim == 2 ? launch_pdl(k_restrict<T, 2>, h.g, h.b, 0, s, r, F.m, bc, C.m)
                           : launch_pdl(k_restrict<T, 3>, h.g, h.b, 0, s, r, F.m, bc, C.m);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_prolong_add(int dim, const Level& F, const Level& C, const cx<T>* ec, cx<T>* u,
                               cudaStream_t s) {
  ProfScope ps(mg_family<T>(), s, (double)sizeof(cx<T>) * (2.0 * F.N + C.N), 0);
  const Shape h = shape_of(C.m + 1, C.m + 1, dim == 3 ? C.m + 1 : 1);            // coarse cells
  cudaError_t e = dim == 2 ? launch_pdl(k_prolong_cells<T, 2>, h.g, h.b, 0, s, ec, C.m, u, F.m)
                           : launch_pdl(k_prolong_cells<T, 3>, h.g, h.b, 0, s, ec, C.m, u, F.m);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T, typename TI>
static cudaError_t coarse_solve(const cx<TI>* inv, int N, const cx<T>* b, cx<T>* u, cudaStream_t s, int rm, int rp) {
  ProfScope ps(mg_family<T>(), s, sizeof(cx<T>) * 2.0 * N + sizeof(cx<TI>) * (double)N * N, 8.0 * N * N);
  constexpr int NA = sizeof(T) == sizeof(TI) ? 8 : 1;
  const int lanes = N <= 128 ? 4 : 32;
  cudaError_t e = launch_pdl(N <= 32 ? k_coarse_solve<T, TI, 4, 1> : N <= 128 ? k_coarse_solve<T, TI, 4, NA>
                                                                            : k_coarse_solve<T, TI, 32, 1>,
                             dim3((lanes * N + 255) / 256), dim3(256), 0, s, inv, N, b, u, rm, rp);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_coarse_solve(const cx<T>* inv, int N, const cx<T>* b, cx<T>* u, cudaStream_t s, int ring_m,
                                int ring_pitch) {
  return coarse_solve<T, T>(inv, N, b, u, s, ring_m, ring_pitch);
}

cudaError_t launch_coarse_solve_f64(const double2* inv, int N, const float2* b, float2* u, cudaStream_t s, int ring_m,
                                    int ring_pitch) {
  return coarse_solve<float, double>(inv, N, b, u, s, ring_m, ring_pitch);
}

cudaError_t launch_resid_norm(int dim, const Level& L, const double2* u, const double2* b, int exp_scale,
                              double* partial, int nblk, double* out, cudaStream_t s) {
  int tx = 32;
  while (tx < L.m && tx < RED_THREADS) tx *= 2;
  const long long rows = dim == 3 ? (long long)L.m * L.m : L.m, need = (rows + RED_THREADS / tx - 1) / (RED_THREADS / tx);
  const int nb = (int)(need < nblk ? need : nblk);
  const double scale = ldexp(1.0, -exp_scale);
  ProfScope ps(PF_MG64, s, 3.0 * sizeof(double2) * L.N, 0);
  cudaError_t e = dim == 2 ? launch_pdl(k_resid_norm<2>, dim3(nb), dim3(RED_THREADS), 0, s, u, b, (const double2*)L.q64,
                                        L.c, L.m, tx, scale, partial)
                           : launch_pdl(k_resid_norm<3>, dim3(nb), dim3(RED_THREADS), 0, s, u, b, (const double2*)L.q64,
                                        L.c, L.m, tx, scale, partial);
  if (e == cudaSuccess)
    e = launch_pdl(k_norm_finish, dim3(1), dim3(RED_THREADS), 0, s, (const double*)partial, nb, ldexp(1.0, exp_scale),
                   out);
  count_launch(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_norm2(const cx<T>* v, long long N, int exp_scale, double* partial, int nblk,
                         double* out, cudaStream_t s) {
  long long need = (N + RED_THREADS - 1) / RED_THREADS;
  int nb = (int)(need < nblk ? (need < 1 ? 1 : need) : nblk);
  if (abs(exp_scale) <= 400) exp_scale = 0;      // squares stay inside the FP64 range
  ProfScope ps(mg_family<T>(), s, (double)sizeof(cx<T>) * N, 0);
  cudaError_t e = launch_pdl(k_norm_partial<T>, dim3(nb), dim3(RED_THREADS), 0, s, v, N, ldexp(1.0, -exp_scale),
                             partial);
  if (e == cudaSuccess)
    e = launch_pdl(k_norm_finish, dim3(1), dim3(RED_THREADS), 0, s, (const double*)partial, nb,
                   ldexp(1.0, exp_scale), out);
  count_launch(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_max_exp(const double2* v, long long N, int* out, cudaStream_t s) {
  k_set_int<<<1, 1, 0, s>>>(out, -2000);
  k_max_exp<<<flat_blocks(N), RED_THREADS, 0, s>>>(v, N, out);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_coefs(int dim, const Level& L, const double2* const* chi_tab, int n_gauss,
                         double k2, cudaStream_t s) {
  TabPtrs t{};
  for (int i = 0; i < n_gauss; ++i) t.p[i] = chi_tab[i];
  dim3 g = grid_of(dim, L.m), blk(BX, BY);
  if (dim == 2)
    k_coefs<2><<<g, blk, 0, s>>>(t, n_gauss, L.m, k2, L.c, L.q64, L.dinv64, L.q32, L.dinv32);
  else
    k_coefs<3><<<g, blk, 0, s>>>(t, n_gauss, L.m, k2, L.c, L.q64, L.dinv64, L.q32, L.dinv32);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_incident(double2* tab, int dim, int m, double lo, double h, double k, double gamma, const double* eta,
                            cudaStream_t s) {
  k_incident<<<dim3((m + 127) / 128, dim), 128, 0, s>>>(tab, m, lo, h, k, eta[0], eta[1], dim == 3 ? eta[2] : 0.0,
                                                        cos(gamma), sin(gamma));
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rhs(int dim, int m, const double2* const* chi_tab, int n_gauss,
                       const double2* uinc_tab, double k2, double2* b, cudaStream_t s, int* emax) {
  TabPtrs t{};
  for (int i = 0; i < n_gauss; ++i) t.p[i] = chi_tab[i];
  dim3 g((m + BX - 1) / BX, (m + BY - 1) / BY, dim == 3 ? (m + 7) / 8 : 1), blk(BX, BY);
  if (emax) {
    k_set_int<<<1, 1, 0, s>>>(emax, -2000);
    count_launch();
  }
  if (dim == 2) k_rhs<2><<<g, blk, 0, s>>>(t, n_gauss, uinc_tab, m, k2, b, emax);
  else k_rhs<3><<<g, blk, 0, s>>>(t, n_gauss, uinc_tab, m, k2, b, emax);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_refine_residual(int dim, const Level& L, const double2* u, const double2* b, int s_exp,
                                   float2* r32, double* partial, int nblk, double* out, cudaStream_t s) {
  if (L.N >= (1ll << 31)) return cudaErrorInvalidValue;
  const int gx = (L.m + RED_THREADS - 1) / RED_THREADS;
  const int nrows = dim == 3 ? L.m * L.m : L.m;
  int gy = nblk / gx;
  gy = gy < 1 ? 1 : (gy > nrows ? nrows : gy);
  if (gx * gy > nblk) return cudaErrorInvalidValue;
  ProfScope ps(PF_MG64, s, (16.0 * 3 + 8.0) * L.N, 0);
  cudaError_t e = (dim == 2)
      ? launch_pdl(k_refine_residual<2>, dim3(gx, gy), dim3(RED_THREADS), 0, s, u, b, (const double2*)L.q64, L.c,
                   L.m, s_exp, r32, partial)
      : launch_pdl(k_refine_residual<3>, dim3(gx, gy), dim3(RED_THREADS), 0, s, u, b, (const double2*)L.q64, L.c,
                   L.m, s_exp, r32, partial);
  if (e == cudaSuccess)
    e = launch_pdl(k_norm_finish, dim3(1), dim3(RED_THREADS), 0, s, (const double*)partial, gx * gy,
                   ldexp(1.0, s_exp), out);
  count_launch(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_update64_fixed(double2* u, const float2* e, long long N, int s_exp, cudaStream_t s) {
  if (N >= (1ll << 31)) return cudaErrorInvalidValue;
  ProfScope ps(PF_MG64, s, 40.0 * N, 0);
  cudaError_t err = launch_pdl(abs(s_exp) <= bits::WIDEN_NEAR ? k_update64_fixed<true> : k_update64_fixed<false>,
                               dim3(flat_blocks(N)), dim3(256), 0, s, u, e, (int)N, s_exp, ldexp(1.0, s_exp));
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_first_residual(const double2* b, long long N, int s_exp, float2* r32, double* partial, int nblk,
                                  double* out, cudaStream_t s) {
  if (N >= (1ll << 31)) return cudaErrorInvalidValue;
  const long long need = (N + RED_THREADS - 1) / RED_THREADS;
  const int nb = (int)(need < nblk ? (need < 1 ? 1 : need) : nblk), ex = abs(s_exp) <= 400 ? 0 : s_exp;
  ProfScope ps(PF_MG64, s, 24.0 * N, 0);
  cudaError_t e = launch_pdl(k_first_residual, dim3(nb), dim3(RED_THREADS), 0, s, b, (int)N, ldexp(1.0, -ex), s_exp, r32,
                             partial);
  if (e == cudaSuccess)
    e = launch_pdl(k_norm_finish, dim3(1), dim3(RED_THREADS), 0, s, (const double*)partial, nb, ldexp(1.0, ex), out);
  count_launch(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_inject_q(int dim, const Level& F, const Level& C, cudaStream_t s) {
  dim3 g = grid_of(dim, C.m), blk(BX, BY);
  if (dim == 2) k_inject_q<2><<<g, blk, 0, s>>>(F.q64, F.m, C.q64, C.m);
  else k_inject_q<3><<<g, blk, 0, s>>>(F.q64, F.m, C.q64, C.m);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_coefs_from_q(int dim, const Level& L, cudaStream_t s) {
  dim3 g = grid_of(dim, L.m), blk(BX, BY);
  if (dim == 2) k_coefs_from_q<2><<<g, blk, 0, s>>>(L.q64, L.m, L.c, L.dinv64, L.q32, L.dinv32);
  else k_coefs_from_q<3><<<g, blk, 0, s>>>(L.q64, L.m, L.c, L.dinv64, L.q32, L.dinv32);
  count_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_zero(cx<T>* v, long long N, cudaStream_t s) {
  ProfScope ps(mg_family<T>(), s, (double)sizeof(cx<T>) * N, 0);
  cudaError_t e = launch_pdl(k_zero<T>, dim3(flat_blocks(N)), dim3(256), 0, s, v, N);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

#define CSFF_INST(T)                                                                                   \
  template cudaError_t launch_residual<T>(int, const Level&, const cx<T>*, const cx<T>*, cx<T>*,       \
                                          cudaStream_t);                                               \
  template cudaError_t launch_jacobi<T>(int, const Level&, double, const cx<T>*, const cx<T>*, cx<T>*, \
                                        cudaStream_t);                                                 \
  template cudaError_t launch_rbgs<T>(int, const Level&, cx<T>*, const cx<T>*, cudaStream_t);         \
  template cudaError_t launch_restrict<T>(int, const Level&, const Level&, const cx<T>*, cx<T>*,       \
                                          cudaStream_t);                                               \
  template cudaError_t launch_prolong_add<T>(int, const Level&, const Level&, const cx<T>*, cx<T>*,    \
                                             cudaStream_t);                                            \
  template cudaError_t launch_coarse_solve<T>(const cx<T>*, int, const cx<T>*, cx<T>*, cudaStream_t, int, int);     \
  template cudaError_t launch_norm2<T>(const cx<T>*, long long, int, double*, int, double*,            \
                                       cudaStream_t);                                                  \
  template cudaError_t launch_zero<T>(cx<T>*, long long, cudaStream_t);

CSFF_INST(double)
CSFF_INST(float)

}  // namespace csff
