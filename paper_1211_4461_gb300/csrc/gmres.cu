// GMRES(m) cycles as the multigrid smoother (Sec. 3.3: a Krylov method such
// as GMRES(m), m = 2 or 3, replaces omega-Jacobi / Gauss-Seidel smoothing so
// that rotation angles near 10 degrees stay stable; Tables 2-3 use GMRES(3)
// at gamma = 9.9 degrees).  One smoothing step from the iterate u:
//
//   r0 = b - A u,  beta = ||r0||,  v_0 = r0 / beta
//   for j < m:  w = A v_j;  for i <= j: h_ij = (v_i, w), w -= h_ij v_i
//               (modified Gram-Schmidt);  h_{j+1,j} = ||w||;  v_{j+1} = w / h_{j+1,j}
//   y = argmin_y || beta e_1 - H y ||_2  (complex Givens rotations),  u += V y
//
// The kernels work with A'' = kappa A and b'' = kappa b, kappa = h^2 e^{2 i
// gamma}: a common factor of the system changes neither the Krylov space nor
// the minimiser, and it makes the stencil's weights real, A'' v = 2d v - sum_nbr
// v - (kappa q) v.  The basis vectors are kept unnormalised, w_0 = r'' and
// w_{j+1} = A'' w_j - sum_i alpha_ij w_i, h_ij = (w_i, w) / (n_i n_j), alpha_ij =
// (w_i, w) / n_i^2, n_i = ||w_i||, so no pass only scales a vector.
//
// Bound by the FP64 pipe on large levels (136 operations an unknown for
// m = 3) and by launches below: every pass that changes a vector also forms
// the inner product that the next one needs.  A pass ends when its blocks have
// written their partial sums, at most GM_NB of each; the passes that need a
// scalar sum the partials themselves, every block for itself and in the same
// order, while their own first loads are in flight (a last block that joins
// them, behind a fence and a counter, costs 2 us a pass on small levels), and
// every pass lets its successor be set up at once.  GMRES(3) takes 11 launches,
// 34 with passes for each inner product, its final sum, each update and each
// scaling; a 129^3 solve (10 cycles) 34.1 -> 21.5 ms, its finest level at about
// four fifths of the FP64 pipe's rate (one warp instruction in 19 clocks an
// SM, one in 65 from a single warp).  A step is graph-capturable and never
// synchronises with the host.  Inner products and norms accumulate in FP64 for
// both cycle precisions.  A zero h_{j+1,j} (the Krylov space is
// invariant: the Arnoldi process breaks down) ends the basis: the least-squares
// step uses the first j+1 columns only.
#include "csff_internal.h"

namespace csff {
namespace {

constexpr int GT = 1024;           // most threads of a block
// partial sums: norm_j in slot j, (w_i, w) of column j in slot dot_slot(i, j)
__host__ __device__ constexpr int dot_slot(int i, int j) { return GM_MAX + 1 + j * (j + 1) / 2 + i; }
static_assert(dot_slot(GM_MAX - 1, GM_MAX - 1) < GM_SLOTS, "partial sums");

__device__ __forceinline__ double2 dmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 dconj(double2 a) { return make_double2(a.x, -a.y); }

// sum over the block, valid in thread 0: halving rounds through shared memory
// (a butterfly would keep every thread's FP64 lanes busy in every round)
__device__ __forceinline__ double2 block_sum2(double2 v, double2* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int h = blockDim.x >> 1; h >= 32; h >>= 1) {
    if (t < h) {
      v.x += sh[t + h].x;
      v.y += sh[t + h].y;
      sh[t] = v;
    }
    __syncthreads();
  }
  if (t < 32)
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
  return v;
}

// y = argmin || beta e_1 - H y ||_2 over the first k columns (k = M, or the
// column after which the Arnoldi process broke down), by complex Givens
// rotations G_j = [c s; -conj(s) c] with c = |a|/r, s = (a/|a|) conj(b)/r,
// r = sqrt(|a|^2 + b^2), which zero the (real) subdiagonal entry b under a, then
// back substitution; the step's coefficients z_j = y_j / n_j (zero from k on).
// sums: the slots' totals.  One thread.
template <int M>
__device__ void gm_lsq(const double2* sums, double2* z) {
  double nrm[M + 1], inv[M + 1];
  int k = M;
#pragma unroll
  for (int j = M; j >= 0; --j) {
    const double n2 = sums[j].x;
    inv[j] = n2 > 0.0 ? rsqrt(n2) : 0.0;
    nrm[j] = n2 > 0.0 ? n2 * inv[j] : sqrt(n2);
    if (nrm[j] == 0.0) k = j;
  }
  if (!(nrm[0] > 0.0)) k = 0;
  double2 R[M][M], g[M + 1];
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M; ++j) R[i][j] = i <= j ? cscale(sums[dot_slot(i, j)], inv[i] * inv[j]) : make_double2(0.0, 0.0);
#pragma unroll
  for (int i = 0; i <= M; ++i) g[i] = make_double2(i == 0 ? nrm[0] : 0.0, 0.0);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    if (j < k) {
      const double2 a = R[j][j];
      const double b = nrm[j + 1] * inv[j], na2 = a.x * a.x + a.y * a.y, r2 = na2 + b * b;
      double c;
      double2 s;
      if (r2 == 0.0) {
        c = 1.0;
        s = make_double2(0.0, 0.0);
      } else if (na2 == 0.0) {
        c = 0.0;
        s = make_double2(1.0, 0.0);
      } else {
        const double ir = rsqrt(r2), ia = rsqrt(na2);
        c = na2 * ia * ir;
        s = make_double2(a.x * ia * b * ir, a.y * ia * b * ir);
      }
      const double2 sc = dconj(s);
      R[j][j] = make_double2(c * a.x + s.x * b, c * a.y + s.y * b);
#pragma unroll
      for (int col = j + 1; col < M; ++col) {
        const double2 x = R[j][col], z = (j + 1 < M) ? R[j + 1 < M ? j + 1 : j][col] : make_double2(0.0, 0.0);
        const double2 sz = dmul(s, z), scx = dmul(sc, x);
        R[j][col] = make_double2(c * x.x + sz.x, c * x.y + sz.y);
        if (j + 1 < M) R[j + 1 < M ? j + 1 : j][col] = make_double2(c * z.x - scx.x, c * z.y - scx.y);
      }
      const double2 gx = g[j], scgx = dmul(sc, gx);       // g[j + 1] is still zero
      g[j] = cscale(gx, c);
      g[j + 1] = make_double2(-scgx.x, -scgx.y);
    }
  }
  double2 y[M];
#pragma unroll
  for (int j = M - 1; j >= 0; --j) {
    y[j] = make_double2(0.0, 0.0);
    if (j < k) {
      double2 t = g[j];
#pragma unroll
      for (int col = j + 1; col < M; ++col)
        if (col < k) {
          const double2 p = dmul(R[j][col], y[col]);
          t = make_double2(t.x - p.x, t.y - p.y);
        }
      const double2 d = R[j][j];
      const double dd = d.x * d.x + d.y * d.y;
      if (dd > 0.0) {
        const double id = 1.0 / dd;
        y[j] = make_double2((t.x * d.x + t.y * d.y) * id, (t.y * d.x - t.x * d.y) * id);
      }
    }
    z[j] = cscale(y[j], inv[j]);
  }
}

// the pass's sum of v over the block into slot q of the partials
__device__ __forceinline__ void gm_put(double2 v, double2* sh, double2* __restrict__ part, int q) {
  v = block_sum2(v, sh);
  if (threadIdx.x == 0) part[(size_t)q * GM_NB + blockIdx.x] = v;
}

// total of the nb partials of a slot, by one warp (in every lane)
__device__ __forceinline__ double2 gm_total(const double2* __restrict__ part, int nb, int q) {
  double2 p[GM_NB / 32 + 1], v = make_double2(0.0, 0.0);
#pragma unroll
  for (int k = 0; k <= GM_NB / 32; ++k) {
    const int t = k * 32 + (threadIdx.x & 31);
    p[k] = t < nb ? part[(size_t)q * GM_NB + t] : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int k = 0; k <= GM_NB / 32; ++k) {
    v.x += p[k].x;
    v.y += p[k].y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}


// A'' v at point i of row (iy, iz): 2 D v - sum_nbr v - kq v, fused
// multiply-adds, the neighbours summed by pairs
template <typename T, int D>
__device__ __forceinline__ cx<T> gm_apply(const cx<T>* __restrict__ v, const cx<T>* __restrict__ kq, cx<T> vj,
                                          long long i, int ix, int iy, int iz, int m) {
  using C = cx<T>;
  const C z = mk<C>((T)0, (T)0);
  C s = cadd(ix > 0 ? v[i - 1] : z, ix < m - 1 ? v[i + 1] : z);
  s = cadd(s, cadd(iy > 0 ? v[i - m] : z, iy < m - 1 ? v[i + m] : z));
  if (D == 3) {
    const long long p = (long long)m * m;
    s = cadd(s, cadd(iz > 0 ? v[i - p] : z, iz < m - 1 ? v[i + p] : z));
  }
  const C q = kq[i];
  const T d = (T)(2 * D);
  return mk<C>(fma(-q.x, vj.x, fma(q.y, vj.y, fma(d, vj.x, -s.x))), fma(-q.x, vj.y, fma(-q.y, vj.x, fma(d, vj.y, -s.y))));
}

// blocks of blockDim.x = tx * ty threads: tx along a row, ty rows at a time
struct Walk { int tx, ix, row; };
__device__ __forceinline__ Walk walk(int tx) {
  const int y = threadIdx.x / tx;
  return Walk{tx, (int)threadIdx.x - y * tx, (int)(blockIdx.x * (blockDim.x / tx)) + y};
}

// w = kappa b - A'' u (the residual r'') and its norm n_0
template <typename T, int D>
__global__ void __launch_bounds__(GT) k_gm_first(const cx<T>* __restrict__ u, const cx<T>* __restrict__ b,
                                                 const cx<T>* __restrict__ kq, cx<T> kappa, int m, int tx,
                                                 cx<T>* __restrict__ w, double2* __restrict__ part) {
  pdl_prologue();
  pdl_trigger();
  __shared__ double2 sh[GT];
  const int nrows = (D == 3) ? m * m : m, step = gridDim.x * (blockDim.x / tx);
  const Walk k = walk(tx);
  double2 acc = make_double2(0.0, 0.0);
  for (int row = k.row; row < nrows; row += step) {
    const int iz = (D == 3) ? row / m : 0, iy = (D == 3) ? row - iz * m : row;
    for (int ix = k.ix; ix < m; ix += tx) {
      const long long i = (long long)row * m + ix;
      const cx<T> a = gm_apply<T, D>(u, kq, u[i], i, ix, iy, iz, m), bj = b[i];
      const cx<T> r = mk<cx<T>>(fma(kappa.x, bj.x, fma(-kappa.y, bj.y, -a.x)), fma(kappa.x, bj.y, fma(kappa.y, bj.x, -a.y)));
      w[i] = r;
      acc.x = fma((double)r.x, (double)r.x, fma((double)r.y, (double)r.y, acc.x));
    }
  }
  gm_put(acc, sh, part, 0);
}

// w = A'' v_j and (v_0, w)
template <typename T, int D>
__global__ void __launch_bounds__(GT) k_gm_apply(const cx<T>* __restrict__ v, const cx<T>* __restrict__ v0,
                                                 const cx<T>* __restrict__ kq, int m, int tx, cx<T>* __restrict__ w,
                                                 double2* __restrict__ part, int j) {
  pdl_prologue();
  pdl_trigger();
  __shared__ double2 sh[GT];
  const int nrows = (D == 3) ? m * m : m, step = gridDim.x * (blockDim.x / tx);
  const Walk k = walk(tx);
  double2 acc = make_double2(0.0, 0.0);
  for (int row = k.row; row < nrows; row += step) {
    const int iz = (D == 3) ? row / m : 0, iy = (D == 3) ? row - iz * m : row;
    for (int ix = k.ix; ix < m; ix += tx) {
      const long long i = (long long)row * m + ix;
      const cx<T> vj = v[i], a = gm_apply<T, D>(v, kq, vj, i, ix, iy, iz, m), x = j == 0 ? vj : v0[i];
      w[i] = a;
      const double xr = x.x, xi = x.y, yr = a.x, yi = a.y;
      acc.x = fma(xr, yr, fma(xi, yi, acc.x));
      acc.y = fma(xr, yi, fma(-xi, yr, acc.y));
    }
  }
  gm_put(acc, sh, part, dot_slot(0, j));
}

// w -= alpha v_i, alpha = (v_i, w) / n_i^2, then (v_{i+1}, w), or with i == j
// the norm n_{j+1}.  ni, nd: blocks of the passes that formed n_i^2 and (v_i, w).
template <typename T>
__global__ void __launch_bounds__(GT) k_gm_orth(cx<T>* __restrict__ w, const cx<T>* __restrict__ vi,
                                                const cx<T>* __restrict__ vn, long long N, double2* __restrict__ part,
                                                int ni, int nd, int i, int j) {
  pdl_prologue();
  pdl_trigger();
  __shared__ double2 sh[GT], tot[2];
  const cx<T> z = mk<cx<T>>((T)0, (T)0);
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  cx<T> a = z, b = z, x = z;
  if (t < N) {
    a = vi[t];
    b = w[t];
    if (i < j) x = vn[t];
  }
  if (threadIdx.x < 64) {
    const bool norm = threadIdx.x >= 32;
    const double2 s = gm_total(part, norm ? ni : nd, norm ? i : dot_slot(i, j));
    if ((threadIdx.x & 31) == 0) tot[norm] = s;
  }
  __syncthreads();
  const double n2 = tot[1].x, in2 = n2 > 0.0 ? 1.0 / n2 : 0.0;
  const double2 h = cscale(tot[0], in2);
  double2 acc = make_double2(0.0, 0.0);
  while (t < N) {
    const double vr = a.x, vm = a.y;
    const cx<T> r = mk<cx<T>>((T)fma(-h.x, vr, fma(h.y, vm, (double)b.x)), (T)fma(-h.x, vm, fma(-h.y, vr, (double)b.y)));
    w[t] = r;
    const double yr = r.x, yi = r.y;
    if (i < j) {
      const double xr = x.x, xi = x.y;
      acc.x = fma(xr, yr, fma(xi, yi, acc.x));
      acc.y = fma(xr, yi, fma(-xi, yr, acc.y));
    } else {
      acc.x = fma(yr, yr, fma(yi, yi, acc.x));
    }
    t += (long long)gridDim.x * blockDim.x;
    if (t < N) {
      a = vi[t];
      b = w[t];
      if (i < j) x = vn[t];
    }
  }
  gm_put(acc, sh, part, i < j ? dot_slot(i + 1, j) : j + 1);
}

// the least-squares solution, u += sum_j z_j w_j.  na, no: blocks of the passes
// over rows (the first and the applications) and of the orthogonalisations.
template <typename T, int M>
__global__ void __launch_bounds__(GT) k_gm_update(cx<T>* __restrict__ u, const cx<T>* __restrict__ V, long long N,
                                                  const double2* __restrict__ part, int na, int no) {
  pdl_prologue();
  pdl_trigger();
  __shared__ double2 sums[GM_SLOTS], z[M];
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int q = warp; q <= dot_slot(M - 1, M - 1); q += nw) {
    if (q > M && q <= GM_MAX) continue;
    bool from_apply = q == 0;                 // n_0 from the first pass, (w_0, w) from the applications
#pragma unroll
    for (int j = 0; j < M; ++j) from_apply |= q == dot_slot(0, j);
    const double2 s = gm_total(part, from_apply ? na : no, q);
    if ((threadIdx.x & 31) == 0) sums[q] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) gm_lsq<M>(sums, z);
  __syncthreads();
  double2 y[M];
#pragma unroll
  for (int j = 0; j < M; ++j) y[j] = z[j];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const cx<T> u0 = u[i];
    double ar = u0.x, ai = u0.y;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const cx<T> v = V[(long long)j * N + i];
      ar = fma(y[j].x, (double)v.x, fma(-y[j].y, (double)v.y, ar));
      ai = fma(y[j].x, (double)v.y, fma(y[j].y, (double)v.x, ai));
    }
    u[i] = mk<cx<T>>((T)ar, (T)ai);
  }
}

// kappa q in both precisions
__global__ void k_gm_coefs(const double2* __restrict__ q, double2 kappa, long long N, double2* __restrict__ kq64,
                           float2* __restrict__ kq32) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = dmul(kappa, q[i]);
    kq64[i] = v;
    kq32[i] = make_float2((float)v.x, (float)v.y);
  }
}

template <typename T> const cx<T>* kq_of(const Level& L);
template <> const double2* kq_of<double>(const Level& L) { return L.kq64; }
template <> const float2* kq_of<float>(const Level& L) { return L.kq32; }

double2 kappa_of(const Level& L) {                    // 1 / c
  const double d = L.c.x * L.c.x + L.c.y * L.c.y;
  return make_double2(L.c.x / d, -L.c.y / d);
}

template <typename T, int M>
cudaError_t gmres_step(int dim, const Level& L, cx<T>* u, const cx<T>* b, cx<T>* V, double2* part, cudaStream_t s) {
  const long long N = L.N;
  // at most one block an SM; small levels in small blocks, so that their FP64
  // work meets many SMs' pipes
  int nt = 64;
  while (nt < GT && (long long)nt * GM_NB < N) nt *= 2;
  int tx = 1;
  while (tx < L.m && tx < nt) tx *= 2;
  const long long rows = dim == 3 ? (long long)L.m * L.m : L.m;
  auto blocks = [&](long long need) { return (int)(need < GM_NB ? (need < 1 ? 1 : need) : GM_NB); };
  const int na = blocks((rows + nt / tx - 1) / (nt / tx)), no = blocks((N + nt - 1) / nt);
  const dim3 gr(na), gf(no), bt(nt);
  const double2 kd = kappa_of(L);
  const cx<T> kappa = mk<cx<T>>((T)kd.x, (T)kd.y);
  const cx<T>* kq = kq_of<T>(L);
  ProfScope ps(mg_family<T>(), s, 0, 0);
  cudaError_t e = cudaSuccess;
  int launches = 0;
  auto ok = [&](cudaError_t r) {
    ++launches;
    if (e == cudaSuccess) e = r;
  };
  if (dim == 2) ok(launch_pdl(k_gm_first<T, 2>, gr, bt, 0, s, (const cx<T>*)u, b, kq, kappa, L.m, tx, V, part));
  else ok(launch_pdl(k_gm_first<T, 3>, gr, bt, 0, s, (const cx<T>*)u, b, kq, kappa, L.m, tx, V, part));
  for (int j = 0; j < M; ++j) {
    const cx<T>* vj = V + (long long)j * N;
    cx<T>* w = V + (long long)(j + 1) * N;
    if (dim == 2) ok(launch_pdl(k_gm_apply<T, 2>, gr, bt, 0, s, vj, (const cx<T>*)V, kq, L.m, tx, w, part, j));
    else ok(launch_pdl(k_gm_apply<T, 3>, gr, bt, 0, s, vj, (const cx<T>*)V, kq, L.m, tx, w, part, j));
    for (int i = 0; i <= j; ++i) {
      const cx<T>* vi = V + (long long)i * N;
      ok(launch_pdl(k_gm_orth<T>, gf, bt, 0, s, w, vi, i < j ? vi + N : vi, N, part, i == 0 ? na : no,
                    i == 0 ? na : no, i, j));
    }
  }
  ok(launch_pdl(k_gm_update<T, M>, gf, bt, 0, s, u, (const cx<T>*)V, N, (const double2*)part, na, no));
  count_launch(launches);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_gmres_coefs(const Level& L, cudaStream_t s) {
  const long long need = (L.N + GT - 1) / GT;
  k_gm_coefs<<<(unsigned)(need < 152 * 8 ? need : 152 * 8), GT, 0, s>>>(L.q64, kappa_of(L), L.N, L.kq64, L.kq32);
  count_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gmres_step(int dim, const Level& L, int m, cx<T>* u, const cx<T>* b, cx<T>* V, double2* part,
                              cudaStream_t s) {
  static_assert(GM_MAX == 4, "the krylov_m that are instantiated");
  switch (m) {
    case 1: return gmres_step<T, 1>(dim, L, u, b, V, part, s);
    case 2: return gmres_step<T, 2>(dim, L, u, b, V, part, s);
    case 3: return gmres_step<T, 3>(dim, L, u, b, V, part, s);
    case 4: return gmres_step<T, 4>(dim, L, u, b, V, part, s);
  }
  return cudaErrorInvalidValue;
}

template cudaError_t launch_gmres_step<double>(int, const Level&, int, double2*, const double2*, double2*, double2*,
                                               cudaStream_t);
template cudaError_t launch_gmres_step<float>(int, const Level&, int, float2*, const float2*, float2*, double2*,
                                              cudaStream_t);

}  // namespace csff
