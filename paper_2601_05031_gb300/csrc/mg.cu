// Poisson kernels: red-black Gauss-Seidel / SOR sweeps, exact-defect
// residual with restriction, trilinear prolongation, coarsest-level solve and
// residual norms.  Main-text eqs. gen1 and gen3 are Poisson problems per
// Cartesian component; the paper solves them "using an iterative method"
// (numerical-implementation section) -- this file is that method on the GPU:
// cell-centred multigrid V-cycles (or red-black SOR), templated on the
// storage type (float for the mixed path, double for the FP64 path).
#include <algorithm>

#include "internal.h"

namespace vsv {

// Visit the neighbour values of cell (i,j,k) on level L in the order x-, x+,
// y-, y+, z-, z+, skipping Dirichlet ghosts, which are counted in nwall
// instead (their value is -alpha * x_c, zero on the fine level).
template <class T, class F>
__device__ __forceinline__ void for_nb(const T* __restrict__ x, const Level& L, int i, int j, int k,
                                       long long c, int& nwall, F&& f) {
  nwall = 0;
  const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
  const long long sy = nx, sz = (long long)nx * ny;
  if (L.act[0]) {
    if (i > 0) f(x[c - 1]); else if (L.per[0]) f(x[c + nx - 1]); else ++nwall;
    if (i < nx - 1) f(x[c + 1]); else if (L.per[0]) f(x[c - (nx - 1)]); else ++nwall;
  }
  if (L.act[1]) {
    if (j > 0) f(x[c - sy]); else if (L.per[1]) f(x[c + (ny - 1) * sy]); else ++nwall;
    if (j < ny - 1) f(x[c + sy]); else if (L.per[1]) f(x[c - (ny - 1) * sy]); else ++nwall;
  }
  if (L.act[2]) {
    if (k > 0) f(x[c - sz]); else if (L.per[2]) f(x[c + (nz - 1) * sz]); else ++nwall;
    if (k < nz - 1) f(x[c + sz]); else if (L.per[2]) f(x[c - (nz - 1) * sz]); else ++nwall;
  }
}

// Sum of the neighbour values as ((x- + x+) + (y- + y+)) + (z- + z+), a
// Dirichlet ghost or an inactive axis contributing zero.  Every sweep,
// residual and transfer kernel sums in this order, so they agree bit for bit.
template <class T>
__device__ __forceinline__ T sum_nb(const T* __restrict__ x, const Level& L, int i, int j, int k,
                                    long long c, int& nwall) {
  nwall = 0;
  const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
  const long long sy = nx, sz = (long long)nx * ny;
  T a = 0, b = 0, s[3];
  if (L.act[0]) {
    if (i > 0) a = x[c - 1]; else if (L.per[0]) a = x[c + nx - 1]; else ++nwall;
    if (i < nx - 1) b = x[c + 1]; else if (L.per[0]) b = x[c - (nx - 1)]; else ++nwall;
  }
  s[0] = a + b;
  a = 0; b = 0;
  if (L.act[1]) {
    if (j > 0) a = x[c - sy]; else if (L.per[1]) a = x[c + (ny - 1) * sy]; else ++nwall;
    if (j < ny - 1) b = x[c + sy]; else if (L.per[1]) b = x[c - (ny - 1) * sy]; else ++nwall;
  }
  s[1] = a + b;
  a = 0; b = 0;
  if (L.act[2]) {
    if (k > 0) a = x[c - sz]; else if (L.per[2]) a = x[c + (nz - 1) * sz]; else ++nwall;
    if (k < nz - 1) b = x[c + sz]; else if (L.per[2]) b = x[c - (nz - 1) * sz]; else ++nwall;
  }
  s[2] = a + b;
  return (s[0] + s[1]) + s[2];
}

// b with the sign of a rhs factor (1 or -1), by an integer operation, which
// takes no FP64 unit's time.
__device__ __forceinline__ double sign_of(double b, double beta) {
  return __hiloint2double(__double2hiint(b) ^ (__double2hiint(beta) & (int)0x80000000u),
                          __double2loint(b));
}
__device__ __forceinline__ float sign_of(float b, float beta) { return beta * b; }

template <class T>
__device__ __forceinline__ T rhs_at(const Rhs3<T>& R, int comp, long long c, int j, int k, int ny) {
  T b = sign_of(R.b_at(comp)[c], R.beta);
  if (R.s_at(comp)) b += R.s_at(comp)[j + (long long)k * ny];
  return b;
}

// ---------------------------------------------------------------- residual value
// r = b - L_h x at one cell, plain arithmetic in T.
template <class T>
__device__ __forceinline__ T resid_plain(const T* __restrict__ x, const Level& L, int i, int j, int k,
                                         long long c, T b) {
  int nwall;
  const T s = sum_nb(x, L, i, j, k, c, nwall);
  return resid_value(b, s, lv_coef<T>(L, nwall), x[c], lv_ih2<T>(L));
}

// Exact defect in FP32 storage: every term of b - (sum_nb - coef x_c)/h^2 is
// accumulated by cascaded summation, so the result equals the real-number
// defect up to one final rounding (the diagonal coefficient enters as an
// FP32 pair; it is the integer 2 d on the fine level of a Poisson problem).
__device__ __forceinline__ float resid_exact(const float* __restrict__ x, const Level& L, int i,
                                             int j, int k, long long c, float b, float ih_hi,
                                             float ih_lo) {
  int nwall;
  CascadeSum t(0.f);
  for_nb(x, L, i, j, k, c, nwall, [&](float v) { t.add(v); });
  t.add_scaled(-L.cdh[nwall], x[c]);
  if (L.cdl[nwall] != 0.f) t.add(-L.cdl[nwall] * x[c]);   // adding -0 would change nothing
  if (ih_hi == 1.f && ih_lo == 0.f) {
    CascadeSum r(b);
    r.add(-t.hi);
    r.add(-t.lo);
    return r.value();
  }
  // (ih_hi + ih_lo) * (t.hi + t.lo) with the leading product split exactly
  float p = __fmul_rn(ih_hi, t.hi);
  float pe = __fmaf_rn(ih_hi, t.hi, -p);
  float rest = __fmaf_rn(ih_hi, t.lo, __fmaf_rn(ih_lo, t.hi, pe));
  CascadeSum r(b);
  r.add(-p);
  r.add(-rest);
  return r.value();
}

template <class T, bool EXACT>
__device__ __forceinline__ T resid_at(const T* __restrict__ x, const Level& L, int i, int j, int k,
                                      long long c, T b, float ih_hi, float ih_lo) {
  if constexpr (EXACT) {
    return resid_exact(x, L, i, j, k, c, b, ih_hi, ih_lo);
  } else {
    return resid_plain(x, L, i, j, k, c, b);
  }
}

// ---------------------------------------------------------------- sweeps
// What a sweep kernel reads of its level, with the constants of relax()
// rounded on the host: a launch carries a third of a Level, and a cell on the
// FP64 path, whose units do two operations per clock and SM, spends no
// operation on them.
template <class T>
struct SweepGeom {
  int nx, ny, nz;
  int act[3], per[3];
  T w[7];          // omega / diagonal for 0 .. 6 wall neighbours
  T h2, c1, beta;  // h^2 (with the sign of the rhs if it has no plane term),
                   // 1 - omega, the sign of the rhs
};

// One colour of a red-black Gauss-Seidel sweep (omega = 1) or SOR sweep
// (the red-black SOR solver, or over-relaxed multigrid smoothing),
// colour = (i + j + k) & 1, in place.  Thread t handles the t-th cell of the
// colour in its x row.  ZERO (colour 0): x is to be taken as zero and holds
// anything: the red cells take the scaled rhs, the black ones zero, as a fill
// and a red half-sweep leave them.
//
// PLANE: the rhs has a plane term (without one the sign of the rhs is in h^2).
// A condition on it, or a factor, inside the kernel becomes a predicate, and an
// FP64 operation that is predicated off takes the units' time like any other.
// FP64: 8 operations per cell and colour (3 with ZERO) instead of 12, 9 with
// PLANE; 139 -> 98 us a colour at 256 x 128 x 128, three components, 139 -> 110
// us with PLANE.
template <class T, bool ZERO, bool PLANE>
__global__ void k_rb_sweep(const __grid_constant__ SweepGeom<T> G, Comp3<T> X, Rhs3<T> R, int color) {
  pdl_begin();
  const int nx = G.nx, ny = G.ny, nz = G.nz;
  int i2, j, k, comp;
  if (!cell3((nx + 1) >> 1, ny, nz, i2, j, k, comp)) return;
  T* __restrict__ x = X.at(comp);
  const int i = 2 * i2 + ((j + k + color) & 1);
  const long long c = lin(i, j, k, nx, ny);
  if (ZERO && (i ^ 1) < nx) x[c + ((i & 1) ? -1 : 1)] = (T)0;
  if (i >= nx) return;
  const long long sy = nx, sz = (long long)nx * ny;
  int nwall = 0;
  T a = 0, b = 0, s[3];
  auto add = [&](int q, bool in, long long d, long long wrap) -> T {
    if (!G.act[q]) return (T)0;
    if (in) return ZERO ? (T)0 : x[c + d];
    if (G.per[q]) return ZERO ? (T)0 : x[c + wrap];
    ++nwall;
    return (T)0;
  };
  a = add(0, i > 0, -1, nx - 1);
  b = add(0, i < nx - 1, 1, 1 - nx);
  s[0] = a + b;
  a = add(1, j > 0, -sy, (ny - 1) * sy);
  b = add(1, j < ny - 1, sy, (1 - ny) * sy);
  s[1] = a + b;
  a = add(2, k > 0, -sz, (nz - 1) * sz);
  b = add(2, k < nz - 1, sz, (1 - nz) * sz);
  s[2] = a + b;
  const T sn = ZERO ? (T)0 : (s[0] + s[1]) + s[2];
  T r = R.b_at(comp)[c];
  if (PLANE) {
    r = sign_of(r, G.beta);
    if (R.s_at(comp)) r += R.s_at(comp)[j + (long long)k * ny];
  }
  x[c] = relax(ZERO ? (T)0 : x[c], nb_term(sn, r, G.h2), G.w[nwall], G.c1);
}

// Residual of the fine (or any) level, restricted to the next coarser level
// by averaging the children of each coarse cell.
template <class T, bool EXACT>
__global__ void k_resid_restrict(Level F, Level C, Comp3<T> X, Rhs3<T> R, Comp3<T> RC, float ih_hi,
                                 float ih_lo) {
  pdl_begin();
  int I, J, K, comp;
  if (!cell3(C.n[0], C.n[1], C.n[2], I, J, K, comp)) return;
  const T* __restrict__ x = X.at(comp);
  const long long t = lin(I, J, K, C.n[0], C.n[1]);
  const int fx = F.n[0] / C.n[0], fy = F.n[1] / C.n[1], fz = F.n[2] / C.n[2];
  T acc = 0;
  for (int dk = 0; dk < fz; ++dk)
    for (int dj = 0; dj < fy; ++dj)
      for (int di = 0; di < fx; ++di) {
        const int i = I * fx + di, j = J * fy + dj, k = K * fz + dk;
        const long long c = lin(i, j, k, F.n[0], F.n[1]);
        const T b = rhs_at(R, comp, c, j, k, F.n[1]);
        acc += resid_at<T, EXACT>(x, F, i, j, k, c, b, ih_hi, ih_lo);
      }
  RC.at(comp)[t] = acc / (T)(fx * fy * fz);
}

// One axis of the cell-centred linear interpolation: the two coarse indices
// and weights for fine index i (child of I = i / f).
template <class T>
struct Interp1 {
  int idx[2];
  T w[2];
};

template <class T>
__device__ __forceinline__ Interp1<T> interp_axis(int i, int f, int nC, int per, T alpha) {
  Interp1<T> r;
  if (f == 1) {
    r.idx[0] = r.idx[1] = i;
    r.w[0] = (T)1;
    r.w[1] = (T)0;
    return r;
  }
  const int I = i >> 1;
  const int off = (i & 1) ? 1 : -1;
  int I2 = I + off;
  r.idx[0] = I;
  r.w[0] = (T)0.75;
  if (I2 < 0 || I2 >= nC) {
    if (per) {
      I2 = (I2 + nC) % nC;
      r.idx[1] = I2;
      r.w[1] = (T)0.25;
    } else {  // ghost = -alpha * e(I)
      r.idx[1] = I;
      r.w[1] = (T)(-0.25) * alpha;
    }
  } else {
    r.idx[1] = I2;
    r.w[1] = (T)0.25;
  }
  return r;
}

// x_fine += P e_coarse (trilinear, cell centred).
template <class T>
__global__ void k_prolong_add(Level F, Level C, Comp3<T> X, Comp3<T> E) {
  pdl_begin();
  int i, j, k, comp;
  if (!cell3(F.n[0], F.n[1], F.n[2], i, j, k, comp)) return;
  const long long t = lin(i, j, k, F.n[0], F.n[1]);
  const T al = lv_alpha<T>(C);
  const Interp1<T> ax = interp_axis<T>(i, F.n[0] / C.n[0], C.n[0], C.per[0], al);
  const Interp1<T> ay = interp_axis<T>(j, F.n[1] / C.n[1], C.n[1], C.per[1], al);
  const Interp1<T> az = interp_axis<T>(k, F.n[2] / C.n[2], C.n[2], C.per[2], al);
  const T* __restrict__ e = E.at(comp);
  T acc = 0;
  for (int c2 = 0; c2 < 2; ++c2)
    for (int b2 = 0; b2 < 2; ++b2)
      for (int a2 = 0; a2 < 2; ++a2) {
        const T w = ax.w[a2] * ay.w[b2] * az.w[c2];
        if (w != (T)0) acc += w * e[lin(ax.idx[a2], ay.idx[b2], az.idx[c2], C.n[0], C.n[1])];
      }
  X.at(comp)[t] += acc;
}

template <class T>
__global__ void k_zero(Comp3<T> X, long long n) {
  pdl_begin();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) X.at(blockIdx.y)[t] = (T)0;
}

// First guess of a solve from the history, written into the oldest buffer
// C: order 0: A; 1: 2A - B; 2: 3(A - B) + C (A = x^n, B = x^{n-1}, C =
// x^{n-2}; extrapolation in time of order 0, 1, 2).
template <class T>
__global__ void k_extrapolate_rot(Comp3<T> A, Comp3<T> B, Comp3<T> C, long long n, int order) {
  pdl_begin();
  const int comp = blockIdx.y;
  const T* __restrict__ a = A.at(comp);
  const T* __restrict__ b = B.at(comp);
  T* __restrict__ c = C.at(comp);
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const T x = a[t];
    if (order == 0) c[t] = x;
    else if (order == 1) c[t] = (T)2 * x - b[t];
    else c[t] = (T)3 * (x - b[t]) + c[t];
  }
}

// y += a x (the inertial right-hand side f - s omega'^n, FP64 path).
template <class T>
__global__ void k_axpy(Comp3<T> Y, Comp3<T> X, T a, long long n) {
  pdl_begin();
  const int comp = blockIdx.y;
  T* __restrict__ y = Y.at(comp);
  const T* __restrict__ x = X.at(comp);
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    y[t] += a * x[t];
}

// Coarsest level: e = 0, then `sweeps` red-black Gauss-Seidel sweeps in
// shared memory by one block per component.
template <class T>
__global__ void k_coarse_solve(Level L, Comp3<T> E, Comp3<T> RR, int sweeps, T h2) {
  pdl_begin();
  extern __shared__ unsigned char smem_raw[];
  T* e = reinterpret_cast<T*>(smem_raw);
  const int comp = blockIdx.y;
  const long long n = L.cells();
  const T* __restrict__ r = RR.at(comp);
  T* rs = e + n;
  for (long long t = threadIdx.x; t < n; t += blockDim.x) {
    e[t] = 0;
    rs[t] = r[t];
  }
  __syncthreads();
  const int nx = L.n[0], ny = L.n[1], nxh = (nx + 1) >> 1;
  const int nh = nxh * ny * L.n[2];   // cells of one colour, rounded up per row
  for (int s = 0; s < sweeps; ++s)
    for (int color = 0; color < 2; ++color) {
      for (int t2 = threadIdx.x; t2 < nh; t2 += blockDim.x) {
        const int i2 = t2 % nxh, q = t2 / nxh;
        const int j = q % ny, k = q / ny;
        const int i = 2 * i2 + ((j + k + color) & 1);
        if (i >= nx) continue;
        const int t = (k * ny + j) * nx + i;
        int nwall;
        const T sum = sum_nb(e, L, i, j, k, t, nwall);
        e[t] = relax(e[t], nb_term(sum, rs[t], h2), lv_rc<T>(L, nwall), (T)0);
      }
      __syncthreads();
    }
  for (long long t = threadIdx.x; t < n; t += blockDim.x) E.at(comp)[t] = e[t];
}

// ||b - L x||^2 and ||b||^2 (FP64 accumulation), published by norm_publish, with
// row_lanes threads on each row.
template <class T, bool EXACT>
__global__ void k_resid_norm(const __grid_constant__ Level L, Comp3<T> X, Rhs3<T> R, double* partials,
                             float ih_hi, float ih_lo, Scalars* S, double* host) {
  pdl_begin();
  const int comp = blockIdx.y;
  const T* __restrict__ x = X.at(comp);
  const int rows = L.n[1] * L.n[2], lanes = row_lanes(L.n[0]);
  double rr = 0.0, bb = 0.0;
  for (int row = (blockIdx.x * kBlock + threadIdx.x) / lanes; row < rows;
       row += gridDim.x * kBlock / lanes) {
    const int k = row / L.n[1], j = row - k * L.n[1];
    T r2 = 0, b2 = 0;   // per-row partial in T, then FP64 across rows
    for (int i = threadIdx.x & (lanes - 1); i < L.n[0]; i += lanes) {
      const long long t = lin(i, j, k, L.n[0], L.n[1]);
      const T b = rhs_at(R, comp, t, j, k, L.n[1]);
      const T r = resid_at<T, EXACT>(x, L, i, j, k, t, b, ih_hi, ih_lo);
      r2 += r * r;
      b2 += b * b;
    }
    rr += (double)r2;
    bb += (double)b2;
  }
  __shared__ double buf[2 * kBlock];
  norm_publish(rr, bb, buf, partials, gridDim.x, gridDim.y, comp, blockIdx.x, S, host);
}

// ---------------------------------------------------------------- blocked transfers
// Both kernels below take one coarse cell per thread and handle its 2x2x2
// fine children together; they require every axis to be coarsened by two
// (the coarse-level index I owns fine cells 2I and 2I+1 on every axis).

// Index of an outer neighbour (one cell beyond a 2-cell block) along one
// axis: wrapped on a periodic axis, -1 for a Dirichlet ghost.
__device__ __forceinline__ int outer_idx(int i, int n, int per) {
  if (i < 0) return per ? i + n : -1;
  if (i >= n) return per ? i - n : -1;
  return i;
}

template <class T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

template <class T>
__device__ __forceinline__ void ld2(const T* p, T& a, T& b) {
  const typename Vec2<T>::type v = *reinterpret_cast<const typename Vec2<T>::type*>(p);
  a = v.x;
  b = v.y;
}

// Residual of the 8 children, averaged onto the coarse cell (plain
// arithmetic, neighbours summed pairwise as in sum_nb).  The
// children of coarse x index I are fine 2I, 2I+1 (an aligned pair).
template <class T>
__global__ void k_restrict_block(Level F, Level C, Comp3<T> X, Rhs3<T> R, Comp3<T> RC) {
  pdl_begin();
  int I, J, K, comp;
  if (!cell3(C.n[0], C.n[1], C.n[2], I, J, K, comp)) return;
  const T* __restrict__ x = X.at(comp);
  const int nx = F.n[0], ny = F.n[1], nz = F.n[2];
  const int i0 = 2 * I, j0 = 2 * J, k0 = 2 * K;
  const int xm = outer_idx(i0 - 1, nx, F.per[0]), xp = outer_idx(i0 + 2, nx, F.per[0]);
  const int ym = outer_idx(j0 - 1, ny, F.per[1]), yp = outer_idx(j0 + 2, ny, F.per[1]);
  const int zm = outer_idx(k0 - 1, nz, F.per[2]), zp = outer_idx(k0 + 2, nz, F.per[2]);
  auto row = [&](int j, int k) { return x + ((long long)k * ny + j) * nx; };
  T c[2][2][2], fxm[2][2], fxp[2][2], fym[2][2], fyp[2][2], fzm[2][2], fzp[2][2], b[2][2][2];
#pragma unroll
  for (int kz = 0; kz < 2; ++kz)
#pragma unroll
    for (int jy = 0; jy < 2; ++jy) {
      const T* r = row(j0 + jy, k0 + kz);
      ld2(r + i0, c[kz][jy][0], c[kz][jy][1]);
      fxm[kz][jy] = xm >= 0 ? r[xm] : (T)0;
      fxp[kz][jy] = xp >= 0 ? r[xp] : (T)0;
      const long long t = ((long long)(k0 + kz) * ny + j0 + jy) * nx + i0;
      ld2(R.b_at(comp) + t, b[kz][jy][0], b[kz][jy][1]);
      b[kz][jy][0] = sign_of(b[kz][jy][0], R.beta);
      b[kz][jy][1] = sign_of(b[kz][jy][1], R.beta);
    }
  // one branch for the plane term (per cell it becomes a predicated FP64
  // operation, which takes the units' time all the same).  FP64: 227 -> 211 us
  // with the sign change off the units, 256 x 128 x 128, three components
  if (R.s_at(comp)) {
#pragma unroll
    for (int kz = 0; kz < 2; ++kz)
#pragma unroll
      for (int jy = 0; jy < 2; ++jy) {
        const T s = R.s_at(comp)[j0 + jy + (long long)(k0 + kz) * ny];
        b[kz][jy][0] += s;
        b[kz][jy][1] += s;
      }
  }
#pragma unroll
  for (int kz = 0; kz < 2; ++kz) {
    if (ym >= 0) ld2(row(ym, k0 + kz) + i0, fym[kz][0], fym[kz][1]); else fym[kz][0] = fym[kz][1] = (T)0;
    if (yp >= 0) ld2(row(yp, k0 + kz) + i0, fyp[kz][0], fyp[kz][1]); else fyp[kz][0] = fyp[kz][1] = (T)0;
  }
#pragma unroll
  for (int jy = 0; jy < 2; ++jy) {
    if (zm >= 0) ld2(row(j0 + jy, zm) + i0, fzm[jy][0], fzm[jy][1]); else fzm[jy][0] = fzm[jy][1] = (T)0;
    if (zp >= 0) ld2(row(j0 + jy, zp) + i0, fzp[jy][0], fzp[jy][1]); else fzp[jy][0] = fzp[jy][1] = (T)0;
  }
  const T ih2 = lv_ih2<T>(F);
  T acc = 0;
#pragma unroll
  for (int kz = 0; kz < 2; ++kz)
#pragma unroll
    for (int jy = 0; jy < 2; ++jy)
#pragma unroll
      for (int ix = 0; ix < 2; ++ix) {
        const T v_xm = ix == 0 ? fxm[kz][jy] : c[kz][jy][0];
        const T v_xp = ix == 1 ? fxp[kz][jy] : c[kz][jy][1];
        const T v_ym = jy == 0 ? fym[kz][ix] : c[kz][0][ix];
        const T v_yp = jy == 1 ? fyp[kz][ix] : c[kz][1][ix];
        const T v_zm = kz == 0 ? fzm[jy][ix] : c[0][jy][ix];
        const T v_zp = kz == 1 ? fzp[jy][ix] : c[1][jy][ix];
        const int nwall = (ix == 0 && xm < 0) + (ix == 1 && xp < 0) + (jy == 0 && ym < 0) +
                          (jy == 1 && yp < 0) + (kz == 0 && zm < 0) + (kz == 1 && zp < 0);
        const T s = ((v_xm + v_xp) + (v_ym + v_yp)) + (v_zm + v_zp);
        acc += resid_value(b[kz][jy][ix], s, lv_coef<T>(F, nwall), c[kz][jy][ix], ih2);
      }
  RC.at(comp)[lin(I, J, K, C.n[0], C.n[1])] = acc * (T)0.125;
}

// Increments P e for the 8 children of coarse cell (I,J,K): weights 3/4 and
// 1/4 per axis; the coarse neighbours come from the coarse level's boundary
// rule: periodic wrap, or -alpha * (adjacent cell) per out-of-range axis (the
// linear extrapolation through zero at the wall).  v[c][b][a] is the child
// (2K+c, 2J+b, 2I+a).
template <class T>
__device__ __forceinline__ void prolong_children(const Level& C, const T* __restrict__ e, int I,
                                                 int J, int K, T v[2][2][2]) {
  const int cx_ = C.n[0], cy = C.n[1], cz = C.n[2];
  const T ma = -lv_alpha<T>(C);
  int ix[3], iy[3], iz[3];
  T fx[3], fy[3], fz[3];
  ix[1] = I; iy[1] = J; iz[1] = K;
  fx[1] = fy[1] = fz[1] = (T)1;
#pragma unroll
  for (int s = 0; s < 3; s += 2) {
    const int d = s - 1;
    int t = outer_idx(I + d, cx_, C.per[0]);
    ix[s] = t >= 0 ? t : I; fx[s] = t >= 0 ? (T)1 : ma;
    t = outer_idx(J + d, cy, C.per[1]);
    iy[s] = t >= 0 ? t : J; fy[s] = t >= 0 ? (T)1 : ma;
    t = outer_idx(K + d, cz, C.per[2]);
    iz[s] = t >= 0 ? t : K; fz[s] = t >= 0 ? (T)1 : ma;
  }
  bool wall = (I == 0 || I == cx_ - 1) && !C.per[0];
  wall = wall || ((J == 0 || J == cy - 1) && !C.per[1]);
  wall = wall || ((K == 0 || K == cz - 1) && !C.per[2]);
  T n[3][3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const T* r = e + ((long long)iz[c] * cy + iy[b]) * cx_;
#pragma unroll
      for (int a = 0; a < 3; ++a) n[c][b][a] = r[ix[a]];
    }
  // the boundary factors are all 1 away from walls: one branch around their
  // multiplications (per-value conditions become selects, and the FP64 units
  // then do every product), decided on integers (an FP64 compare is an FP64
  // operation too)
  if (wall) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const T f = fz[c] * fy[b];
#pragma unroll
        for (int a = 0; a < 3; ++a) n[c][b][a] = f * fx[a] * n[c][b][a];
      }
  }
  // the x-interpolated value of each of the nine rows on the even and the odd
  // child's side.  FP64: 76 operations per coarse cell with the eight updates
  // instead of 167; 344 -> 209 us at 256 x 128 x 128, three components
  T p[3][3][2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      p[c][b][0] = prolong_pair(n[c][b][1], n[c][b][0]);
      p[c][b][1] = prolong_pair(n[c][b][1], n[c][b][2]);
    }
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a)
        v[c][b][a] = prolong_sum(p[1][1][a], p[1][2 * b][a], p[2 * c][1][a], p[2 * c][2 * b][a]);
}

// x_fine += P e for the 8 children of one coarse cell per thread.
template <class T>
__global__ void k_prolong_block(Level F, Level C, Comp3<T> X, Comp3<T> E) {
  pdl_begin();
  int I, J, K, comp;
  if (!cell3(C.n[0], C.n[1], C.n[2], I, J, K, comp)) return;
  T v[2][2][2];
  prolong_children<T>(C, E.at(comp), I, J, K, v);
  T* __restrict__ x = X.at(comp);
  const int nx = F.n[0], ny = F.n[1];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      T* p = x + ((long long)(2 * K + c) * ny + 2 * J + b) * nx + 2 * I;
      typename Vec2<T>::type cur = *reinterpret_cast<typename Vec2<T>::type*>(p);
      cur.x += v[c][b][0];
      cur.y += v[c][b][1];
      *reinterpret_cast<typename Vec2<T>::type*>(p) = cur;
    }
}

__host__ __device__ bool blocked_transfer_ok(const Level& F, const Level& C) {
  for (int a = 0; a < 3; ++a)
    if (F.n[a] != 2 * C.n[a]) return false;
  return true;
}

// ---------------------------------------------------------------- coarse V-cycle in one CTA
// The levels from `first` down to the coarsest are small enough to live in
// shared memory; one CTA per component runs the whole lower part of the
// V-cycle there (same operations as the level-by-level kernels: red-black
// sweeps, residual restricted by averaging, trilinear prolongation), which
// replaces dozens of latency-bound launches per V-cycle by one.
//
// One SM runs it once, so its time is set by the instructions it issues, by
// its chain of dependent phases (about 55 on five levels) and by the code it
// has to fetch.  Each level keeps its two colours ((i + j + k) & 1) in
// separate arrays of half the row length: a cell's neighbours are all in the
// other colour's array, at the cell's own index for y and z and at that index
// and one beside it for x, without unused lanes or bank conflicts.  A thread
// holds a run of 1, 2, 4 or 8 planes of one column pair in registers, on the
// coarsest level also 3 or 5 (24 x 12 x 10 cells, 24 sweeps: 22.5 us in runs of
// 5, 57 us in the loop over shared memory that levels which no such runs cover
// evenly take), and the
// boundary rule is resolved once per visit of a level.  A level is worked on
// by only as many warps as it has runs, on a named barrier of its own (a
// single warp needs none); the other warps wait for it to come back.
//
// Measured, one visit of 32 x 16 x 16 cells and below (three CTAs, cold
// caches): 61 -> 44 us, 245 k -> 121 k warp instructions per CTA; 21 us from
// 16 x 8 x 8 cells down.  What is left waits on barriers (2.4 of 8 stall
// cycles per issue), instruction fetch (2.6) and fixed latencies (1.8).  One
// copy of the code serves both directions: separate copies took 97 k
// instructions but 57 us, fetching instructions (8.1), and loops over shared
// memory alone (compact code, 217 k instructions) 59 us.

// q = a / d, with rem = a - q d (0 <= a, 0 < d): a shift and a mask where d
// is a power of two (every level of a power-of-two grid), else a division.
__device__ __forceinline__ int cv_divmod(int a, int d, int& rem) {
  if ((d & (d - 1)) == 0) {
    rem = a & (d - 1);
    return a >> (__ffs(d) - 1);
  }
  const int q = a / d;
  rem = a - q * d;
  return q;
}

__device__ __forceinline__ void cv_sync(int id, int n) {
  if (n == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// A level in shared memory: e and r of each colour, `half` elements apart.
struct CvLevel {
  int e, r;                   // element offsets
  int nx, ny, nz, nxh, cols, half;
  int n;                      // threads that work on it
  int runs, len;              // column pairs x runs along z; planes per run
  bool reg;                   // runs of 1, 2, 4 or 8 planes (3 or 5 too on the coarsest
                              // level) cover the level evenly
  __device__ __forceinline__ CvLevel(const CoarseCycle& CC, int l) {
    const Level& L = CC.lv[l];
    nx = L.n[0]; ny = L.n[1]; nz = L.n[2];
    nxh = (nx + 1) >> 1;
    cols = nxh * ny;
    half = cols * nz;
    e = (int)CC.off[l];
    r = e + 2 * half;
    n = CC.threads[l];
    len = CC.run[l];
    runs = CC.runs[l];
    reg = CC.reg[l];
  }
  __device__ __forceinline__ int at(int i, int j, int k) const {
    return ((i + j + k) & 1) * half + (k * ny + j) * nxh + (i >> 1);
  }
};

// A run: planes k0 .. k1 - 1 of the column pair (2 i2, 2 i2 + 1, j).
struct CvRun {
  int i2, j, k0, k1;
  __device__ __forceinline__ void set(const CvLevel& V, int t) {
    int col;
    const int seg = cv_divmod(t, V.cols, col);
    j = cv_divmod(col, V.nxh, i2);
    k0 = seg * V.len;
    k1 = min(k0 + V.len, V.nz);
  }
};

// The level's runs of this thread, one after the other (one, except on a
// level with more column pairs than threads).
template <class F>
__device__ __forceinline__ void cv_runs(const CvLevel& V, F&& f) {
  for (int t = threadIdx.x; t < V.runs; t += V.n) {
    CvRun R;
    R.set(V, t);
    f(R);
  }
}

// The prolonged values that a run of column pairs takes from level W (below V,
// every axis halved): plane() forms those of coarse plane K interpolated in x (the
// wall factors included) on the even (v[0]) and odd column (v[1]) of the run's own
// coarse row, and of the row beside it (v[2], v[3]); child() sums the values of a
// fine plane's own coarse plane (c) and of the one beside it (n).
template <class T>
struct CvProlong {
  int i2, J, xl, xr, jn;
  T ma, fl, fr, fy;
  __device__ __forceinline__ CvProlong(const CvRun& R, const CvLevel& W, const Level& C) {
    ma = -lv_alpha<T>(C);
    i2 = R.i2;
    J = R.j >> 1;
    xl = outer_idx(i2 - 1, W.nx, C.per[0]);
    xr = outer_idx(i2 + 1, W.nx, C.per[0]);
    jn = outer_idx(J + ((R.j & 1) ? 1 : -1), W.ny, C.per[1]);
    fl = xl >= 0 ? (T)1 : ma;
    fr = xr >= 0 ? (T)1 : ma;
    fy = jn >= 0 ? (T)1 : ma;
    if (xl < 0) xl = i2;
    if (xr < 0) xr = i2;
    if (jn < 0) jn = J;
  }
  __device__ __forceinline__ void plane(const CvLevel& W, const Level& C, const T* we, int K, T v[4]) const {
    int kk = outer_idx(K, W.nz, C.per[2]);
    const T fz = kk >= 0 ? (T)1 : ma;
    if (kk < 0) kk = K < 0 ? 0 : W.nz - 1;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int jj = b ? jn : J;
      const T f = fz * (b ? fy : (T)1);
      const T* row = we + (kk * W.ny + jj) * W.nxh;
      const int sc = (i2 + jj + kk) & 1, hc = sc * W.half, hx = (1 - sc) * W.half;
      const T n0 = mul_t(f, row[hc + (i2 >> 1)]);
      v[2 * b] = prolong_pair(n0, mul_t(f * fl, row[((xl ^ i2) & 1 ? hx : hc) + (xl >> 1)]));
      v[2 * b + 1] = prolong_pair(n0, mul_t(f * fr, row[((xr ^ i2) & 1 ? hx : hc) + (xr >> 1)]));
    }
  }
  static __device__ __forceinline__ T child(const T c[4], const T n[4], int x) {
    return prolong_sum(c[x], c[2 + x], n[x], n[2 + x]);
  }
};

// `sweeps` red-black sweeps (from_zero: e is zero on entry and may hold
// anything), then (resid) the residual of both colours into the scratch.
// The neighbour sum, the wall count and the update are those of sum_nb and
// the per-colour sweep.
template <class T>
__device__ __forceinline__ void cv_passes(const CoarseCycle& CC, int l, const CvLevel& V, T* sm,
                                          int sweeps, T omega, bool from_zero, bool resid) {
  const Level& L = CC.lv[l];
  const T h2 = (T)CC.h2[l], c1 = (T)1 - omega, ih2 = lv_ih2<T>(L);
  const bool ax = L.act[0], ay = L.act[1], az = L.act[2];
  const bool px = L.per[0], py = L.per[1], pz = L.per[2];
  const int passes = 2 * sweeps + (resid ? 2 : 0), bar = 1 + l - CC.first;
  const bool once = V.runs <= V.n;
  CvRun R;
  bool hu = false, hd = false, hs0 = false, hs1 = false;
  int o = 0, du = 0, dd = 0, ds0 = 0, ds1 = 0, nw0 = 0, nw1 = 0, last1 = 0;
  T w0 = 0, w1 = 0;
  for (int pass = 0; pass < passes; ++pass) {
    const int c = pass & 1;
    const bool zero = from_zero && pass == 0, rs = pass >= 2 * sweeps;
    for (int t = threadIdx.x; t < V.runs; t += V.n) {
      if (pass == 0 || !once) {
        R.set(V, t);
        o = V.e + (R.k0 * V.ny + R.j) * V.nxh + R.i2;
        hu = ay && (py || R.j > 0);
        hd = ay && (py || R.j < V.ny - 1);
        du = R.j > 0 ? -V.nxh : (V.ny - 1) * V.nxh;
        dd = R.j < V.ny - 1 ? V.nxh : (1 - V.ny) * V.nxh;
        // beside the own index: left of an even column, right of an odd one
        hs0 = ax && (px || R.i2 > 0);
        hs1 = ax && (px || R.i2 < V.nxh - 1);
        ds0 = R.i2 > 0 ? -1 : V.nxh - 1;
        ds1 = R.i2 < V.nxh - 1 ? 1 : 1 - V.nxh;
        const int yw = ay && !py ? (R.j == 0) + (R.j == V.ny - 1) : 0;
        const bool xw = ax && !px;
        last1 = (V.nx & 1) && R.i2 == V.nxh - 1;   // the odd column lies beyond the wall
        nw0 = yw + (xw ? (R.i2 == 0) + last1 : 0);
        nw1 = yw + (xw ? R.i2 == V.nxh - 1 : 0);
        w0 = wscale(omega, lv_rc<T>(L, nw0));
        w1 = wscale(omega, lv_rc<T>(L, nw1));
      }
      T* own = sm + o + c * V.half;
      const T* oth = sm + o + (1 - c) * V.half;
      const T* rr = own + 2 * V.half;
      T* out = rs ? sm + CC.scratch + (o - V.e) + c * V.half : own;
      // zm, m, zp: the other colour's column below, at and above the plane
      T zm = 0, m = 0;
      if (!zero) {
        if (az && R.k0 > 0) zm = oth[-V.cols];
        else if (az && pz) zm = oth[(V.nz - 1 - R.k0) * V.cols];
        m = oth[0];
      }
      bool par = (R.j + R.k0 + c) & 1;
#pragma unroll 2
      for (int k = R.k0; k < R.k1; ++k) {
        const int q = (k - R.k0) * V.cols;
        T zp = 0, x = 0, u = 0, d = 0;
        if (!zero) {
          if (az && k < V.nz - 1) zp = oth[q + V.cols];
          else if (az && pz) zp = oth[q + (1 - V.nz) * V.cols];
          if (par ? hs1 : hs0) x = oth[q + (par ? ds1 : ds0)];
          if (hu) u = oth[q + du];
          if (hd) d = oth[q + dd];
        }
        const T mid = ax ? m : (T)0;
        const T s = ((mid + x) + (u + d)) + (zm + zp), b = rr[q];
        const T xo = from_zero && pass < 2 ? (T)0 : own[q];
        T w = par ? w1 : w0;
        int nw = par ? nw1 : nw0;
        if (az && !pz && (k == 0 || k == V.nz - 1)) {
          nw += (k == 0) + (k == V.nz - 1);
          w = wscale(omega, lv_rc<T>(L, nw));
        }
        const T v = rs ? resid_value(b, s, lv_coef<T>(L, nw), xo, ih2) : relax(xo, nb_term(s, b, h2), w, c1);
        // the spare cell of an odd row stays zero: it is the ghost beyond the wall
        out[q] = par && last1 ? (T)0 : v;
        zm = m;
        m = zp;
        par = !par;
      }
    }
    cv_sync(bar, V.n);
  }
}

// The visit of a level whose runs of LEN planes a thread holds in registers,
// both colours (values and rhs): of a cell's neighbours only the two in y, one
// in x and those at the run's ends are loads.  Cell q of colour c has column
// parity (p0 + q + c) & 1, p0 = (j + k0) & 1; what depends on it is kept by
// a = (q + c) & 1, so that every index is known at compile time.
template <class T, int LEN>
struct CvRegRun {
  T e[2][LEN], r[2][LEN];
  CvRun R;
  bool on, ok[2];        // the thread has a run; the column exists (odd extents have a spare cell)
  bool hs[2], hu, hd;    // neighbours present: x beside the own index, y - 1, y + 1
  int ds[2], du, dd;     // and their distances
  bool hlo, hhi;         // planes below and above the run
  int dlo, dhi;
  int o;                 // offset of the run's first cell in a colour
  T* p[2];               // and its place among the values of each colour
  bool mid;              // x couples
  int nw[2], zb, zt;     // wall neighbours without z; z walls at the run's first and last plane

  __device__ __forceinline__ CvRegRun(const Level& L, const CvLevel& V, T* sm) {
    on = (int)threadIdx.x < V.runs;
    R.set(V, on ? (int)threadIdx.x : 0);
    const bool ax = L.act[0], ay = L.act[1], az = L.act[2];
    const bool px = L.per[0], py = L.per[1], pz = L.per[2];
    o = (R.k0 * V.ny + R.j) * V.nxh + R.i2;
    p[0] = sm + V.e + o;
    p[1] = p[0] + V.half;
    mid = ax;
    const bool xw = ax && !px, spare = (V.nx & 1) && R.i2 == V.nxh - 1;
    const int yw = ay && !py ? (R.j == 0) + (R.j == V.ny - 1) : 0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const bool odd = (R.j + R.k0 + a) & 1;
      hs[a] = ax && (px || (odd ? R.i2 < V.nxh - 1 : R.i2 > 0));
      ds[a] = odd ? (R.i2 < V.nxh - 1 ? 1 : 1 - V.nxh) : (R.i2 > 0 ? -1 : V.nxh - 1);
      ok[a] = !(odd && spare);
      nw[a] = yw + (xw ? (odd ? R.i2 == V.nxh - 1 : (R.i2 == 0) + spare) : 0);
    }
    hu = ay && (py || R.j > 0);
    hd = ay && (py || R.j < V.ny - 1);
    du = R.j > 0 ? -V.nxh : (V.ny - 1) * V.nxh;
    dd = R.j < V.ny - 1 ? V.nxh : (1 - V.ny) * V.nxh;
    hlo = az && (pz || R.k0 > 0);
    hhi = az && (pz || R.k1 < V.nz);
    dlo = R.k0 > 0 ? -V.cols : (V.nz - 1) * V.cols;
    dhi = R.k1 < V.nz ? LEN * V.cols : -R.k0 * V.cols;
    zb = az && !pz && R.k0 == 0;
    zt = az && !pz && R.k1 == V.nz;
  }
  __device__ __forceinline__ int walls(int a, int q) const {
    return nw[a] + (q == 0 ? zb : 0) + (q == LEN - 1 ? zt : 0);
  }
  // rhs from shared memory, or that of the first level from global memory (g)
  __device__ __forceinline__ void load_r(const CvLevel& V, const T* __restrict__ g) {
#pragma unroll
    for (int q = 0; q < LEN; ++q) {
      T even = 0, odd = 0;
      if (g && on) {
        const T* s = g + ((R.k0 + q) * V.ny + R.j) * V.nx + 2 * R.i2;
        even = s[0];
        if (2 * R.i2 + 1 < V.nx) odd = s[1];
      }
      const bool par = (R.j + R.k0 + q) & 1;   // column parity of colour 0
      r[0][q] = g ? (par ? odd : even) : p[0][2 * V.half + q * V.cols];
      r[1][q] = g ? (par ? even : odd) : p[1][2 * V.half + q * V.cols];
    }
  }
  __device__ __forceinline__ void store_global(const CvLevel& V, T* __restrict__ g) const {
    if (!on) return;
#pragma unroll
    for (int q = 0; q < LEN; ++q) {
      T* d = g + ((R.k0 + q) * V.ny + R.j) * V.nx + 2 * R.i2;
      const bool par = (R.j + R.k0 + q) & 1;
      d[0] = par ? e[1][q] : e[0][q];
      if (2 * R.i2 + 1 < V.nx) d[1] = par ? e[0][q] : e[1][q];
    }
  }
  __device__ __forceinline__ void load_e(const CvLevel& V) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int q = 0; q < LEN; ++q) e[c][q] = p[c][q * V.cols];
  }
  // neighbour sums of colour c, ((x- + x+) + (y- + y+)) + (z- + z+)
  __device__ __forceinline__ void sums(const CvLevel& V, int c, T* s) const {
    const T* oth = p[1 - c];
    T lo = 0, hi = 0;
    if (hlo) lo = oth[dlo];
    if (hhi) hi = oth[dhi];
#pragma unroll
    for (int q = 0; q < LEN; ++q) {
      const T* at = oth + q * V.cols;
      T x = 0, u = 0, d = 0;
      if (hs[(q + c) & 1]) x = at[ds[(q + c) & 1]];
      if (hu) u = at[du];
      if (hd) d = at[dd];
      const T m = mid ? e[1 - c][q] : (T)0;
      const T zm = q > 0 ? e[1 - c][q > 0 ? q - 1 : 0] : lo;
      const T zp = q < LEN - 1 ? e[1 - c][q < LEN - 1 ? q + 1 : 0] : hi;
      s[q] = ((m + x) + (u + d)) + (zm + zp);
    }
  }
  // e += P e(W) of the run (every axis halved)
  __device__ __forceinline__ void prolong(const CvLevel& V, const CvLevel& W, const Level& C, const T* we) {
    if (!on) return;
    const CvProlong<T> I(R, W, C);
    auto plane = [&](int K, T v[4]) { I.plane(W, C, we, K, v); };
    auto add = [&](int q, const T c[4], const T n[4]) {
      const T v[2] = {I.child(c, n, 0), I.child(c, n, 1)};
      const bool par = (R.j + R.k0 + q) & 1;
      e[0][q] += par ? v[1] : v[0];
      e[1][q] += par ? v[0] : v[1];
      p[0][q * V.cols] = e[0][q];
      p[1][q * V.cols] = e[1][q];
    };
    const int K = R.k0 >> 1;
    T a[4], c[4], n[4];
    plane(K, c);
    if constexpr (LEN == 1) {
      plane(K + ((R.k0 & 1) ? 1 : -1), n);
      add(0, c, n);
    } else {
      plane(K - 1, a);
#pragma unroll
      for (int h = 0; h < LEN / 2; ++h) {
        plane(K + h + 1, n);
        add(2 * h, c, a);
        add(2 * h + 1, c, n);
#pragma unroll
        for (int x = 0; x < 4; ++x) { a[x] = c[x]; c[x] = n[x]; }
      }
    }
  }
};

// One visit of level l: down: `sweeps` sweeps from e = 0, then (resid) the
// residual into the scratch; up: e += P e(W) where every axis is halved
// (`blocked`; else it is already in e), then the sweeps; the first level's
// result also goes to global memory.
template <class T, int LEN>
__device__ __forceinline__ void cv_visit(const CoarseCycle& CC, int l, const CvLevel& V,
                                         const CvLevel& W, T* sm, const T* rr, T* e_out, int sweeps,
                                         T omega, bool down, bool resid, bool blocked) {
  const Level& L = CC.lv[l];
  const T h2 = (T)CC.h2[l], c1 = (T)1 - omega;
  const int bar = 1 + l - CC.first;
  constexpr bool kLast = LEN == 3 || LEN == 5;   // the coarsest level only: from zero, no residual
  CvRegRun<T, LEN> X(L, V, sm);
  X.load_r(V, l == CC.first ? rr : nullptr);
  if (down) {
#pragma unroll
    for (int q = 0; q < LEN; ++q) X.e[0][q] = X.e[1][q] = (T)0;
  } else {
    X.load_e(V);
    if constexpr (!kLast) {
      if (blocked) {
        X.prolong(V, W, CC.lv[l + 1], sm + W.e);
        cv_sync(bar, V.n);
      }
    }
  }
  T w[2][3];   // omega / diagonal: at the run's first plane, inside, at its last
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    w[a][0] = wscale(omega, lv_rc<T>(L, X.walls(a, 0)));
    w[a][1] = wscale(omega, lv_rc<T>(L, X.nw[a]));
    w[a][2] = wscale(omega, lv_rc<T>(L, X.walls(a, LEN - 1)));
  }
  T s[LEN];
#pragma unroll 1
  for (int it = 0; it < sweeps; ++it) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (X.on) {
        if (c == 0 && down && it == 0) {   // from zero: every neighbour is zero
#pragma unroll
          for (int q = 0; q < LEN; ++q) s[q] = (T)0;
        } else {
          X.sums(V, c, s);
        }
#pragma unroll
        for (int q = 0; q < LEN; ++q) {
          const int a = (q + c) & 1;
          if (X.ok[a]) {
            X.e[c][q] = relax(X.e[c][q], nb_term(s[q], X.r[c][q], h2),
                              w[a][q == 0 ? 0 : (q == LEN - 1 ? 2 : 1)], c1);
            X.p[c][q * V.cols] = X.e[c][q];
          }
        }
      }
      cv_sync(bar, V.n);
    }
  }
  if (kLast) return;
  if (resid) {
    if (X.on) {
      const T ih2 = lv_ih2<T>(L);
      T* const sc = sm + CC.scratch + X.o;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        X.sums(V, c, s);
#pragma unroll
        for (int q = 0; q < LEN; ++q)
          sc[c * V.half + q * V.cols] =
              resid_value(X.r[c][q], s[q], lv_coef<T>(L, X.walls((q + c) & 1, q)), X.e[c][q], ih2);
      }
    }
    cv_sync(bar, V.n);
  }
  if (!down && l == CC.first) X.store_global(V, e_out);
}

// The residuals in the scratch averaged onto the rhs of W, children in order.
template <class T>
__device__ __forceinline__ void cv_restrict(const CoarseCycle& CC, int l, const CvLevel& V,
                                            const CvLevel& W, T* sm) {
  const int nc = W.nx * W.ny * W.nz;
  const int fx = V.nx / W.nx, fy = V.ny / W.ny, fz = V.nz / W.nz;
  const T* S = sm + CC.scratch;
  for (int t = threadIdx.x; t < nc; t += V.n) {
    int I, J;
    const int K = cv_divmod(cv_divmod(t, W.nx, I), W.ny, J);
    T acc = 0;
    for (int dk = 0; dk < fz; ++dk)
      for (int dj = 0; dj < fy; ++dj)
        for (int di = 0; di < fx; ++di) acc += S[V.at(I * fx + di, J * fy + dj, K * fz + dk)];
    sm[W.r + W.at(I, J, K)] = acc / (T)(fx * fy * fz);
  }
  cv_sync(1 + l - CC.first, V.n);
}

// e(V) += P e(W)
template <class T>
__device__ __forceinline__ void cv_prolong(const CoarseCycle& CC, int l, const CvLevel& V,
                                           const CvLevel& W, T* sm) {
  const Level& F = CC.lv[l];
  const Level& C = CC.lv[l + 1];
  const T* we = sm + W.e;
  if (blocked_transfer_ok(F, C)) {   // the values of k_prolong_block
    cv_runs(V, [&](const CvRun& R) {
      const CvProlong<T> I(R, W, C);
      auto plane = [&](int K, T v[4]) { I.plane(W, C, we, K, v); };
      auto add = [&](int k, const T c[4], const T n[4]) {
        const T v[2] = {I.child(c, n, 0), I.child(c, n, 1)};
        T* e = sm + V.e + (k * V.ny + R.j) * V.nxh + R.i2;
        const int par = (R.j + k) & 1;   // the even column's colour
        e[par * V.half] += v[0];
        e[(1 - par) * V.half] += v[1];
      };
      // planes 2K and 2K + 1 from coarse planes K - 1, K and K, K + 1
      T a[4], c[4], n[4];
      int K = R.k0 >> 1;
      plane(K, c);
      if (!(R.k0 & 1)) plane(K - 1, a);
#pragma unroll 1
      for (int k = R.k0; k < R.k1; ++K) {
        if (!(k & 1)) add(k++, c, a);
        if (k < R.k1) {
          plane(K + 1, n);
          add(k++, c, n);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) { a[x] = c[x]; c[x] = n[x]; }
      }
    });
  } else {                             // as k_prolong_add
    const int nf = V.nx * V.ny * V.nz;
    const T al = lv_alpha<T>(C);
    for (int t = threadIdx.x; t < nf; t += V.n) {
      int i, j;
      const int k = cv_divmod(cv_divmod(t, V.nx, i), V.ny, j);
      const Interp1<T> ax = interp_axis<T>(i, F.n[0] / C.n[0], C.n[0], C.per[0], al);
      const Interp1<T> ay = interp_axis<T>(j, F.n[1] / C.n[1], C.n[1], C.per[1], al);
      const Interp1<T> az = interp_axis<T>(k, F.n[2] / C.n[2], C.n[2], C.per[2], al);
      T acc = 0;
      for (int c2 = 0; c2 < 2; ++c2)
        for (int b2 = 0; b2 < 2; ++b2)
          for (int a2 = 0; a2 < 2; ++a2) {
            const T w = ax.w[a2] * ay.w[b2] * az.w[c2];
            if (w != (T)0) acc += w * we[W.at(ax.idx[a2], ay.idx[b2], az.idx[c2])];
          }
      sm[V.e + V.at(i, j, k)] += acc;
    }
  }
  cv_sync(1 + l - CC.first, V.n);
}

// The lower V-cycle of one component in one CTA: rhs rr (level CC.first,
// global memory) -> correction e_out, every level in shared memory `sm`.
// MAX_LEN: the longest run whose registers fit.
template <class T, int MAX_LEN>
__device__ __forceinline__ void coarse_vcycle_cta(const CoarseCycle& CC, const T* __restrict__ rr,
                                                  T* __restrict__ e_out, T* sm) {
  const int f = CC.first, l_last = CC.last, tid = threadIdx.x;
  if (!CC.reg[f]) {   // the loop reads its rhs from shared memory
    const CvLevel V(CC, f);
    if (tid < V.n)
      cv_runs(V, [&](const CvRun& R) {
        for (int k = R.k0; k < R.k1; ++k) {
          const T* p = rr + (k * V.ny + R.j) * V.nx + 2 * R.i2;
          T* r = sm + V.r + (k * V.ny + R.j) * V.nxh + R.i2;
          const int par = (R.j + k) & 1;   // the even column's colour
          r[par * V.half] = p[0];
          if (2 * R.i2 + 1 < V.nx) r[(1 - par) * V.half] = p[1];
        }
      });
    __syncthreads();
  }
  // down to the last level this thread works on, then back up; where a level
  // has fewer threads the others wait at the barrier of the level above
  bool down = true;
  int l = tid < CC.threads[f] ? f : f - 1;
  while (l >= f) {
    const CvLevel V(CC, l);
    const bool last = l == l_last;
    const CvLevel W(CC, last ? l : l + 1);
    const bool blocked = !last && blocked_transfer_ok(CC.lv[l], CC.lv[l + 1]);
    if (!down) {
      cv_sync(1 + l - f, V.n);   // the levels below are done
      if (!V.reg || !blocked) cv_prolong<T>(CC, l, V, W, sm);
    }
    const int sweeps = last ? CC.coarse_sweeps : (down ? CC.nu1 : CC.nu2);
    const T om = last ? (T)1 : (T)CC.omega;
    const bool rs = down && !last;
    if (down && sweeps == 0) {   // no pre-smoothing: e = 0 has to be there
      for (int t = tid; t < 2 * V.half; t += V.n) sm[V.e + t] = (T)0;
      cv_sync(1 + l - f, V.n);
    }
    if (!V.reg) cv_passes<T>(CC, l, V, sm, sweeps, om, down, rs);
    else if (V.len == 1) cv_visit<T, 1>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    else if (V.len == 2) cv_visit<T, 2>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    else if (V.len == 4) cv_visit<T, 4>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    else if (V.len == 3) cv_visit<T, 3>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    else if (V.len == 5) cv_visit<T, 5>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    else cv_visit<T, MAX_LEN>(CC, l, V, W, sm, rr, e_out, sweeps, om, down, rs, blocked);
    if (rs) {
      cv_restrict<T>(CC, l, V, W, sm);
      if (tid < W.n) ++l;
      else down = false;          // waits at the top of the loop for the levels below
    } else {
      down = false;
      --l;
    }
  }
  if (CC.reg[f] && f < l_last) return;   // stored from the runs
  __syncthreads();
  const CvLevel V(CC, f);
  if (tid < V.n)
    cv_runs(V, [&](const CvRun& R) {
      for (int k = R.k0; k < R.k1; ++k) {
        T* p = e_out + (k * V.ny + R.j) * V.nx + 2 * R.i2;
        const T* e = sm + V.e + (k * V.ny + R.j) * V.nxh + R.i2;
        const int par = (R.j + k) & 1;
        p[0] = e[par * V.half];
        if (2 * R.i2 + 1 < V.nx) p[1] = e[(1 - par) * V.half];
      }
    });
}

// kCvThreads = 512: registers for runs of eight planes in FP32, four in FP64.

template <class T>
__global__ void __launch_bounds__(kCvThreads)
k_coarse_vcycle(const __grid_constant__ CoarseCycle CC, Comp3<T> E, Comp3<T> RR) {
  pdl_begin();
  extern __shared__ unsigned char smem_cv[];
  const int comp = blockIdx.x;
  coarse_vcycle_cta<T, sizeof(T) == 4 ? 8 : 4>(CC, RR.at(comp), E.at(comp), reinterpret_cast<T*>(smem_cv));
}

template <class T>
bool launch_coarse_vcycle(Ctx& cx, const CoarseCycle& CC, Comp3<T> E, Comp3<T> R, int ncomp) {
  const size_t smem = (size_t)CC.total * sizeof(T);
  if (smem > kCoarseCycleSmem) return false;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(k_coarse_vcycle<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return false;
  cx.before(VSV_KCLASS_SMOOTH);
  launch_k(cx, k_coarse_vcycle<T>, ncomp, kCvThreads, smem, CC, E, R);
  // r of the first level read, e written; the rest stays in shared memory
  cx.after(VSV_KCLASS_SMOOTH, 2.0 * (double)sizeof(T) * (double)CC.lv[CC.first].cells() * ncomp);
  return true;
}

// ---------------------------------------------------------------- persistent lower V-cycle
// The levels below the finest fit in L2 and are bound by launch and
// barrier latency when run level by level (dozens of launches of a few to
// tens of microseconds each per V-cycle).  One cooperative launch runs them
// instead: every CTA of the grid (all co-resident) sweeps, restricts and
// prolongs levels first .. cc-1 with grid-stride loops, separated by grid
// barriers, and the levels cc .. last run as the one-CTA coarse cycle above
// (CTAs 0 .. ncomp-1, one component each) while the others wait.  Every
// operation is the per-colour reference kernels' arithmetic (sum_nb, relax,
// resid_plain, prolong_children / interp_axis), so the result is bit for
// bit that of the level-by-level V-cycle.

// Cells (a, j, k, comp) of a [ncomp][nz][ny][na] index space visited by a
// grid-stride loop: the flat index advances by the total thread count with
// carries instead of divisions.
struct StrideWalk {
  int a, j, k, c;
  int sa, sj, sk, sc;
  int na, ny, nz;
  __device__ __forceinline__ void init(long long t0, long long stride, int na_, int ny_, int nz_) {
    na = na_; ny = ny_; nz = nz_;
    long long q = t0;
    a = (int)(q % na); q /= na; j = (int)(q % ny); q /= ny; k = (int)(q % nz); c = (int)(q / nz);
    q = stride;
    sa = (int)(q % na); q /= na; sj = (int)(q % ny); q /= ny; sk = (int)(q % nz);
    sc = (int)(q / nz);
  }
  __device__ __forceinline__ void next() {
    a += sa;
    int cj = sj;
    if (a >= na) { a -= na; ++cj; }
    j += cj;
    int ck = sk;
    if (j >= ny) { j -= ny; ++ck; }
    k += ck;
    int cc = sc;
    if (k >= nz) { k -= nz; ++cc; }
    c += cc;
  }
};

// Bounded grid barrier (see GridBarrier).  Arrivals count up monotonically
// from zero (the host zeroes the counter before each launch), so barrier n
// waits until n * (gridDim.x + extra) arrivals.  Returns false when the
// wait ran out (bit kSyncTimeout of *status set, by this CTA or another);
// the caller then leaves the kernel.
__device__ __forceinline__ bool grid_sync(const GridBarrier& B, unsigned& epoch) {
  __shared__ int ok_s;
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();                                    // publish this CTA's writes
    atomicAdd(B.count, 1u);
    const unsigned target = epoch * (gridDim.x + B.extra);
    const volatile unsigned* vc = B.count;
    const volatile int* vs = B.status;
    const unsigned long long t0 = global_ns();
    while (*vc < target) {
      if (*vs & kSyncTimeout) { ok = 0; break; }
      if (global_ns() - t0 > B.limit_ns) {
        atomicOr(B.status, kSyncTimeout);
        ok = 0;
        break;
      }
      __nanosleep(32);
    }
    __threadfence();                                    // see the other CTAs' writes
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

// Number of Dirichlet ghosts among the 7-point neighbours of (i, j, k).
__device__ __forceinline__ int wall_count(const Level& L, int i, int j, int k) {
  int n = 0;
  if (L.act[0] && !L.per[0]) n += (i == 0) + (i == L.n[0] - 1);
  if (L.act[1] && !L.per[1]) n += (j == 0) + (j == L.n[1] - 1);
  if (L.act[2] && !L.per[2]) n += (k == 0) + (k == L.n[2] - 1);
  return n;
}

// One colour of a red-black sweep of level l, every component.  first:
// e is not yet initialised (a correction from zero): the red cells take
// their value from the rhs alone and the black cells are set to zero, as
// zeroing e and sweeping its red cells does.
template <class T>
__device__ void lc_sweep(const LowerCycle<T>& P, int l, int color, bool first, T omega) {
  const Level& L = P.lv[l];
  const int nx = L.n[0], nxh = (nx + 1) >> 1;
  const T h2 = (T)P.h2[l];
  StrideWalk w;
  w.init((long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, nxh,
         L.n[1], L.n[2]);
  for (; w.c < P.ncomp; w.next()) {
    T* __restrict__ x = P.e[l][w.c];
    const T* __restrict__ b = P.r[l][w.c];
    const int red = 2 * w.a + ((w.j + w.k + color) & 1);
    const long long row = lin(0, w.j, w.k, nx, L.n[1]);
    if (first) {
      // color is 0 here: the pair (2a, 2a + 1) holds one red and one black cell
      const int blk = red ^ 1;
      if (red < nx) {
        const long long c = row + red;
        x[c] = relax((T)0, nb_term((T)0, b[c], h2),
                     wscale(omega, lv_rc<T>(L, wall_count(L, red, w.j, w.k))), (T)1 - omega);
      }
      if (blk < nx) x[row + blk] = (T)0;
      continue;
    }
    if (red >= nx) continue;
    const long long c = row + red;
    int nwall;
    const T sn = sum_nb(x, L, red, w.j, w.k, c, nwall);
    x[c] = relax(x[c], nb_term(sn, b[c], h2), wscale(omega, lv_rc<T>(L, nwall)), (T)1 - omega);
  }
}

// Residual of level l restricted to level l + 1 (as k_resid_restrict).
template <class T>
__device__ void lc_restrict(const LowerCycle<T>& P, int l) {
  const Level& F = P.lv[l];
  const Level& C = P.lv[l + 1];
  const int fx = F.n[0] / C.n[0], fy = F.n[1] / C.n[1], fz = F.n[2] / C.n[2];
  StrideWalk w;
  w.init((long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x,
         C.n[0], C.n[1], C.n[2]);
  for (; w.c < P.ncomp; w.next()) {
    const T* __restrict__ x = P.e[l][w.c];
    const T* __restrict__ b = P.r[l][w.c];
    T acc = 0;
    for (int dk = 0; dk < fz; ++dk)
      for (int dj = 0; dj < fy; ++dj)
        for (int di = 0; di < fx; ++di) {
          const int i = w.a * fx + di, j = w.j * fy + dj, k = w.k * fz + dk;
          const long long c = lin(i, j, k, F.n[0], F.n[1]);
          acc += resid_plain(x, F, i, j, k, c, b[c]);
        }
    P.r[l + 1][w.c][lin(w.a, w.j, w.k, C.n[0], C.n[1])] = acc / (T)(fx * fy * fz);
  }
}

// e(l) += P e(l + 1) (as k_prolong_block, or k_prolong_add where an axis
// is not coarsened).
template <class T>
__device__ void lc_prolong(const LowerCycle<T>& P, int l) {
  const Level& F = P.lv[l];
  const Level& C = P.lv[l + 1];
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  StrideWalk w;
  if (blocked_transfer_ok(F, C)) {
    w.init(t0, stride, C.n[0], C.n[1], C.n[2]);
    for (; w.c < P.ncomp; w.next()) {
      T v[2][2][2];
      prolong_children<T>(C, P.e[l + 1][w.c], w.a, w.j, w.k, v);
      T* __restrict__ x = P.e[l][w.c];
      for (int c = 0; c < 2; ++c)
        for (int b = 0; b < 2; ++b) {
          T* p = x + ((long long)(2 * w.k + c) * F.n[1] + 2 * w.j + b) * F.n[0] + 2 * w.a;
          p[0] += v[c][b][0];
          p[1] += v[c][b][1];
        }
    }
    return;
  }
  const T al = lv_alpha<T>(C);
  w.init(t0, stride, F.n[0], F.n[1], F.n[2]);
  for (; w.c < P.ncomp; w.next()) {
    const Interp1<T> ax = interp_axis<T>(w.a, F.n[0] / C.n[0], C.n[0], C.per[0], al);
    const Interp1<T> ay = interp_axis<T>(w.j, F.n[1] / C.n[1], C.n[1], C.per[1], al);
    const Interp1<T> az = interp_axis<T>(w.k, F.n[2] / C.n[2], C.n[2], C.per[2], al);
    const T* __restrict__ ec = P.e[l + 1][w.c];
    T acc = 0;
    for (int c2 = 0; c2 < 2; ++c2)
      for (int b2 = 0; b2 < 2; ++b2)
        for (int a2 = 0; a2 < 2; ++a2) {
          const T wt = ax.w[a2] * ay.w[b2] * az.w[c2];
          if (wt != (T)0) acc += wt * ec[lin(ax.idx[a2], ay.idx[b2], az.idx[c2], C.n[0], C.n[1])];
        }
    P.e[l][w.c][lin(w.a, w.j, w.k, F.n[0], F.n[1])] += acc;
  }
}

// e(l) = 0 (a correction from zero that takes no pre-smoothing sweep).
template <class T>
__device__ void lc_zero(const LowerCycle<T>& P, int l) {
  const Level& L = P.lv[l];
  StrideWalk w;
  w.init((long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x,
         L.n[0], L.n[1], L.n[2]);
  for (; w.c < P.ncomp; w.next()) P.e[l][w.c][lin(w.a, w.j, w.k, L.n[0], L.n[1])] = (T)0;
}

template <class T>
__global__ void __launch_bounds__(1024)
k_lower_vcycle(const __grid_constant__ LowerCycle<T> P) {
  extern __shared__ unsigned char smem_lc[];
  unsigned epoch = 0;
  const T om = (T)P.omega;
  auto sweeps = [&](int l, int nu, bool from_zero) -> bool {
    if (nu == 0 && from_zero) {
      lc_zero<T>(P, l);
      return grid_sync(P.bar, epoch);
    }
    for (int s = 0; s < nu; ++s)
      for (int color = 0; color < 2; ++color) {
        lc_sweep<T>(P, l, color, from_zero && s == 0 && color == 0, om);
        if (!grid_sync(P.bar, epoch)) return false;
      }
    return true;
  };
  const int lw = P.cc;   // first level of the one-CTA part (last + 1: none)
  for (int l = P.first; l < lw; ++l) {
    if (l == P.last) {   // coarsest level solved grid-wide: plain Gauss-Seidel from zero
      for (int s = 0; s < P.coarse_sweeps; ++s)
        for (int color = 0; color < 2; ++color) {
          lc_sweep<T>(P, l, color, s == 0 && color == 0, (T)1);
          if (!grid_sync(P.bar, epoch)) return;
        }
      break;
    }
    if (!sweeps(l, P.nu1, true)) return;
    lc_restrict<T>(P, l);
    if (!grid_sync(P.bar, epoch)) return;
  }
  if (lw <= P.last) {
    if (blockIdx.x < (unsigned)P.ncomp)
      coarse_vcycle_cta<T, sizeof(T) == 4 ? 8 : 4>(P.cc_plan, P.r[lw][blockIdx.x], P.e[lw][blockIdx.x],
                           reinterpret_cast<T*>(smem_lc));
    if (!grid_sync(P.bar, epoch)) return;
  }
  for (int l = min(lw, P.last) - 1; l >= P.first; --l) {
    lc_prolong<T>(P, l);
    if (!grid_sync(P.bar, epoch)) return;
    if (!sweeps(l, P.nu2, false)) return;
  }
}

// The barrier alone, for tests of its bound: `rounds` barriers of a grid
// that expects `extra` arrivals more per barrier than it has CTAs (extra > 0
// means the wait can only end by running out).
__global__ void k_barrier_probe(GridBarrier B, int rounds) {
  unsigned epoch = 0;
  for (int r = 0; r < rounds; ++r)
    if (!grid_sync(B, epoch)) return;
}

template <class T>
int lower_cycle_blocks(int sms, size_t smem) {
  int per_sm = 0;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(k_lower_vcycle<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lower_vcycle<T>, 1024, smem) !=
      cudaSuccess)
    return 0;
  return per_sm * sms;
}

template <class T>
bool launch_lower_vcycle(Ctx& cx, const LowerCycle<T>& P) {
  const size_t smem = P.cc <= P.last ? (size_t)P.cc_plan.total * sizeof(T) : 0;
  if (smem > kCoarseCycleSmem) return false;
  const int nb = lower_cycle_blocks<T>(cx.sms, smem);
  if (nb < P.ncomp || nb < 1) return false;
  if (cudaMemsetAsync(P.bar.count, 0, sizeof(unsigned), cx.stream) != cudaSuccess) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nb);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = cx.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // all CTAs co-resident, or no launch
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cx.before(VSV_KCLASS_SMOOTH);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_lower_vcycle<T>, P);
  // r of the first level read, e written; the lower levels stay in L2
  cx.after(VSV_KCLASS_SMOOTH, 2.0 * (double)sizeof(T) * (double)P.lv[P.first].cells() * P.ncomp);
  return e == cudaSuccess;
}

int barrier_probe_max_blocks(int sms) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_barrier_probe, 128, 0) != cudaSuccess)
    return 0;
  return per_sm * sms;
}

bool launch_barrier_probe(cudaStream_t s, GridBarrier B, int blocks, int rounds) {
  if (cudaMemsetAsync(B.count, 0, sizeof(unsigned), s) != cudaSuccess) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_barrier_probe, B, rounds) == cudaSuccess;
}

// ---------------------------------------------------------------- launchers
static inline unsigned blocks_for(long long n) { return (unsigned)((n + kBlock - 1) / kBlock); }

template <class T>
static SweepGeom<T> sweep_geom(const Level& L, const Rhs3<T>& R, double omega, double h2) {
  SweepGeom<T> G;
  G.nx = L.n[0]; G.ny = L.n[1]; G.nz = L.n[2];
  for (int a = 0; a < 3; ++a) {
    G.act[a] = L.act[a];
    G.per[a] = L.per[a];
  }
  const T om = (T)omega;
  for (int q = 0; q < 7; ++q) G.w[q] = om * lv_rc<T>(L, q);
  G.h2 = (T)h2;
  G.c1 = (T)1 - om;
  G.beta = R.beta;
  return G;
}

template <class T>
void launch_rb_sweep(Ctx& cx, const Level& L, Comp3<T> X, Rhs3<T> R, int ncomp, int color,
                     double omega, double h2, int kclass, bool zero) {
  const dim3 grid = grid3((L.n[0] + 1) / 2, L.n[1], L.n[2], ncomp);
  SweepGeom<T> G = sweep_geom<T>(L, R, omega, h2);
  bool plane = false;
  for (int q = 0; q < ncomp; ++q) plane = plane || R.S[q];
  if (!plane) G.h2 *= R.beta;
  auto kern = plane ? (zero ? k_rb_sweep<T, true, true> : k_rb_sweep<T, false, true>)
                    : (zero ? k_rb_sweep<T, true, false> : k_rb_sweep<T, false, false>);
  cx.before(kclass);
  launch_k(cx, kern, grid, block3(), 0, G, X, R, color);
  // one colour: the other colour's values and this colour's rhs read, this colour written
  // (and read, for SOR): 1.5 words per cell; from zero this colour's rhs read, both written
  cx.after(kclass, (zero || omega == 1.0 ? 1.5 : 2.0) * (double)sizeof(T) * (double)L.cells() * ncomp);
}

template <class T>
void launch_resid_restrict(Ctx& cx, const Level& F, const Level& C, Comp3<T> X, Rhs3<T> R,
                           Comp3<T> RC, int ncomp, bool exact) {
  const dim3 grid = grid3(C.n[0], C.n[1], C.n[2], ncomp);
  if constexpr (std::is_same<T, float>::value) {
    if (!exact && cx.tiled && launch_restrict_tiled(cx, F, C, X, R, RC, ncomp)) return;
  }
  if (!exact && blocked_transfer_ok(F, C)) {
    cx.before(VSV_KCLASS_RESTRICT);
    launch_k(cx, k_restrict_block<T>, grid, block3(), 0, F, C, X, R, RC);
    cx.after(VSV_KCLASS_RESTRICT, 2.125 * (double)sizeof(T) * (double)F.cells() * ncomp);
    return;
  }
  cx.before(VSV_KCLASS_RESTRICT);
  float ih_hi = (float)F.inv_h2, ih_lo = (float)(F.inv_h2 - (double)ih_hi);
  if constexpr (std::is_same<T, float>::value) {
    if (exact)
      launch_k(cx, k_resid_restrict<float, true>, grid, block3(), 0, F, C, X, R, RC, ih_hi, ih_lo);
    else
      launch_k(cx, k_resid_restrict<float, false>, grid, block3(), 0, F, C, X, R, RC, ih_hi, ih_lo);
  } else {
    launch_k(cx, k_resid_restrict<T, false>, grid, block3(), 0, F, C, X, R, RC, ih_hi, ih_lo);
  }
  cx.after(VSV_KCLASS_RESTRICT, (2.0 * (double)F.cells() + (double)C.cells()) * (double)sizeof(T) * ncomp);
}

template <class T>
void launch_prolong_add(Ctx& cx, const Level& F, const Level& C, Comp3<T> X, Comp3<T> E, int ncomp) {
  if constexpr (std::is_same<T, float>::value) {
    if (cx.tiled && launch_prolong_tiled(cx, F, C, X, E, ncomp)) return;
  }
  if (blocked_transfer_ok(F, C)) {
    cx.before(VSV_KCLASS_PROLONG);
    launch_k(cx, k_prolong_block<T>, grid3(C.n[0], C.n[1], C.n[2], ncomp), block3(), 0, F, C, X, E);
    cx.after(VSV_KCLASS_PROLONG, 2.125 * (double)sizeof(T) * (double)F.cells() * ncomp);
    return;
  }
  const dim3 grid = grid3(F.n[0], F.n[1], F.n[2], ncomp);
  cx.before(VSV_KCLASS_PROLONG);
  launch_k(cx, k_prolong_add<T>, grid, block3(), 0, F, C, X, E);
  cx.after(VSV_KCLASS_PROLONG, (2.0 * (double)F.cells() + (double)C.cells()) * (double)sizeof(T) * ncomp);
}

template <class T>
void launch_zero(Ctx& cx, Comp3<T> X, long long n, int ncomp) {
  dim3 grid(blocks_for(n), ncomp);
  cx.before(-1);
  launch_k(cx, k_zero<T>, grid, kBlock, 0, X, n);
  cx.after(-1, (double)sizeof(T) * (double)n * ncomp);
}

template <class T>
void launch_extrapolate_rot(Ctx& cx, Comp3<T> A, Comp3<T> B, Comp3<T> C, long long n, int ncomp,
                            int order) {
  const long long b = std::min<long long>(blocks_for(n), 4LL * cx.sms);
  dim3 grid((unsigned)b, ncomp);
  cx.before(-1);
  launch_k(cx, k_extrapolate_rot<T>, grid, kBlock, 0, A, B, C, n, order);
  // the history words read (A; A, B; A, B, C), the guess written
  cx.after(-1, (double)(order + 2) * (double)sizeof(T) * (double)n * ncomp);
}

template <class T>
void launch_axpy(Ctx& cx, Comp3<T> Y, Comp3<T> X, double a, long long n, int ncomp) {
  const long long b = std::min<long long>(blocks_for(n), 4LL * cx.sms);
  dim3 grid((unsigned)b, ncomp);
  cx.before(-1);
  launch_k(cx, k_axpy<T>, grid, kBlock, 0, Y, X, (T)a, n);
  cx.after(-1, 3.0 * (double)sizeof(T) * (double)n * ncomp);
}

template <class T>
bool launch_coarse_solve(Ctx& cx, const Level& L, Comp3<T> E, Comp3<T> R, int ncomp, int sweeps,
                         double h2) {
  const long long n = L.cells();
  const size_t smem = (size_t)n * 2 * sizeof(T);
  if (smem > 96 * 1024) return false;
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(k_coarse_solve<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  dim3 grid(1, ncomp);
  cx.before(VSV_KCLASS_SMOOTH);
  launch_k(cx, k_coarse_solve<T>, grid, 512, smem, L, E, R, sweeps, (T)h2);
  cx.after(VSV_KCLASS_SMOOTH, 2.0 * (double)sizeof(T) * (double)n * ncomp);
  return true;
}

template <class T>
void launch_resid_norm(Ctx& cx, const Level& L, Comp3<T> X, Rhs3<T> R, int ncomp, bool exact,
                       double* partials, int nblocks, Scalars* S, double* host) {
  dim3 grid(row_blocks(L, nblocks), ncomp);
  float ih_hi = (float)L.inv_h2, ih_lo = (float)(L.inv_h2 - (double)ih_hi);
  cx.before(-1);
  if constexpr (std::is_same<T, float>::value) {
    if (exact)
      launch_k(cx, k_resid_norm<float, true>, grid, kBlock, 0, L, X, R, partials, ih_hi, ih_lo, S, host);
    else
      launch_k(cx, k_resid_norm<float, false>, grid, kBlock, 0, L, X, R, partials, ih_hi, ih_lo, S, host);
  } else {
    launch_k(cx, k_resid_norm<T, false>, grid, kBlock, 0, L, X, R, partials, ih_hi, ih_lo, S, host);
  }
  cx.after(-1);
}

#define VSV_INST(T)                                                                                \
  template void launch_rb_sweep<T>(Ctx&, const Level&, Comp3<T>, Rhs3<T>, int, int, double, double, \
                                   int, bool);                                                     \
  template void launch_resid_restrict<T>(Ctx&, const Level&, const Level&, Comp3<T>, Rhs3<T>,      \
                                         Comp3<T>, int, bool);                                     \
  template void launch_prolong_add<T>(Ctx&, const Level&, const Level&, Comp3<T>, Comp3<T>, int);  \
  template void launch_zero<T>(Ctx&, Comp3<T>, long long, int);                                    \
  template void launch_axpy<T>(Ctx&, Comp3<T>, Comp3<T>, double, long long, int);                  \
  template void launch_extrapolate_rot<T>(Ctx&, Comp3<T>, Comp3<T>, Comp3<T>, long long, int, int); \
  template bool launch_coarse_vcycle<T>(Ctx&, const CoarseCycle&, Comp3<T>, Comp3<T>, int);        \
  template bool launch_lower_vcycle<T>(Ctx&, const LowerCycle<T>&);                                \
  template bool launch_coarse_solve<T>(Ctx&, const Level&, Comp3<T>, Comp3<T>, int, int, double);  \
  template void launch_resid_norm<T>(Ctx&, const Level&, Comp3<T>, Rhs3<T>, int, bool, double*,    \
                                     int, Scalars*, double*);
VSV_INST(float)
VSV_INST(double)
#undef VSV_INST

}  // namespace vsv
