// Phase-field kernels: explicit phi update (eq. gen2), chemical potentials
// (eq. 31 Cahn-Hilliard; eq. 30 / SM eq. 35 Helfrich), vorticity source
// (eq. gen1), volume / area reductions (SM eqs. 32, 37-38), velocity
// v = curl psi (eq. vecpot), the observables of the in-plane-shear and
// results sections, and the FP64 base-flow tables of the channel flows
// (boundary-conditions section).
//
// Fields are [nz][ny][nx] without halos.  Scalars (phi, mu, g) use the
// face mirror at walls and wrap on periodic axes; the flow perturbation
// psi' = psi - psi0 is zero on the wall nodes.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "internal.h"

namespace vsv {

__device__ __forceinline__ int mirror_idx(int j, int n) {
  return j < 0 ? -1 - j : (j >= n ? 2 * n - 1 - j : j);
}
__device__ __forceinline__ int wrap_idx(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <class T>
struct ScalarView {  // periodic x, mirror y, mirror / periodic z
  const T* __restrict__ a;
  int nx, ny, nz, zper;
  __device__ __forceinline__ T operator()(int i, int j, int k) const {
    i = wrap_idx(i, nx);
    j = mirror_idx(j, ny);
    k = zper ? wrap_idx(k, nz) : mirror_idx(k, nz);
    return a[lin(i, j, k, nx, ny)];
  }
};

template <class T>
struct PertView {  // periodic x, zero on the wall nodes
  const T* __restrict__ a;
  int nx, ny, nz, zper;
  __device__ __forceinline__ T operator()(int i, int j, int k) const {
    i = wrap_idx(i, nx);
    if (zper) k = wrap_idx(k, nz);
    if (j < 0 || j >= ny || k < 0 || k >= nz) return (T)0;
    return a[lin(i, j, k, nx, ny)];
  }
};

template <class T, class V>
__device__ __forceinline__ T lap7(const V& f, int i, int j, int k, T ih2) {
  return (f(i + 1, j, k) + f(i - 1, j, k) + f(i, j + 1, k) + f(i, j - 1, k) + f(i, j, k + 1) +
          f(i, j, k - 1) - (T)6 * f(i, j, k)) * ih2;
}

__device__ __forceinline__ void cell_of(long long t, int nx, int ny, int& i, int& j, int& k) {
  i = (int)(t % nx);
  const long long q = t / nx;
  j = (int)(q % ny);
  k = (int)(q / ny);
}

template <class T> __device__ __forceinline__ T sc_lambda(const Scalars* S);
template <> __device__ __forceinline__ float sc_lambda<float>(const Scalars* S) { return S->lambda_vf; }
template <> __device__ __forceinline__ double sc_lambda<double>(const Scalars* S) { return S->lambda_v; }
template <class T> __device__ __forceinline__ T sc_gamma(const Scalars* S);
template <> __device__ __forceinline__ float sc_gamma<float>(const Scalars* S) { return S->gamma_af; }
template <> __device__ __forceinline__ double sc_gamma<double>(const Scalars* S) { return S->gamma_a; }

static inline unsigned nblk(long long n) { return (unsigned)((n + kBlock - 1) / kBlock); }

// ---------------------------------------------------------------- phi update (eq. gen2)
// phi^{n+1} = phi^n + dt [ M (lap mu + lambda_V) - v . grad phi ],
// v = v0(y, z) + curl psi' (central differences).
template <class T>
__global__ void k_phi_update(PhaseParams P, const T* __restrict__ phi, const T* __restrict__ mu,
                             Comp3<T> psi, Comp3<T> v0, Scalars* S, T dt, T* __restrict__ out) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const T ih2 = (T)P.inv_h2, hih = (T)(0.5 * P.inv_h);
  ScalarView<T> M{mu, P.nx, P.ny, P.nz, P.zper};
  ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
  PertView<T> X{psi.p[0], P.nx, P.ny, P.nz, P.zper};
  PertView<T> Y{psi.p[1], P.nx, P.ny, P.nz, P.zper};
  PertView<T> Z{psi.p[2], P.nx, P.ny, P.nz, P.zper};
  const T lmu = lap7<T>(M, i, j, k, ih2);
  const T gx = (F(i + 1, j, k) - F(i - 1, j, k)) * hih;
  const T gy = (F(i, j + 1, k) - F(i, j - 1, k)) * hih;
  const T gz = (F(i, j, k + 1) - F(i, j, k - 1)) * hih;
  const long long jk = j + (long long)k * P.ny;
  const T vx = v0.p[0][jk] + ((Z(i, j + 1, k) - Z(i, j - 1, k)) - (Y(i, j, k + 1) - Y(i, j, k - 1))) * hih;
  const T vy = v0.p[1][jk] + ((X(i, j, k + 1) - X(i, j, k - 1)) - (Z(i + 1, j, k) - Z(i - 1, j, k))) * hih;
  const T vz = v0.p[2][jk] + ((Y(i + 1, j, k) - Y(i - 1, j, k)) - (X(i, j + 1, k) - X(i, j - 1, k))) * hih;
  const T rate = (T)P.mobility * (lmu + sc_lambda<T>(S)) - (vx * gx + vy * gy + vz * gz);
  const T v = phi[t] + dt * rate;
  out[t] = v;
  if (!isfinite(v)) atomicOr(&S->nonfinite, 1);
}

// ---------------------------------------------------------------- reductions (SM eqs. 32, 37)
// V, A and the penalty multipliers lambda_V = K_V (V - V0), gamma_A = K_A (A -
// A0) 3 eps / (2 sqrt 2), by the last CTA of the reduction (15.8 + 7.2 -> 14.4 us at
// 128 x 64 x 64 against a kernel of its own and CTAs without rows).
__device__ __forceinline__ void va_publish(double sphi, double sarea, double* buf, double* partials,
                                           long long ncells, Scalars* S, int init) {
  if (!grid_sums(sphi, sarea, buf, partials, gridDim.x, 1, 0, blockIdx.x, S)) return;
  if (threadIdx.x == 0) {
    const double V = 0.5 * S->h3 * ((double)ncells - buf[0]);
    const double A = S->h3 * buf[1];
    S->V = V;
    S->A = A;
    if (init) {
      S->V0 = V;
      S->A0 = A;
    }
    S->lambda_v = S->k_vol * (V - S->V0);
    S->gamma_a = S->k_area * (A - S->A0) * 3.0 * S->eps / (2.0 * 1.4142135623730951);
    S->lambda_vf = (float)S->lambda_v;
    S->gamma_af = (float)S->gamma_a;
  }
}

// Per-block partial sums of sum(phi) and of the area density
// 3/(2 sqrt2) [eps/2 |grad phi|^2 + (phi^2 - 1)^2 / (4 eps)].
template <class T>
__global__ void k_reduce_va(PhaseParams P, const T* __restrict__ phi, const T* __restrict__ phi_lo,
                            double* partials, Scalars* S, int init) {
  ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
  const T hih = (T)(0.5 * P.inv_h);
  const T c_a = (T)(3.0 / (2.0 * 1.4142135623730951));
  const T he = (T)(0.5 * P.eps), q = (T)(0.25 / P.eps);
  const int lanes = row_lanes(P.nx), row0 = (blockIdx.x * kBlock + threadIdx.x) / lanes;
  double sphi = 0.0, sarea = 0.0;
  if constexpr (std::is_same<T, float>::value) {
    // The penalty multipliers use the small differences V - V0 and A - A0,
    // so both sums are formed in double-word arithmetic from phi = hi + lo.
    ScalarView<float> FL{phi_lo, P.nx, P.ny, P.nz, P.zper};
    CascadeSum cp(0.f), ca(0.f);
    // density c_A (eps/2 |grad phi|^2 + (phi^2 - 1)^2 / (4 eps)) from the
    // raw central differences, the constant factors folded into two pairs
    const FF agf{P.ag_hi, P.ag_lo}, awf{P.aw_hi, P.aw_lo};
    for (int row = row0; row < P.ny * P.nz; row += gridDim.x * kBlock / lanes) {
     const int k = row / P.ny, j = row - k * P.ny;
     for (int i = threadIdx.x & (lanes - 1); i < P.nx; i += lanes) {
      const long long t = lin(i, j, k, P.nx, P.ny);
      const FF f{phi[t], phi_lo[t]};
      auto diff = [&](int i1, int j1, int k1, int i0, int j0, int k0) {
        const FF a{F(i1, j1, k1), FL(i1, j1, k1)}, b{F(i0, j0, k0), FL(i0, j0, k0)};
        return ff_add(a, ff_neg(b));
      };
      const FF gx = diff(i + 1, j, k, i - 1, j, k);
      const FF gy = diff(i, j + 1, k, i, j - 1, k);
      const FF gz = diff(i, j, k + 1, i, j, k - 1);
      const FF g2 = ff_add(ff_add(ff_mul(gx, gx), ff_mul(gy, gy)), ff_mul(gz, gz));
      const FF w = ff_add_f(ff_mul(f, f), -1.f);
      const FF dens = ff_add(ff_mul(g2, agf), ff_mul(ff_mul(w, w), awf));
      cp.add(f.hi);
      cp.add(f.lo);
      ca.add(dens.hi);
      ca.add(dens.lo);
     }
    }
    sphi = (double)cp.hi + (double)cp.lo;
    sarea = (double)ca.hi + (double)ca.lo;
  } else {
    for (int row = row0; row < P.ny * P.nz; row += gridDim.x * kBlock / lanes) {
     const int k = row / P.ny, j = row - k * P.ny;
     for (int i = threadIdx.x & (lanes - 1); i < P.nx; i += lanes) {
      const long long t = lin(i, j, k, P.nx, P.ny);
      const double f = phi[t];
      const double gx = (F(i + 1, j, k) - F(i - 1, j, k)) * hih;
      const double gy = (F(i, j + 1, k) - F(i, j - 1, k)) * hih;
      const double gz = (F(i, j, k + 1) - F(i, j, k - 1)) * hih;
      const double w = f * f - 1.0;
      sphi += f;
      sarea += c_a * (he * (gx * gx + gy * gy + gz * gz) + w * w * q);
     }
    }
  }
  __shared__ double buf[2 * kBlock];
  va_publish(sphi, sarea, buf, partials, (long long)P.nx * P.ny * P.nz, S, init);
}

// ---------------------------------------------------------------- chemical potential
// Helfrich: g = phi^3 - phi - eps^2 lap phi.
template <class T>
__global__ void k_helfrich_g(PhaseParams P, const T* __restrict__ phi, T* __restrict__ g) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
  const T f = phi[t];
  g[t] = f * f * f - f - (T)(P.eps * P.eps) * lap7<T>(F, i, j, k, (T)P.inv_h2);
}

// CH (fe_kind 0): mu = phi^3 - phi - sigma lap phi.
// Helfrich: mu = cf2 [(3 phi^2 - 1) g - eps^2 lap g] - gamma_A lap phi
//           (+ beta_t g with a membrane tension).
template <class T>
__global__ void k_mu(PhaseParams P, const T* __restrict__ phi, const T* __restrict__ g,
                     const Scalars* S, T* __restrict__ mu) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const T ih2 = (T)P.inv_h2;
  ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
  const T f = phi[t];
  const T lphi = lap7<T>(F, i, j, k, ih2);
  if (P.fe_kind == VSV_CAHN_HILLIARD) {
    mu[t] = f * f * f - f - (T)P.sigma * lphi;
  } else {
    ScalarView<T> G{g, P.nx, P.ny, P.nz, P.zper};
    const T lg = lap7<T>(G, i, j, k, ih2);
    T m = (T)P.cf2 * (((T)3 * f * f - (T)1) * g[t] - (T)(P.eps * P.eps) * lg) -
          sc_gamma<T>(S) * lphi;
    if (P.beta_t != 0.0) m += (T)P.beta_t * g[t];
    mu[t] = m;
  }
}

// ---------------------------------------------------------------- vorticity source (eq. gen1)
// f = grad phi x grad mu / eta - s_omega(y, z)   (rhs of lap omega' = f - s_omega)
template <class T>
__global__ void k_source(PhaseParams P, const T* __restrict__ phi, const T* __restrict__ mu,
                         Comp3<T> s_omega, Comp3<T> f) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const T hih = (T)(0.5 * P.inv_h), ie = (T)P.inv_eta;
  ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
  ScalarView<T> M{mu, P.nx, P.ny, P.nz, P.zper};
  const T ax = (F(i + 1, j, k) - F(i - 1, j, k)) * hih;
  const T ay = (F(i, j + 1, k) - F(i, j - 1, k)) * hih;
  const T az = (F(i, j, k + 1) - F(i, j, k - 1)) * hih;
  const T bx = (M(i + 1, j, k) - M(i - 1, j, k)) * hih;
  const T by = (M(i, j + 1, k) - M(i, j - 1, k)) * hih;
  const T bz = (M(i, j, k + 1) - M(i, j, k - 1)) * hih;
  const long long jk = j + (long long)k * P.ny;
  f.p[0][t] = (ay * bz - az * by) * ie - s_omega.p[0][jk];
  f.p[1][t] = (az * bx - ax * bz) * ie - s_omega.p[1][jk];
  f.p[2][t] = (ax * by - ay * bx) * ie - s_omega.p[2][jk];
}

// ---------------------------------------------------------------- velocity (eq. vecpot)
// One component of v = v0 + curl psi' per launch (a field export needs one
// component, the observables ask for those they read).  Component c is
// dA/da - dB/db with (A, a; B, b) = (psi_z, y; psi_y, z), (psi_x, z; psi_z, x),
// (psi_y, x; psi_x, y).  Plain FP64 path:
template <class T>
__global__ void k_velocity(PhaseParams P, Comp3<T> psi, const T* __restrict__ v0, int c,
                           T* __restrict__ v) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const T hih = (T)(0.5 * P.inv_h);
  PertView<T> A{psi.at(c == 0 ? 2 : c - 1), P.nx, P.ny, P.nz, P.zper};
  PertView<T> B{psi.at(c == 2 ? 0 : c + 1), P.nx, P.ny, P.nz, P.zper};
  const int ax = c == 2, ay = c == 0, az = c == 1;       // axis a
  const int bx = c == 1, by = c == 2, bz = c == 0;       // axis b
  v[lin(i, j, k, P.nx, P.ny)] =
      v0[j + (long long)k * P.ny] +
      ((A(i + ax, j + ay, k + az) - A(i - ax, j - ay, k - az)) -
       (B(i + bx, j + by, k + bz) - B(i - bx, j - by, k - bz))) * hih;
}

// Velocity of the mixed path as a double word (hi + lo) for the observables
// and the exports (not on the time-stepping path): v = v0 + ((a+ - a-) - (b+ -
// b-)) / 2h from the double-word stream vector and the FP64 base-flow table.
// FP64 units do two operations per clock and SM here, so the eight words are
// summed by error-free FP32 transforms instead: high words, low words and the
// errors of both as a three-word expansion, scaled by the words of 1 / 2h and
// added to the three words of v0.  What is dropped is of order 2^-72 of the
// operands; the result is v rounded to its two words, at least as close to the
// real value as the FP64 evaluation it replaces (about 105 FP32 operations
// instead of 22 FP64 ones; 492 -> 33 us for three components at
// 256 x 128 x 128).
struct VelScale {
  float c1, c2, c3;   // 1 / 2h in three words
};
__device__ __forceinline__ void vel_dw(float aph, float apl, float amh, float aml, float bph, float bpl,
                                       float bmh, float bml, VelScale C, float v1, float v2, float v3,
                                       float& hi, float& lo) {
  float s, s2, e1, e2, e3, t, t2, f1, f2, f3, g1, g2, g3;
  two_sum(aph, -amh, s, e1);
  two_sum(bmh, -bph, s2, e2);
  two_sum(s, s2, s, e3);
  two_sum(apl, -aml, t, f1);
  two_sum(bml, -bpl, t2, f2);
  two_sum(t, t2, t, f3);
  two_sum(t, e1, t, g1);
  two_sum(t, e2, t, g2);
  two_sum(t, e3, t, g3);
  float f = __fadd_rn(__fadd_rn(__fadd_rn(f1, f2), f3), __fadd_rn(__fadd_rn(g1, g2), g3));
  // (s + t + f) (c1 + c2 + c3): leading words split exactly
  const float p = __fmul_rn(s, C.c1), pe = __fmaf_rn(s, C.c1, -p);
  float q = __fmul_rn(t, C.c1);
  f = __fmaf_rn(f, C.c1, __fmaf_rn(t, C.c1, -q));
  two_sum(q, pe, q, g1);
  f = __fadd_rn(f, g1);
  if (C.c2 != 0.f || C.c3 != 0.f) {
    const float r = __fmul_rn(s, C.c2);
    two_sum(q, r, q, g1);
    f = __fadd_rn(f, __fadd_rn(g1, __fmaf_rn(s, C.c2, -r)));
    f = __fmaf_rn(s, C.c3, __fmaf_rn(t, C.c2, f));
  }
  float u, w;
  two_sum(p, v1, u, w);
  two_sum(w, q, w, g1);
  two_sum(w, v2, w, g2);
  f = __fadd_rn(f, __fadd_rn(__fadd_rn(g1, g2), v3));
  two_sum(u, w, u, w);
  two_sum(w, f, w, f);
  const FF r = fast_two_sum(u, w);
  hi = r.hi;
  lo = __fadd_rn(r.lo, f);
  // the transforms turn an infinity into NaN: keep it in the high word
  const float plain = v1 + ((aph - amh) - (bph - bmh)) * C.c1;
  if (!isfinite(plain)) {
    hi = plain;
    lo = plain - plain;
  }
}

__device__ __forceinline__ void split3(double v, float& a, float& b, float& c) {
  a = __double2float_rn(v);
  const double r = v - (double)a;
  b = __double2float_rn(r);
  c = __double2float_rn(r - (double)b);
}

// What the kernel writes: the two words (f, f_lo), the high word alone into a
// caller's FP32 field, or their sum into a caller's FP64 field.
enum { kVelWords = 0, kVelF32 = 1, kVelF64 = 2 };

template <int C, int OUT>
__global__ void k_velocity_dw(PhaseParams P, const float* __restrict__ ah, const float* __restrict__ al,
                              const float* __restrict__ bh, const float* __restrict__ bl,
                              const double* __restrict__ v0, VelScale S, float* __restrict__ vh,
                              float* __restrict__ vl, double* __restrict__ vd) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  PertView<float> A{ah, P.nx, P.ny, P.nz, P.zper}, AL{al, P.nx, P.ny, P.nz, P.zper};
  PertView<float> B{bh, P.nx, P.ny, P.nz, P.zper}, BL{bl, P.nx, P.ny, P.nz, P.zper};
  constexpr int ax = C == 2, ay = C == 0, az = C == 1, bx = C == 1, by = C == 2, bz = C == 0;
  float v1, v2, v3, hi, lo;
  split3(v0[j + (long long)k * P.ny], v1, v2, v3);
  vel_dw(A(i + ax, j + ay, k + az), AL(i + ax, j + ay, k + az), A(i - ax, j - ay, k - az),
         AL(i - ax, j - ay, k - az), B(i + bx, j + by, k + bz), BL(i + bx, j + by, k + bz),
         B(i - bx, j - by, k - bz), BL(i - bx, j - by, k - bz), S, v1, v2, v3, hi, lo);
  const long long t = lin(i, j, k, P.nx, P.ny);
  if (OUT != kVelF64) vh[t] = hi;
  if (OUT == kVelWords) vl[t] = lo;
  if (OUT == kVelF64) vd[t] = (double)hi + (double)lo;
}

// ---------------------------------------------------------------- observables
// A field value in FP64 (lo: the low word of a double word on the mixed path).
__device__ __forceinline__ double val64(const double* __restrict__ a, const double*, long long t) {
  return a[t];
}
__device__ __forceinline__ double val64(const float* __restrict__ a, const float* __restrict__ lo,
                                        long long t) {
  return lo ? f2d(a[t]) + f2d(lo[t]) : f2d(a[t]);
}

// Velocity (materialised; lo: the low words of a double-word velocity, or
// null) with the no-slip wall velocity on the wall nodes.
template <class T>
struct VelView {
  const T* __restrict__ a;
  const T* __restrict__ lo;
  int nx, ny, nz, zper, comp;
  const PhaseParams* P;
  __device__ __forceinline__ double operator()(int i, int j, int k) const {
    i = wrap_idx(i, nx);
    if (zper) k = wrap_idx(k, nz);
    if (j < 0) return P->vwall[0][comp];
    if (j >= ny) return P->vwall[1][comp];
    if (k < 0) return P->vwall[2][comp];
    if (k >= nz) return P->vwall[3][comp];
    return val64(a, lo, lin(i, j, k, nx, ny));
  }
};

// Base-flow velocity table (x-invariant) with the same wall values.
struct V0View {
  const double* a;
  int ny, nz, zper, comp;
  const PhaseParams* P;
  __device__ __forceinline__ double operator()(int j, int k) const {
    if (zper) k = wrap_idx(k, nz);
    if (j < 0) return P->vwall[0][comp];
    if (j >= ny) return P->vwall[1][comp];
    if (k < 0) return P->vwall[2][comp];
    if (k >= nz) return P->vwall[3][comp];
    return a[j + (long long)k * ny];
  }
};

// |x| as an integer that orders like it (0 for a NaN, which fmax skips too)
__device__ __forceinline__ long long abs_bits(double x) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffLL;
  return b <= 0x7ff0000000000000LL ? b : 0;
}

// q: 0 dissipation integrand, 1 body-free dissipation integrand, 2 |omega'|^2,
// 3 |psi'|^2, 4 w = (1-phi)/2, 5..7 w x, w y, w z, 8 energy density,
// 9 max |div v|, 10 max |div psi|, 11 max sigma_t, 12 (Helfrich with a
// membrane tension) the face-difference area density over c_A / eps.
// vel_lo, om_lo, ps_lo: low words of double-word velocity, omega' and psi'
// (mixed path), or null pointers.  Two kernels: the velocity's quantities
// (0, 1, 9, 11), and the others.
//
// Bound by the FP64 units (two operations per clock and SM, long latency):
// conversions go through f2d, the strain is taken from raw differences (its
// scale 1 / 2h, the viscosity and h are applied once per block), each
// symmetric pair once, maxima compare bits, the one square root is taken of
// the maximum, and what does not depend on x is done once per row (a warp
// takes whole rows).  About 80 FP64 operations per cell instead of 270:
// 2,114 -> 406 + 326 us at 256 x 128 x 128 (470 G operations/s; additions alone
// reach 490 here).
template <class T>
__global__ void __launch_bounds__(kBlock, 4)
k_diag_flow(PhaseParams P, Comp3<T> vel, Comp3<T> vel_lo, Comp3<const double> v0d, double* partials) {
  double diss = 0.0, diss0 = 0.0;
  long long mv = 0, ms = 0;   // maxima of |div v| and of the squared shears
  const double hih = 0.5 * P.inv_h, eta = 1.0 / P.inv_eta;
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  for (int row = blockIdx.x * wpb + (threadIdx.x >> 5); row < P.ny * P.nz; row += gridDim.x * wpb) {
    const int k = row / P.ny, j = row - k * P.ny;
    if (lane == 0) {   // the body-free flow does not depend on x
      double G0[3][3];
      for (int c = 0; c < 3; ++c) {
        V0View W{v0d.p[c], P.ny, P.nz, P.zper, c, &P};
        G0[c][0] = 0.0;
        G0[c][1] = W(j + 1, k) - W(j - 1, k);
        G0[c][2] = W(j, k + 1) - W(j, k - 1);
      }
      double d0 = 0.0;
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
          const double e0 = G0[a][b] + G0[b][a];
          d0 += e0 * e0;
        }
      diss0 += d0 * (double)P.nx;
    }
    // rows of the six neighbours' kinds (negative: a wall, whose index is kept)
    const int km = P.zper ? wrap_idx(k - 1, P.nz) : k - 1, kp = P.zper ? wrap_idx(k + 1, P.nz) : k + 1;
    const long long rc = (long long)row * P.nx, ps = (long long)P.ny * P.nx;
    const long long rym = j > 0 ? rc - P.nx : -1, ryp = j < P.ny - 1 ? rc + P.nx : -2;
    const long long rzm = km >= 0 ? rc + (km - k) * ps : -3, rzp = kp < P.nz ? rc + (kp - k) * ps : -4;
    auto v = [&](int c, long long r, int i) {
      return r >= 0 ? val64(vel.at(c), vel_lo.at(c), r + i) : P.vwall[-1 - r][c];
    };
    for (int i = lane; i < P.nx; i += 32) {
      const int il = i > 0 ? i - 1 : P.nx - 1, ir = i < P.nx - 1 ? i + 1 : 0;
      // raw central differences
      const double xx = v(0, rc, ir) - v(0, rc, il);
      const double yy = v(1, ryp, i) - v(1, rym, i);
      const double zz = v(2, rzp, i) - v(2, rzm, i);
      const double xy = (v(0, ryp, i) - v(0, rym, i)) + (v(1, rc, ir) - v(1, rc, il));
      const double yz = (v(1, rzp, i) - v(1, rzm, i)) + (v(2, ryp, i) - v(2, rym, i));
      const double xz = (v(0, rzp, i) - v(0, rzm, i)) + (v(2, rc, ir) - v(2, rc, il));
      const double dg = xx * xx + yy * yy + zz * zz, sh = xy * xy + yz * yz + xz * xz;
      diss += 2.0 * dg + sh;          // half of sum_ij (2 e_ij)^2
      ms = max(ms, abs_bits(sh));
      mv = max(mv, abs_bits(xx + yy + zz));
    }
  }
  diss = block_sum(diss * (2.0 * hih * hih));
  diss0 = block_sum(diss0 * (hih * hih));
  const double dv = block_max(__longlong_as_double(mv) * hih);
  const double st = block_max(eta * hih * sqrt(__longlong_as_double(ms)));
  if (threadIdx.x == 0) {
    double* out = partials + (long long)blockIdx.x * kDiagQ;
    out[0] = diss;
    out[1] = diss0;
    out[9] = dv;
    out[11] = st;
  }
}

template <class T>
__global__ void __launch_bounds__(kBlock, 4)
k_diag_state(PhaseParams P, const T* __restrict__ phi, const T* __restrict__ phi_lo,
             const T* __restrict__ g, const T* __restrict__ g_lo, Comp3<T> omega, Comp3<T> om_lo,
             Comp3<T> psi, Comp3<T> ps_lo, Comp3<const double> psi0r, double* partials) {
  double q[7], q12 = 0.0;   // quantities 2 .. 8
  for (int a = 0; a < 7; ++a) q[a] = 0.0;
  long long mp = 0;         // maximum of |div psi|
  const double hih = 0.5 * P.inv_h, h = P.h;
  const bool tension = P.fe_kind == VSV_HELFRICH && P.beta_t != 0.0;
  const int ny2 = P.ny + 2, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  for (int row = blockIdx.x * wpb + (threadIdx.x >> 5); row < P.ny * P.nz; row += gridDim.x * wpb) {
    const int k = row / P.ny, j = row - k * P.ny;
    const int km = P.zper ? wrap_idx(k - 1, P.nz) : k - 1, kp = P.zper ? wrap_idx(k + 1, P.nz) : k + 1;
    const long long rc = (long long)row * P.nx, ps = (long long)P.ny * P.nx;
    const long long rym = j > 0 ? rc - P.nx : -1, ryp = j < P.ny - 1 ? rc + P.nx : -1;
    const long long rzm = km >= 0 ? rc + (km - k) * ps : -1, rzp = kp < P.nz ? rc + (kp - k) * ps : -1;
    // div psi with psi = psi0(y, z) + psi'; psi0 ring table holds the wall data
    auto r0 = [&](int c, int jj, int kk) { return psi0r.p[c][(jj + 1) + (long long)(kk + 1) * ny2]; };
    const double div0 = (r0(1, j + 1, k) - r0(1, j - 1, k)) + (r0(2, j, kp) - r0(2, j, km));
    auto p = [&](int c, long long r, int i) {
      return r >= 0 ? val64(psi.at(c), ps_lo.at(c), r + i) : 0.0;
    };
    double wr = 0.0;
    for (int i = lane; i < P.nx; i += 32) {
      const int il = i > 0 ? i - 1 : P.nx - 1, ir = i < P.nx - 1 ? i + 1 : 0;
      const long long t = rc + i;
      mp = max(mp, abs_bits((p(0, rc, ir) - p(0, rc, il)) + (p(1, ryp, i) - p(1, rym, i)) +
                            (p(2, rzp, i) - p(2, rzm, i)) + div0));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double o = val64(omega.at(c), om_lo.at(c), t), s = val64(psi.at(c), ps_lo.at(c), t);
        q[0] += o * o;
        q[1] += s * s;
      }
      const double f = val64(phi, phi_lo, t);
      const double w = 0.5 - 0.5 * f;
      wr += w;
      q[3] += w * f2d((float)i + 0.5f);
      if (P.fe_kind == VSV_HELFRICH) {
        const double gg = val64(g, g_lo, t);
        q[6] += gg * gg;
        if (tension) {   // the face-difference area density
          ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
          ScalarView<T> FL{phi_lo ? phi_lo : phi, P.nx, P.ny, P.nz, P.zper};
          auto val = [&](int ii, int jj, int kk) {
            return (double)F(ii, jj, kk) + (phi_lo ? (double)FL(ii, jj, kk) : 0.0);
          };
          const double dx = (val(i + 1, j, k) - f) * P.inv_h;
          double faces = dx * dx;
          if (j + 1 < P.ny) {
            const double dy = (val(i, j + 1, k) - f) * P.inv_h;
            faces += dy * dy;
          }
          if (P.zper || k + 1 < P.nz) {
            const double dz = (val(i, j, k + 1) - f) * P.inv_h;
            faces += dz * dz;
          }
          q12 += 0.25 * (f * f - 1.0) * (f * f - 1.0) + 0.5 * P.eps * P.eps * faces;
        }
      } else {
        ScalarView<T> F{phi, P.nx, P.ny, P.nz, P.zper};
        double e = 0.25 * (f * f - 1.0) * (f * f - 1.0);
        const double dx = ((double)F(i + 1, j, k) - f) * P.inv_h;
        double faces = dx * dx;
        if (j + 1 < P.ny) {
          const double dy = ((double)F(i, j + 1, k) - f) * P.inv_h;
          faces += dy * dy;
        }
        if (P.zper || k + 1 < P.nz) {
          const double dz = ((double)F(i, j, k + 1) - f) * P.inv_h;
          faces += dz * dz;
        }
        q[6] += e + 0.5 * P.sigma * faces;
      }
    }
    q[2] += wr;
    q[4] += wr * (j + 1.0);
    q[5] += wr * (P.zper ? (k + 0.5) : (k + 1.0));
  }
  q[3] *= h; q[4] *= h; q[5] *= h;
  double* out = partials + (long long)blockIdx.x * kDiagQ;
  for (int a = 0; a < 7; ++a) {
    const double s = block_sum(q[a]);
    if (threadIdx.x == 0) out[2 + a] = s;
  }
  const double m = block_max(__longlong_as_double(mp) * hih), s12 = block_sum(q12);
  if (threadIdx.x == 0) {
    out[10] = m;
    out[12] = s12;
  }
}

// The in-plane stress sigma_t = eta sqrt((2 e_xy)^2 + (2 e_yz)^2 + (2 e_xz)^2)
// of one cell in FP64 (f = eta / 2h), for values up to the type's ends: each shear
// is scaled before it is squared.
template <class T>
__device__ __forceinline__ double sigma_t64(const PhaseParams& P, const Comp3<T>& vel, const Comp3<T>& vel_lo,
                                            double f, int i, int j, int k) {
  VelView<T> X{vel.at(0), vel_lo.at(0), P.nx, P.ny, P.nz, P.zper, 0, &P};
  VelView<T> Y{vel.at(1), vel_lo.at(1), P.nx, P.ny, P.nz, P.zper, 1, &P};
  VelView<T> Z{vel.at(2), vel_lo.at(2), P.nx, P.ny, P.nz, P.zper, 2, &P};
  const double xy = f * ((X(i, j + 1, k) - X(i, j - 1, k)) + (Y(i + 1, j, k) - Y(i - 1, j, k)));
  const double yz = f * ((Y(i, j, k + 1) - Y(i, j, k - 1)) + (Z(i, j + 1, k) - Z(i, j - 1, k)));
  const double xz = f * ((X(i, j, k + 1) - X(i, j, k - 1)) + (Z(i + 1, j, k) - Z(i - 1, j, k)));
  return sqrt(xy * xy + yz * yz + xz * xz);
}
__device__ __noinline__ float sigma_t32(const PhaseParams& P, const Comp3<float>& vel,
                                        const Comp3<float>& vel_lo, double f, int i, int j, int k) {
  return (float)sigma_t64(P, vel, vel_lo, f, i, j, k);
}

__global__ void k_sigma_t(const __grid_constant__ PhaseParams P, Comp3<double> vel, Comp3<double> vel_lo,
                          double f, double* __restrict__ out) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  out[lin(i, j, k, P.nx, P.ny)] = sigma_t64(P, vel, vel_lo, f, i, j, k);
}

// A shear (a+ - a-) + (b+ - b-) of double words, as vel_dw sums them: exactly but
// for the last word, whose roundings are below 5 x 2^-24 `tail`.
__device__ __forceinline__ FF shear_dw(FF ap, FF am, FF bp, FF bm, float& tail) {
  float s, s2, e1, e2, e3, t, t2, f1, f2, f3, g1, g2, g3;
  two_sum(ap.hi, -am.hi, s, e1);
  two_sum(bp.hi, -bm.hi, s2, e2);
  two_sum(s, s2, s, e3);
  two_sum(ap.lo, -am.lo, t, f1);
  two_sum(bp.lo, -bm.lo, t2, f2);
  two_sum(t, t2, t, f3);
  two_sum(t, e1, t, g1);
  two_sum(t, e2, t, g2);
  two_sum(t, e3, t, g3);
  float f = __fadd_rn(__fadd_rn(__fadd_rn(f1, f2), f3), __fadd_rn(__fadd_rn(g1, g2), g3));
  tail += fabsf(f1) + fabsf(f2) + fabsf(f3) + fabsf(g1) + fabsf(g2) + fabsf(g3);
  two_sum(s, t, s, t);
  two_sum(t, f, t, f);
  two_sum(s, t, s, t);
  return FF{s, __fadd_rn(t, f)};
}

// The mixed path's stress field: the stress of the velocity's double words,
// rounded to FP32 once, by FP32 operations clear of the FP64 units.  The shears
// are summed without error and scaled by the power of two of their size (so that
// squares neither overflow nor vanish); squares, root and the factor f = fm 2^fe
// are double words, with a relative error below 2^-41 in all.  Cells whose
// rounding that leaves open (one in 2^15), whose shears cancel by more than about
// 2^20 or are out of the operations' range (zeros, infinities, NaN, results near
// FP32's ends), and those beside a wall, whose velocity has 53 bits, take the
// FP64 evaluation.  83 us at 256 x 128 x 128 (in FP32 double words throughout, with
// neither the range nor the last bits, 87); the export with its velocity 169 us, on
// the FP64 path 345.
__global__ void k_sigma_t_dw(const __grid_constant__ PhaseParams P, const __grid_constant__ Comp3<float> vel,
                             const __grid_constant__ Comp3<float> vel_lo, double f, FF fm, int fe,
                             float* __restrict__ out) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long c = lin(i, j, k, P.nx, P.ny), plane = (long long)P.nx * P.ny;
  const bool wall = j == 0 || j == P.ny - 1 || (!P.zper && (k == 0 || k == P.nz - 1));
  if (!wall) {
    const long long xp = c + (i < P.nx - 1 ? 1 : 1 - P.nx), xm = c + (i > 0 ? -1 : P.nx - 1);
    const long long zp = c + (k < P.nz - 1 ? plane : (1 - P.nz) * plane);
    const long long zm = c + (k > 0 ? -plane : (P.nz - 1) * plane);
    auto v = [&](int q, long long t) { return FF{vel.at(q)[t], vel_lo.at(q)[t]}; };
    float tail = 0.f;
    FF a = shear_dw(v(0, c + P.nx), v(0, c - P.nx), v(1, xp), v(1, xm), tail);
    FF b = shear_dw(v(1, zp), v(1, zm), v(2, c + P.nx), v(2, c - P.nx), tail);
    FF d = shear_dw(v(0, zp), v(0, zm), v(2, xp), v(2, xm), tail);
    const float m = fabsf(a.hi) + fabsf(b.hi) + fabsf(d.hi);   // a NaN stays one
    if (m >= 0x1p-80f && m <= 0x1p80f && tail * 0x1p24f <= m) {
      const int e = __float_as_int(m) >> 23;
      const float sc = __int_as_float((254 - e) << 23);
      a = FF{a.hi * sc, a.lo * sc};
      b = FF{b.hi * sc, b.lo * sc};
      d = FF{d.hi * sc, d.lo * sc};
      const FF s = ff_add(ff_add(ff_mul(a, a), ff_mul(b, b)), ff_mul(d, d));
      const float r = __fsqrt_rn(s.hi);
      const FF y = ff_mul(fast_two_sum(r, (__fmaf_rn(-r, r, s.hi) + s.lo) * __fdividef(0.5f, r)), fm);
      const float lo = __fmaf_rn(y.hi, -0x1p-40f, y.lo), hi = __fmaf_rn(y.hi, 0x1p-40f, y.lo);
      const float q = __fadd_rn(y.hi, lo);
      const int x = e + fe;   // the result's exponent field, but for the factor 2 q
      if (q == __fadd_rn(y.hi, hi) && x >= 2 && x <= 250) {
        out[c] = q * __int_as_float(x << 23);
        return;
      }
    }
  }
  out[c] = sigma_t32(P, vel, vel_lo, f, i, j, k);
}

// one block per quantity
__global__ void k_diag_finalize(const double* partials, int nblocks, double* out) {
  const int a = blockIdx.x;   // 0..8 and 12 are sums, 9..11 maxima
  const bool sum = a < 9 || a == 12;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    const double v = partials[(long long)b * kDiagQ + a];
    s = sum ? s + v : fmax(s, v);
  }
  s = sum ? block_sum(s) : block_max(s);
  if (threadIdx.x == 0) out[a] = s;
}

// <sigma_xy>(y) = eta <d_y v_x + d_x v_y> over x and z.  The mean of the
// periodic central difference d_x v_y vanishes term by term, so v_y is not read (a
// NaN in it alone shows in the diagnostics, not here); the differences of
// v_x are formed and summed in FP64 (sums of v_x would lose to the subtraction of
// neighbouring rows what v exceeds its differences by).  One block per row and
// chunk of planes: four FP64 operations a cell.  256 x 128 x 128: 45 + 3 us
// (sums of v_x in FP32 double words 13 + 4); the call 101 us (69), on the FP64 path
// 100 (sums of v_x 90); with d_x v_y summed too, one block a row, 830 and 322.
template <class T>
__global__ void k_stress_profile(const __grid_constant__ PhaseParams P, const T* __restrict__ vx,
                                 const T* __restrict__ vx_lo, int kchunk, double scale,
                                 double* __restrict__ sums) {
  const int j = blockIdx.x, kb = blockIdx.y * kchunk, ke = min(kb + kchunk, P.nz);
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const bool up = j + 1 < P.ny, down = j > 0;
  double s = 0.0;
  for (int k = kb + (threadIdx.x >> 5); k < ke; k += wpb)
    for (int i = lane; i < P.nx; i += 32) {
      const long long t = lin(i, j, k, P.nx, P.ny);
      s += (up ? val64(vx, vx_lo, t + P.nx) : P.vwall[1][0]) - (down ? val64(vx, vx_lo, t - P.nx) : P.vwall[0][0]);
    }
  s = block_sum(s);
  if (threadIdx.x == 0) sums[(long long)blockIdx.y * P.ny + j] = s * scale;
}
__global__ void k_profile_total(const double* __restrict__ sums, int ny, int chunks, double scale,
                                double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ny) return;
  double s = 0.0;
  for (int c = 0; c < chunks; ++c) s += sums[(long long)c * ny + j];
  out[j] = s * scale;
}

// ---------------------------------------------------------------- small utilities
template <class Tin, class Tout>
__global__ void k_convert(const Tin* __restrict__ in, Tout* __restrict__ out, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) out[t] = (Tout)in[t];
}

// out = pert + table(y, z); ring = 1: table in ring layout ((ny+2) x (nz+2)).
template <class T>
__global__ void k_full_field(PhaseParams P, const T* __restrict__ pert, const T* __restrict__ lo,
                             const double* __restrict__ tab, int ring, T* __restrict__ out) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const double b = ring ? tab[(j + 1) + (long long)(k + 1) * (P.ny + 2)] : tab[j + (long long)k * P.ny];
  out[t] = (T)((double)pert[t] + (lo ? (double)lo[t] : 0.0) + b);
}

// Full field in FP64 from a double-word perturbation: out = hi + lo + table.
__global__ void k_full_field_dw(PhaseParams P, const float* __restrict__ hi, const float* __restrict__ lo,
                                const double* __restrict__ tab, int ring, double* __restrict__ out) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const double b = tab ? (ring ? tab[(j + 1) + (long long)(k + 1) * (P.ny + 2)] : tab[j + (long long)k * P.ny]) : 0.0;
  out[t] = (double)hi[t] + (double)lo[t] + b;
}

void launch_full_field_dw(Ctx& cx, const PhaseParams& P, const float* hi, const float* lo,
                          const double* tab, int ring, double* out) {
  cx.before(-1);
  k_full_field_dw<<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, hi, lo, tab, ring, out);
  cx.after(-1);
}

template <class T>
__global__ void k_scale_copy(const T* __restrict__ in, T* __restrict__ out, long long n, T a) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) out[t] = a * in[t];
}

// ---------------------------------------------------------------- time-dependent walls
// One thread: the device time of the wall data, advanced by one step (or
// set), so that a captured graph of steps carries the time with it.
__global__ void k_wall_time(double* t_dev, double dt, int set_time, double t_set) {
  *t_dev = set_time ? t_set : *t_dev + dt;
}

__device__ __forceinline__ double wall_speed(const WallTables& W, int w, double t) {
  return W.s0[w] + W.ramp[w] * t + W.amp[w] * sin(2.0 * 3.14159265358979323846 * W.freq[w] * t +
                                                  W.phase[w]);
}

// Current tables = s_0(t) B_0 + s_1(t) B_1, every table and component in
// one grid-stride loop over a flat index.
template <class T>
__global__ void k_wall_tables(const __grid_constant__ WallTables W) {
  const double t = *W.t_dev;
  const double a = wall_speed(W, 0, t), b = wall_speed(W, 1, t);
  const long long nr = W.n_ring, nt = W.n_tab;
  const long long total = 3 * (2 * nr + 3 * nt);
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    long long r = q;
    const int c = (int)(r / (2 * nr + 3 * nt));
    r -= c * (2 * nr + 3 * nt);
    if (r < nr) {
      W.om[c][r] = a * W.bom[0][c][r] + b * W.bom[1][c][r];
    } else if ((r -= nr) < nr) {
      W.ps[c][r] = a * W.bps[0][c][r] + b * W.bps[1][c][r];
    } else if ((r -= nr) < nt) {
      const double v = a * W.bv0[0][c][r] + b * W.bv0[1][c][r];
      W.v0[c][r] = v;
      ((T*)W.v0t[c])[r] = (T)v;
    } else if ((r -= nt) < nt) {
      const double v = a * W.bsom[0][c][r] + b * W.bsom[1][c][r];
      W.som[c][r] = v;
      ((T*)W.somt[c])[r] = (T)v;
    } else {
      r -= nt;
      const double v = a * W.bsps[0][c][r] + b * W.bsps[1][c][r];
      W.sps[c][r] = v;
      ((T*)W.spsnt[c])[r] = (T)(-v);
    }
  }
}

template <class T>
void launch_wall_tables(Ctx& cx, const WallTables& W, double dt, bool set_time, double t_set) {
  cx.before(-1);
  k_wall_time<<<1, 1, 0, cx.stream>>>(W.t_dev, dt, set_time ? 1 : 0, t_set);
  cx.after(-1);
  const long long total = 3LL * (2LL * W.n_ring + 3LL * W.n_tab);
  const unsigned blocks = (unsigned)std::min<long long>((total + kBlock - 1) / kBlock, 4LL * cx.sms);
  cx.before(-1);
  k_wall_tables<T><<<blocks, kBlock, 0, cx.stream>>>(W);
  cx.after(-1, 8.0 * (double)total * 3.0);
}
template void launch_wall_tables<float>(Ctx&, const WallTables&, double, bool, double);
template void launch_wall_tables<double>(Ctx&, const WallTables&, double, bool, double);

// ---------------------------------------------------------------- base-flow tables (FP64)
// Ring layout: entry (j, k), j in [-1, ny], k in [-1, nz], at (j+1) + (k+1)(ny+2).
__device__ __forceinline__ long long ring_at(int j, int k, int ny) {
  return (j + 1) + (long long)(k + 1) * (ny + 2);
}

// Duct wall data from u0 and chi (interior layout j + k ny): normal
// derivative on a wall node by (4 f_1 - f_2) / (2h) (f = 0 on the wall),
// tangential derivatives zero.
__global__ void k_duct_ring(int ny, int nz, double h, const double* u0, const double* chi,
                            double* omy, double* omz, double* psy, double* psz) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const double ih = 1.0 / (2.0 * h);
  if (t < nz) {  // y walls at row k = t
    const int k = t;
    const double* u = u0 + (long long)k * ny;
    const double* c = chi + (long long)k * ny;
    const double du_lo = (4.0 * u[0] - u[1]) * ih, du_hi = -(4.0 * u[ny - 1] - u[ny - 2]) * ih;
    const double dc_lo = (4.0 * c[0] - c[1]) * ih, dc_hi = -(4.0 * c[ny - 1] - c[ny - 2]) * ih;
    omz[ring_at(-1, k, ny)] = -du_lo;
    omz[ring_at(ny, k, ny)] = -du_hi;
    psz[ring_at(-1, k, ny)] = dc_lo;
    psz[ring_at(ny, k, ny)] = dc_hi;
    omy[ring_at(-1, k, ny)] = 0.0;
    omy[ring_at(ny, k, ny)] = 0.0;
    psy[ring_at(-1, k, ny)] = 0.0;
    psy[ring_at(ny, k, ny)] = 0.0;
  }
  if (t < ny) {  // z walls at column j = t
    const int j = t;
    const double el = (4.0 * u0[j] - u0[j + ny]) * ih;
    const double eh = -(4.0 * u0[j + (long long)(nz - 1) * ny] - u0[j + (long long)(nz - 2) * ny]) * ih;
    const double cl = (4.0 * chi[j] - chi[j + ny]) * ih;
    const double ch = -(4.0 * chi[j + (long long)(nz - 1) * ny] - chi[j + (long long)(nz - 2) * ny]) * ih;
    omy[ring_at(j, -1, ny)] = el;
    omy[ring_at(j, nz, ny)] = eh;
    psy[ring_at(j, -1, ny)] = -cl;
    psy[ring_at(j, nz, ny)] = -ch;
    omz[ring_at(j, -1, ny)] = 0.0;
    omz[ring_at(j, nz, ny)] = 0.0;
    psz[ring_at(j, -1, ny)] = 0.0;
    psz[ring_at(j, nz, ny)] = 0.0;
  }
}

// out = scale * in - (wall-node contribution of `ring` to the 2-D
// Laplacian), both walls in y and z (the duct section).
__global__ void k_ring_rhs(int ny, int nz, double h, const double* ring, double scale,
                           const double* in, double* out) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)ny * nz) return;
  const int j = (int)(t % ny), k = (int)(t / ny);
  double b = 0.0;
  if (j == 0) b += ring[ring_at(-1, k, ny)];
  if (j == ny - 1) b += ring[ring_at(ny, k, ny)];
  if (k == 0) b += ring[ring_at(j, -1, ny)];
  if (k == nz - 1) b += ring[ring_at(j, nz, ny)];
  out[t] = (in ? scale * in[t] : 0.0) - b / (h * h);
}

__global__ void k_ring_fill(int ny, int nz, const double* interior, double* ring) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)ny * nz) return;
  const int j = (int)(t % ny), k = (int)(t / ny);
  ring[ring_at(j, k, ny)] = interior[t];
}

// v0 = curl psi0 (x-invariant), s_omega = lap omega0, s_psi = lap psi0 + omega0,
// all on the interior (y, z) cells from ring tables.
__global__ void k_base_derived(int ny, int nz, int zper, double h, Comp3<const double> om,
                               Comp3<const double> ps, Comp3<double> v0, Comp3<double> som,
                               Comp3<double> sps) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)ny * nz) return;
  const int j = (int)(t % ny), k = (int)(t / ny);
  auto at = [&](const double* r, int jj, int kk) -> double {
    if (zper) kk = wrap_idx(kk, nz);
    return r[ring_at(jj, kk, ny)];
  };
  const double hih = 0.5 / h, ih2 = 1.0 / (h * h);
  const double* px = ps.p[0];
  const double* py = ps.p[1];
  const double* pz = ps.p[2];
  v0.p[0][t] = ((at(pz, j + 1, k) - at(pz, j - 1, k)) - (at(py, j, k + 1) - at(py, j, k - 1))) * hih;
  v0.p[1][t] = (at(px, j, k + 1) - at(px, j, k - 1)) * hih;
  v0.p[2][t] = -(at(px, j + 1, k) - at(px, j - 1, k)) * hih;
  for (int c = 0; c < 3; ++c) {
    const double* o = om.p[c];
    const double* p = ps.p[c];
    const double lo = (at(o, j + 1, k) + at(o, j - 1, k) + at(o, j, k + 1) + at(o, j, k - 1) -
                       4.0 * at(o, j, k)) * ih2;
    const double lp = (at(p, j + 1, k) + at(p, j - 1, k) + at(p, j, k + 1) + at(p, j, k - 1) -
                       4.0 * at(p, j, k)) * ih2;
    som.p[c][t] = lo;
    sps.p[c][t] = lp + at(o, j, k);
  }
}

__global__ void k_max_abs(const double* x, long long n, double* out) {
  double m = 0.0;
  for (long long t = threadIdx.x; t < n; t += blockDim.x) m = fmax(m, fabs(x[t]));
  m = block_max(m);
  if (threadIdx.x == 0) *out = m;
}

__global__ void k_fill(double* x, long long n, double v) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) x[t] = v;
}

// ---------------------------------------------------------------- mixed path: double-word phi
// Unscaled 7-point Laplacian sum (x+ + x- + y+ + y- + z+ + z- - 6 c) of a
// double-word field: the hi parts are summed by cascaded summation
// (error-free up to the final rounding), the lo parts in FP32 (their own
// rounding is below 2^-48 of the field).  Callers apply 1/h^2 together with
// their own coefficient, as one double-word product.
template <class V>
__device__ __forceinline__ FF lap7_ff(const V& H, const V& L, int i, int j, int k) {
  CascadeSum s(H(i + 1, j, k));
  s.add(H(i - 1, j, k));
  s.add(H(i, j + 1, k));
  s.add(H(i, j - 1, k));
  s.add(H(i, j, k + 1));
  s.add(H(i, j, k - 1));
  s.add_scaled(-6.f, H(i, j, k));
  const float lsum = L(i + 1, j, k) + L(i - 1, j, k) + L(i, j + 1, k) + L(i, j - 1, k) +
                     L(i, j, k + 1) + L(i, j, k - 1) - 6.f * L(i, j, k);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, lsum));
}

// phi^{n+1} = phi^n + dt * rate with phi^n = hi + lo; the rate itself is an
// O(1e-4) increment and is formed in FP32 as in the FP64 path.
__global__ void k_phi_update_ff(PhaseParams P, const float* __restrict__ phi,
                                const float* __restrict__ phi_lo, const float* __restrict__ mu,
                                Comp3<float> psi, Comp3<float> v0, Scalars* S, float dt,
                                float* __restrict__ out, float* __restrict__ out_lo) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  const float ih2 = (float)P.inv_h2, hih = (float)(0.5 * P.inv_h);
  ScalarView<float> M{mu, P.nx, P.ny, P.nz, P.zper};
  ScalarView<float> F{phi, P.nx, P.ny, P.nz, P.zper};
  PertView<float> X{psi.p[0], P.nx, P.ny, P.nz, P.zper};
  PertView<float> Y{psi.p[1], P.nx, P.ny, P.nz, P.zper};
  PertView<float> Z{psi.p[2], P.nx, P.ny, P.nz, P.zper};
  const float lmu = lap7<float>(M, i, j, k, ih2);
  const float gx = (F(i + 1, j, k) - F(i - 1, j, k)) * hih;
  const float gy = (F(i, j + 1, k) - F(i, j - 1, k)) * hih;
  const float gz = (F(i, j, k + 1) - F(i, j, k - 1)) * hih;
  const long long jk = j + (long long)k * P.ny;
  const float vx = v0.p[0][jk] + ((Z(i, j + 1, k) - Z(i, j - 1, k)) - (Y(i, j, k + 1) - Y(i, j, k - 1))) * hih;
  const float vy = v0.p[1][jk] + ((X(i, j, k + 1) - X(i, j, k - 1)) - (Z(i + 1, j, k) - Z(i - 1, j, k))) * hih;
  const float vz = v0.p[2][jk] + ((Y(i + 1, j, k) - Y(i - 1, j, k)) - (X(i, j + 1, k) - X(i, j - 1, k))) * hih;
  const float rate = (float)P.mobility * (lmu + S->lambda_vf) - (vx * gx + vy * gy + vz * gz);
  const FF v = ff_add_f(FF{phi[t], phi_lo[t]}, dt * rate);
  out[t] = v.hi;
  out_lo[t] = v.lo;
  if (!isfinite(v.hi)) atomicOr(&S->nonfinite, 1);
}

// g = phi^3 - phi - eps^2 lap phi in double-word arithmetic.
__global__ void k_helfrich_g_ff(PhaseParams P, const float* __restrict__ phi,
                                const float* __restrict__ phi_lo, float* __restrict__ g,
                                float* __restrict__ g_lo) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  ScalarView<float> H{phi, P.nx, P.ny, P.nz, P.zper};
  ScalarView<float> L{phi_lo, P.nx, P.ny, P.nz, P.zper};
  const FF f{phi[t], phi_lo[t]};
  const FF lphi = lap7_ff(H, L, i, j, k);
  const FF cubic = ff_mul(f, ff_add_f(ff_mul(f, f), -1.f));
  const FF r = ff_add(cubic, ff_neg(ff_mul(lphi, FF{P.e2ih_hi, P.e2ih_lo})));
  g[t] = r.hi;
  g_lo[t] = r.lo;
}

// CH:       mu = phi^3 - phi - sigma lap phi
// Helfrich: mu = cf2 [(3 phi^2 - 1) g - eps^2 lap g] - gamma_A lap phi (+ beta_t g)
__global__ void k_mu_ff(PhaseParams P, const float* __restrict__ phi, const float* __restrict__ phi_lo,
                        const float* __restrict__ g, const float* __restrict__ g_lo,
                        const Scalars* S, float* __restrict__ mu, float* __restrict__ mu_lo) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  ScalarView<float> H{phi, P.nx, P.ny, P.nz, P.zper};
  ScalarView<float> L{phi_lo, P.nx, P.ny, P.nz, P.zper};
  const FF f{phi[t], phi_lo[t]};
  const FF lphi = lap7_ff(H, L, i, j, k);
  if (P.fe_kind == VSV_CAHN_HILLIARD) {
    const FF cubic = ff_mul(f, ff_add_f(ff_mul(f, f), -1.f));
    const FF m = ff_add(cubic, ff_neg(ff_mul(lphi, FF{P.sgih_hi, P.sgih_lo})));
    mu[t] = m.hi;
    mu_lo[t] = m.lo;
    return;
  }
  ScalarView<float> GH{g, P.nx, P.ny, P.nz, P.zper};
  ScalarView<float> GL{g_lo, P.nx, P.ny, P.nz, P.zper};
  const FF gg{g[t], g_lo[t]};
  const FF lg = lap7_ff(GH, GL, i, j, k);
  const FF w = ff_add_f(ff_mul_f(ff_mul(f, f), 3.f), -1.f);
  const FF inner = ff_add(ff_mul(w, gg), ff_neg(ff_mul(lg, FF{P.e2ih_hi, P.e2ih_lo})));
  const FF gih = ff_mul_f(FF{P.ih2_hi, P.ih2_lo}, S->gamma_af);   // gamma_A / h^2
  FF m = ff_add(ff_mul(inner, FF{P.cf2_hi, P.cf2_lo}), ff_neg(ff_mul(lphi, gih)));
  if (P.bt_hi != 0.f) m = ff_add(m, ff_mul(gg, FF{P.bt_hi, P.bt_lo}));
  mu[t] = m.hi;
  mu_lo[t] = m.lo;
}

__global__ void k_split_ff(const double* __restrict__ in, float* __restrict__ hi,
                           float* __restrict__ lo, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double d = in[t];
  const float h = (float)d;
  hi[t] = h;
  lo[t] = (float)(d - (double)h);
}

__global__ void k_merge_ff(const float* __restrict__ hi, const float* __restrict__ lo,
                           double* __restrict__ out, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) out[t] = (double)hi[t] + (double)lo[t];
}

// The same splits and merges four elements per thread with 16-byte accesses
// (every array 16-byte aligned), grid-strided; the last n % 4 elements are
// done one per thread.  Used for device buffers and for mapped host memory,
// where fewer, wider requests cross the host link.
//
// The conversions between the formats run on the FP64 units (two a clock and
// SM), so four of them a cell, not the 16 bytes, bounded the split: it is done
// by integer operations where |d| is 0 or in [2^-74, 2^127), and the merge's
// exact conversions too.  33.5 M cells: split 243 -> 76 us, merge 182 -> 89 us.
__device__ __noinline__ float2 split_fp64(double d) {
  const float h = (float)d;
  return make_float2(h, (float)(d - (double)h));
}
// (h, l) = (RN(d), RN(d - h)) from the bits of d: the upper 23 fraction bits
// rounded to even, and the signed remainder (29 bits) times its power of two.
// False (nothing set) outside the range.
__device__ __forceinline__ bool split_bits(double d, float& h, float& l) {
  const unsigned u = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned ef = (u >> 20) & 0x7ffu;
  const bool zero = (u << 1 | lo) == 0u;
  if (!zero && ef - 949u > 200u) return false;
  const unsigned m = ((u << 3) & 0x7fffffu) | (lo >> 29);
  int rem = (int)(lo & 0x1fffffffu);
  const int up = rem + (int)(m & 1u) > (1 << 28);
  rem -= up << 29;
  h = __uint_as_float((u & 0x80000000u) | (zero ? 0u : ((ef - 896u) << 23 | m) + up));
  l = __int2float_rn((u & 0x80000000u) ? -rem : rem) *
      __uint_as_float(zero ? 0x3f800000u : (ef - 948u) << 23);
  return true;
}

__global__ void k_split_ff_v4(const double* __restrict__ in, float* __restrict__ hi,
                              float* __restrict__ lo, long long n) {
  const long long n4 = n >> 2, stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const double2* in2 = reinterpret_cast<const double2*>(in);
  for (long long t = t0; t < n4; t += stride) {
    const double2 a = in2[2 * t], b = in2[2 * t + 1];
    float4 h, l;
    bool ok = split_bits(a.x, h.x, l.x);
    ok &= split_bits(a.y, h.y, l.y);
    ok &= split_bits(b.x, h.z, l.z);
    ok &= split_bits(b.y, h.w, l.w);
    if (!ok) {
      const float2 p = split_fp64(a.x), q = split_fp64(a.y), r = split_fp64(b.x), s = split_fp64(b.y);
      h = make_float4(p.x, q.x, r.x, s.x);
      l = make_float4(p.y, q.y, r.y, s.y);
    }
    reinterpret_cast<float4*>(hi)[t] = h;
    reinterpret_cast<float4*>(lo)[t] = l;
  }
  const long long r = 4 * n4 + t0;
  if (r < n) {
    const double d = in[r];
    const float h = (float)d;
    hi[r] = h;
    lo[r] = (float)(d - (double)h);
  }
}

__global__ void k_merge_ff_v4(const float* __restrict__ hi, const float* __restrict__ lo,
                              double* __restrict__ out, long long n) {
  const long long n4 = n >> 2, stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double2* out2 = reinterpret_cast<double2*>(out);
  for (long long t = t0; t < n4; t += stride) {
    const float4 h = reinterpret_cast<const float4*>(hi)[t];
    const float4 l = reinterpret_cast<const float4*>(lo)[t];
    out2[2 * t] = make_double2(f2d(h.x) + f2d(l.x), f2d(h.y) + f2d(l.y));
    out2[2 * t + 1] = make_double2(f2d(h.z) + f2d(l.z), f2d(h.w) + f2d(l.w));
  }
  const long long r = 4 * n4 + t0;
  if (r < n) out[r] = (double)hi[r] + (double)lo[r];
}

// ---------------------------------------------------------------- 4-cell kernels
// The same double-word kernels with one thread per 4 consecutive x cells
// (nx a multiple of 4): the own cells and the y / z neighbours are 16-byte
// loads, the x neighbours two scalars, and the boundary index arithmetic is
// done once per row instead of once per access.  Per-cell arithmetic is that
// of the 1-cell kernels above, term for term.
namespace {

// A field around the 4 cells (i0 .. i0+3, j, k): own values c, the rows
// above / below (ym, yp), the planes below / above (zm, zp) and the x
// neighbours xl (i0 - 1) and xr (i0 + 4).
struct St4 {
  float4 c, ym, yp, zm, zp;
  float xl, xr;
};

__device__ __forceinline__ float e4(const float4& v, int o) {
  return o == 0 ? v.x : (o == 1 ? v.y : (o == 2 ? v.z : v.w));
}
__device__ __forceinline__ float4 ld4g(const float* p) { return *reinterpret_cast<const float4*>(p); }

// Row offsets of the 4-cell group's neighbourhood, with the boundary rule of
// scalars (mirror at walls) or of the flow perturbation (zero beyond walls,
// flagged by a negative offset); x wraps in both.
struct Geo4 {
  long long rc, rym, ryp, rzm, rzp;   // row offsets (plane * ny + row) * nx
  int il, ir;                          // x indices of the two x neighbours
  int i0;
};

__device__ __forceinline__ Geo4 geo4(const PhaseParams& P, int i0, int j, int k, bool pert) {
  Geo4 G;
  const long long nx = P.nx, ny = P.ny;
  auto row = [&](int jj, int kk) { return ((long long)kk * ny + jj) * nx; };
  G.i0 = i0;
  G.il = i0 == 0 ? P.nx - 1 : i0 - 1;
  G.ir = i0 + 4 == P.nx ? 0 : i0 + 4;
  G.rc = row(j, k);
  if (pert) {
    G.rym = j > 0 ? row(j - 1, k) : -1;
    G.ryp = j < P.ny - 1 ? row(j + 1, k) : -1;
    const int km = P.zper ? wrap_idx(k - 1, P.nz) : k - 1;
    const int kp = P.zper ? wrap_idx(k + 1, P.nz) : k + 1;
    G.rzm = km >= 0 ? row(j, km) : -1;
    G.rzp = kp < P.nz ? row(j, kp) : -1;
  } else {
    G.rym = row(mirror_idx(j - 1, P.ny), k);
    G.ryp = row(mirror_idx(j + 1, P.ny), k);
    G.rzm = row(j, P.zper ? wrap_idx(k - 1, P.nz) : mirror_idx(k - 1, P.nz));
    G.rzp = row(j, P.zper ? wrap_idx(k + 1, P.nz) : mirror_idx(k + 1, P.nz));
  }
  return G;
}

__device__ __forceinline__ St4 load4(const float* __restrict__ a, const Geo4& G) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  St4 S;
  S.c = ld4g(a + G.rc + G.i0);
  S.ym = G.rym >= 0 ? ld4g(a + G.rym + G.i0) : z;
  S.yp = G.ryp >= 0 ? ld4g(a + G.ryp + G.i0) : z;
  S.zm = G.rzm >= 0 ? ld4g(a + G.rzm + G.i0) : z;
  S.zp = G.rzp >= 0 ? ld4g(a + G.rzp + G.i0) : z;
  S.xl = a[G.rc + G.il];
  S.xr = a[G.rc + G.ir];
  return S;
}

// neighbours of cell o of the group
__device__ __forceinline__ float xp4(const St4& S, int o) { return o == 3 ? S.xr : e4(S.c, o + 1); }
__device__ __forceinline__ float xm4(const St4& S, int o) { return o == 0 ? S.xl : e4(S.c, o - 1); }

// lap7_ff on cell o (same order of operations)
// lap7_ff on cell o of a 4-cell group: the unscaled sum, same order
__device__ __forceinline__ FF lap7_ff4(const St4& H, const St4& L, int o) {
  CascadeSum s(xp4(H, o));
  s.add(xm4(H, o));
  s.add(e4(H.yp, o));
  s.add(e4(H.ym, o));
  s.add(e4(H.zp, o));
  s.add(e4(H.zm, o));
  s.add_scaled(-6.f, e4(H.c, o));
  const float lsum = xp4(L, o) + xm4(L, o) + e4(L.yp, o) + e4(L.ym, o) + e4(L.zp, o) +
                     e4(L.zm, o) - 6.f * e4(L.c, o);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, lsum));
}

// lap7 in plain FP32 on cell o (same order as lap7)
__device__ __forceinline__ float lap7_4(const St4& M, int o, float ih2) {
  return (xp4(M, o) + xm4(M, o) + e4(M.yp, o) + e4(M.ym, o) + e4(M.zp, o) + e4(M.zm, o) -
          6.f * e4(M.c, o)) * ih2;
}

__device__ __forceinline__ bool cell4(const PhaseParams& P, int& i0, int& j, int& k) {
  i0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  j = blockIdx.y * blockDim.y + threadIdx.y;
  k = blockIdx.z;
  return i0 < P.nx && j < P.ny;
}

}  // namespace

// k_velocity_dw on 4-cell groups
template <int C, int OUT>
__global__ void __launch_bounds__(256) k_velocity_dw4(PhaseParams P, const float* __restrict__ ah,
                                                      const float* __restrict__ al,
                                                      const float* __restrict__ bh,
                                                      const float* __restrict__ bl,
                                                      const double* __restrict__ v0, VelScale S,
                                                      float* __restrict__ vh, float* __restrict__ vl,
                                                      double* __restrict__ vd) {
  int i0, j, k;
  if (!cell4(P, i0, j, k)) return;
  const Geo4 G = geo4(P, i0, j, k, true);
  float v1, v2, v3;
  split3(v0[j + (long long)k * P.ny], v1, v2, v3);
  // plus and minus neighbours along axis D of the four cells
  auto pm = [&](const float* __restrict__ a, int axis, float4& p, float4& m) {
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    if (axis == 0) {
      const float4 c = ld4g(a + G.rc + i0);
      p = make_float4(c.y, c.z, c.w, a[G.rc + G.ir]);
      m = make_float4(a[G.rc + G.il], c.x, c.y, c.z);
    } else if (axis == 1) {
      p = G.ryp >= 0 ? ld4g(a + G.ryp + i0) : z;
      m = G.rym >= 0 ? ld4g(a + G.rym + i0) : z;
    } else {
      p = G.rzp >= 0 ? ld4g(a + G.rzp + i0) : z;
      m = G.rzm >= 0 ? ld4g(a + G.rzm + i0) : z;
    }
  };
  constexpr int aa = C == 2 ? 0 : (C == 0 ? 1 : 2), ab = C == 1 ? 0 : (C == 2 ? 1 : 2);
  float4 aph, amh, apl, aml, bph, bmh, bpl, bml;
  pm(ah, aa, aph, amh);
  pm(al, aa, apl, aml);
  pm(bh, ab, bph, bmh);
  pm(bl, ab, bpl, bml);
  float h[4], l[4];
#pragma unroll
  for (int o = 0; o < 4; ++o)
    vel_dw(e4(aph, o), e4(apl, o), e4(amh, o), e4(aml, o), e4(bph, o), e4(bpl, o), e4(bmh, o),
           e4(bml, o), S, v1, v2, v3, h[o], l[o]);
  const long long t = G.rc + i0;
  if (OUT != kVelF64) *reinterpret_cast<float4*>(vh + t) = make_float4(h[0], h[1], h[2], h[3]);
  if (OUT == kVelWords) *reinterpret_cast<float4*>(vl + t) = make_float4(l[0], l[1], l[2], l[3]);
  if (OUT == kVelF64) {
    double2* d = reinterpret_cast<double2*>(vd + t);
    d[0] = make_double2((double)h[0] + (double)l[0], (double)h[1] + (double)l[1]);
    d[1] = make_double2((double)h[2] + (double)l[2], (double)h[3] + (double)l[3]);
  }
}

__global__ void __launch_bounds__(256, 3) k_phi_update_ff4(PhaseParams P, const float* __restrict__ phi,
                                 const float* __restrict__ phi_lo, const float* __restrict__ mu,
                                 Comp3<float> psi, Comp3<float> v0, Scalars* S, float dt,
                                 float* __restrict__ out, float* __restrict__ out_lo) {
  pdl_begin();
  int i0, j, k;
  if (!cell4(P, i0, j, k)) return;
  const float ih2 = (float)P.inv_h2, hih = (float)(0.5 * P.inv_h);
  const Geo4 Gs = geo4(P, i0, j, k, false), Gp = geo4(P, i0, j, k, true);
  const St4 M = load4(mu, Gs), F = load4(phi, Gs);
  const St4 X = load4(psi.p[0], Gp), Y = load4(psi.p[1], Gp), Z = load4(psi.p[2], Gp);
  const long long jk = j + (long long)k * P.ny;
  const float v0x = v0.p[0][jk], v0y = v0.p[1][jk], v0z = v0.p[2][jk];
  const float lam = S->lambda_vf, mob = (float)P.mobility;
  const float4 fh = ld4g(phi + Gs.rc + i0), fl = ld4g(phi_lo + Gs.rc + i0);
  float oh[4], ol[4];
  bool finite = true;
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const float lmu = lap7_4(M, o, ih2);
    const float gx = (xp4(F, o) - xm4(F, o)) * hih;
    const float gy = (e4(F.yp, o) - e4(F.ym, o)) * hih;
    const float gz = (e4(F.zp, o) - e4(F.zm, o)) * hih;
    const float vx = v0x + ((e4(Z.yp, o) - e4(Z.ym, o)) - (e4(Y.zp, o) - e4(Y.zm, o))) * hih;
    const float vy = v0y + ((e4(X.zp, o) - e4(X.zm, o)) - (xp4(Z, o) - xm4(Z, o))) * hih;
    const float vz = v0z + ((xp4(Y, o) - xm4(Y, o)) - (e4(X.yp, o) - e4(X.ym, o))) * hih;
    const float rate = mob * (lmu + lam) - (vx * gx + vy * gy + vz * gz);
    const FF v = ff_add_f(FF{e4(fh, o), e4(fl, o)}, dt * rate);
    oh[o] = v.hi;
    ol[o] = v.lo;
    finite = finite && isfinite(v.hi);
  }
  *reinterpret_cast<float4*>(out + Gs.rc + i0) = make_float4(oh[0], oh[1], oh[2], oh[3]);
  *reinterpret_cast<float4*>(out_lo + Gs.rc + i0) = make_float4(ol[0], ol[1], ol[2], ol[3]);
  if (!finite) atomicOr(&S->nonfinite, 1);
}

__global__ void __launch_bounds__(256) k_helfrich_g_ff4(PhaseParams P, const float* __restrict__ phi,
                                 const float* __restrict__ phi_lo, float* __restrict__ g,
                                 float* __restrict__ g_lo) {
  pdl_begin();
  int i0, j, k;
  if (!cell4(P, i0, j, k)) return;
  const Geo4 G = geo4(P, i0, j, k, false);
  const St4 H = load4(phi, G), L = load4(phi_lo, G);
  float oh[4], ol[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const FF f{e4(H.c, o), e4(L.c, o)};
    const FF lphi = lap7_ff4(H, L, o);
    const FF cubic = ff_mul(f, ff_add_f(ff_mul(f, f), -1.f));
    const FF r = ff_add(cubic, ff_neg(ff_mul(lphi, FF{P.e2ih_hi, P.e2ih_lo})));
    oh[o] = r.hi;
    ol[o] = r.lo;
  }
  *reinterpret_cast<float4*>(g + G.rc + i0) = make_float4(oh[0], oh[1], oh[2], oh[3]);
  *reinterpret_cast<float4*>(g_lo + G.rc + i0) = make_float4(ol[0], ol[1], ol[2], ol[3]);
}

__global__ void __launch_bounds__(256) k_mu_ff4(PhaseParams P, const float* __restrict__ phi,
                                                const float* __restrict__ phi_lo,
                                                const float* __restrict__ g,
                                                const float* __restrict__ g_lo, const Scalars* S,
                                                float* __restrict__ mu, float* __restrict__ mu_lo) {
  pdl_begin();
  int i0, j, k;
  if (!cell4(P, i0, j, k)) return;
  const Geo4 G = geo4(P, i0, j, k, false);
  const St4 H = load4(phi, G), L = load4(phi_lo, G);
  float oh[4], ol[4];
  if (P.fe_kind == VSV_CAHN_HILLIARD) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const FF f{e4(H.c, o), e4(L.c, o)};
      const FF lphi = lap7_ff4(H, L, o);
      const FF cubic = ff_mul(f, ff_add_f(ff_mul(f, f), -1.f));
      const FF mm = ff_add(cubic, ff_neg(ff_mul(lphi, FF{P.sgih_hi, P.sgih_lo})));
      oh[o] = mm.hi;
      ol[o] = mm.lo;
    }
  } else {
    const St4 GH = load4(g, G), GL = load4(g_lo, G);
    const FF gih = ff_mul_f(FF{P.ih2_hi, P.ih2_lo}, S->gamma_af);   // gamma_A / h^2
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const FF f{e4(H.c, o), e4(L.c, o)};
      const FF lphi = lap7_ff4(H, L, o);
      const FF gg{e4(GH.c, o), e4(GL.c, o)};
      const FF lg = lap7_ff4(GH, GL, o);
      const FF w = ff_add_f(ff_mul_f(ff_mul(f, f), 3.f), -1.f);
      const FF inner = ff_add(ff_mul(w, gg), ff_neg(ff_mul(lg, FF{P.e2ih_hi, P.e2ih_lo})));
      FF mm = ff_add(ff_mul(inner, FF{P.cf2_hi, P.cf2_lo}), ff_neg(ff_mul(lphi, gih)));
      if (P.bt_hi != 0.f) mm = ff_add(mm, ff_mul(gg, FF{P.bt_hi, P.bt_lo}));
      oh[o] = mm.hi;
      ol[o] = mm.lo;
    }
  }
  *reinterpret_cast<float4*>(mu + G.rc + i0) = make_float4(oh[0], oh[1], oh[2], oh[3]);
  *reinterpret_cast<float4*>(mu_lo + G.rc + i0) = make_float4(ol[0], ol[1], ol[2], ol[3]);
}

__global__ void __launch_bounds__(256) k_source_ff4(PhaseParams P, const float* __restrict__ phi,
                                                    const float* __restrict__ phi_lo,
                                                    const float* __restrict__ mu,
                                                    const float* __restrict__ mu_lo,
                                                    Comp3<float> s_omega, Comp3<float> f,
                                                    Comp3<float> f_lo) {
  pdl_begin();
  int i0, j, k;
  if (!cell4(P, i0, j, k)) return;
  const Geo4 G = geo4(P, i0, j, k, false);
  const St4 FH = load4(phi, G), FL = load4(phi_lo, G), MH = load4(mu, G), ML = load4(mu_lo, G);
  // raw central differences; (1/2h)^2 / eta is applied once to each
  // component of the cross product
  const FF ie{P.src_hi, P.src_lo};
  const long long jk = j + (long long)k * P.ny;
  const float s0 = s_omega.p[0][jk], s1 = s_omega.p[1][jk], s2 = s_omega.p[2][jk];
  auto dd = [&](float ah, float al, float bh, float bl) {
    return ff_add(FF{ah, al}, ff_neg(FF{bh, bl}));
  };
  float o0h[4], o0l[4], o1h[4], o1l[4], o2h[4], o2l[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const FF ax = dd(xp4(FH, o), xp4(FL, o), xm4(FH, o), xm4(FL, o));
    const FF ay = dd(e4(FH.yp, o), e4(FL.yp, o), e4(FH.ym, o), e4(FL.ym, o));
    const FF az = dd(e4(FH.zp, o), e4(FL.zp, o), e4(FH.zm, o), e4(FL.zm, o));
    const FF bx = dd(xp4(MH, o), xp4(ML, o), xm4(MH, o), xm4(ML, o));
    const FF by = dd(e4(MH.yp, o), e4(ML.yp, o), e4(MH.ym, o), e4(ML.ym, o));
    const FF bz = dd(e4(MH.zp, o), e4(ML.zp, o), e4(MH.zm, o), e4(ML.zm, o));
    const FF c0 = ff_add_f(ff_mul(ff_add(ff_mul(ay, bz), ff_neg(ff_mul(az, by))), ie), -s0);
    const FF c1 = ff_add_f(ff_mul(ff_add(ff_mul(az, bx), ff_neg(ff_mul(ax, bz))), ie), -s1);
    const FF c2 = ff_add_f(ff_mul(ff_add(ff_mul(ax, by), ff_neg(ff_mul(ay, bx))), ie), -s2);
    o0h[o] = c0.hi; o0l[o] = c0.lo;
    o1h[o] = c1.hi; o1l[o] = c1.lo;
    o2h[o] = c2.hi; o2l[o] = c2.lo;
  }
  const long long t = G.rc + i0;
  *reinterpret_cast<float4*>(f.p[0] + t) = make_float4(o0h[0], o0h[1], o0h[2], o0h[3]);
  *reinterpret_cast<float4*>(f_lo.p[0] + t) = make_float4(o0l[0], o0l[1], o0l[2], o0l[3]);
  *reinterpret_cast<float4*>(f.p[1] + t) = make_float4(o1h[0], o1h[1], o1h[2], o1h[3]);
  *reinterpret_cast<float4*>(f_lo.p[1] + t) = make_float4(o1l[0], o1l[1], o1l[2], o1l[3]);
  *reinterpret_cast<float4*>(f.p[2] + t) = make_float4(o2h[0], o2h[1], o2h[2], o2h[3]);
  *reinterpret_cast<float4*>(f_lo.p[2] + t) = make_float4(o2l[0], o2l[1], o2l[2], o2l[3]);
}

// Threads on a row's 4-cell groups in k_reduce_va_ff4.
__host__ __device__ inline int va4_lanes(int nx) { return nx > 64 ? 32 : (nx > 32 ? 16 : 8); }

// Partial sums of sum(phi) and of the area density over 4-cell groups; one
// (phi, area) pair per block, as k_reduce_va.  Each warp takes whole x rows
// (row index and plane from one 32-bit division per row), its lanes the
// rows' 4-cell groups.  WITH_G: the Helfrich g of the same cells is formed
// from the same staged stencil and stored as k_helfrich_g_ff4 stores it
// (same operations, same values), saving that kernel's pass over phi.
template <bool WITH_G>
__global__ void __launch_bounds__(256) k_reduce_va_ff4(PhaseParams P, const float* __restrict__ phi,
                                                       const float* __restrict__ phi_lo,
                                                       double* partials, float* __restrict__ g,
                                                       float* __restrict__ g_lo, Scalars* S,
                                                       int init) {
  pdl_begin();
  const int ng = P.nx >> 2;
  const int rows = P.ny * P.nz;
  const int lanes = va4_lanes(P.nx);
  const FF agf{P.ag_hi, P.ag_lo}, awf{P.aw_hi, P.aw_lo};
  CascadeSum cp(0.f), ca(0.f);
  for (int row = (blockIdx.x * kBlock + threadIdx.x) / lanes; row < rows;
       row += gridDim.x * kBlock / lanes)
  for (int gi = threadIdx.x & (lanes - 1); gi < ng; gi += lanes) {
    const int k = row / P.ny, j = row - k * P.ny;
    const Geo4 G = geo4(P, 4 * gi, j, k, false);
    const St4 H = load4(phi, G), L = load4(phi_lo, G);
    float oh[4], ol[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const FF f{e4(H.c, o), e4(L.c, o)};
      auto diff = [&](float ah, float al, float bh, float bl) {
        return ff_add(FF{ah, al}, ff_neg(FF{bh, bl}));
      };
      const FF gx = diff(xp4(H, o), xp4(L, o), xm4(H, o), xm4(L, o));
      const FF gy = diff(e4(H.yp, o), e4(L.yp, o), e4(H.ym, o), e4(L.ym, o));
      const FF gz = diff(e4(H.zp, o), e4(L.zp, o), e4(H.zm, o), e4(L.zm, o));
      const FF g2 = ff_add(ff_add(ff_mul(gx, gx), ff_mul(gy, gy)), ff_mul(gz, gz));
      const FF w = ff_add_f(ff_mul(f, f), -1.f);
      const FF dens = ff_add(ff_mul(g2, agf), ff_mul(ff_mul(w, w), awf));
      cp.add(f.hi);
      cp.add(f.lo);
      ca.add(dens.hi);
      ca.add(dens.lo);
      if constexpr (WITH_G) {
        // g = phi (phi^2 - 1) - eps^2 lap phi, as k_helfrich_g_ff4 (w is its
        // phi^2 - 1)
        const FF r = ff_add(ff_mul(f, w),
                            ff_neg(ff_mul(lap7_ff4(H, L, o), FF{P.e2ih_hi, P.e2ih_lo})));
        oh[o] = r.hi;
        ol[o] = r.lo;
      }
    }
    if constexpr (WITH_G) {
      *reinterpret_cast<float4*>(g + G.rc + 4 * gi) = make_float4(oh[0], oh[1], oh[2], oh[3]);
      *reinterpret_cast<float4*>(g_lo + G.rc + 4 * gi) = make_float4(ol[0], ol[1], ol[2], ol[3]);
    }
  }
  __shared__ double buf[2 * kBlock];
  va_publish((double)cp.hi + (double)cp.lo, (double)ca.hi + (double)ca.lo, buf, partials,
             (long long)P.nx * P.ny * P.nz, S, init);
}

static bool use4(const PhaseParams& P) { return P.nx % 4 == 0 && P.nx >= 8; }
static dim3 grid4(const PhaseParams& P) {
  return dim3((unsigned)((P.nx / 4 + 31) / 32), (unsigned)((P.ny + 7) / 8), (unsigned)P.nz);
}

void launch_phi_update_ff(Ctx& cx, const PhaseParams& P, const float* phi, const float* phi_lo,
                          const float* mu, Comp3<float> psi, Comp3<float> v0, const Scalars* S,
                          float dt, float* out, float* out_lo) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  cx.before(VSV_KCLASS_PHASE);
  if (use4(P))
    launch_k(cx, k_phi_update_ff4, grid4(P), dim3(32, 8), 0, P, phi, phi_lo, mu, psi, v0,
             const_cast<Scalars*>(S), dt, out, out_lo);
  else
    k_phi_update_ff<<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(
        P, phi, phi_lo, mu, psi, v0, const_cast<Scalars*>(S), dt, out, out_lo);
  // phi (two words), mu, psi' (3) read; phi (two words) written
  cx.after(VSV_KCLASS_PHASE, 32.0 * (double)n);
}

void launch_mu_ff(Ctx& cx, const PhaseParams& P, const float* phi, const float* phi_lo, float* g,
                  float* g_lo, float* mu, float* mu_lo, const Scalars* S, bool g_ready) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  if (P.fe_kind == VSV_HELFRICH && !g_ready) {
    cx.before(VSV_KCLASS_PHASE);
    if (use4(P))
      launch_k(cx, k_helfrich_g_ff4, grid4(P), dim3(32, 8), 0, P, phi, phi_lo, g, g_lo);
    else
      k_helfrich_g_ff<<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, phi_lo, g, g_lo);
    cx.after(VSV_KCLASS_PHASE, 16.0 * (double)n);   // phi read, g written (two words each)
  }
  cx.before(VSV_KCLASS_PHASE);
  if (use4(P))
    launch_k(cx, k_mu_ff4, grid4(P), dim3(32, 8), 0, P, phi, phi_lo, g, g_lo, S, mu, mu_lo);
  else
    k_mu_ff<<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, phi_lo, g, g_lo, S, mu,
                                                                       mu_lo);
  // phi (and g for Helfrich) read, mu written, two words each
  cx.after(VSV_KCLASS_PHASE, (P.fe_kind == VSV_HELFRICH ? 24.0 : 16.0) * (double)n);
}

// f = grad phi x grad mu / eta - s_omega in double-word arithmetic from
// phi = hi + lo and mu = hi + lo; written as hi + lo.  The stream vector
// psi' = L^{-2}(-f) is dominated by the small low-wavenumber content of this
// dipole-like source, so FP32 rounding of f would be amplified ~10^3 in psi'.
__global__ void k_source_ff(PhaseParams P, const float* __restrict__ phi, const float* __restrict__ phi_lo,
                            const float* __restrict__ mu, const float* __restrict__ mu_lo,
                            Comp3<float> s_omega, Comp3<float> f, Comp3<float> f_lo) {
  int i, j, k, comp_;
  if (!cell3(P.nx, P.ny, P.nz, i, j, k, comp_)) return;
  const long long t = lin(i, j, k, P.nx, P.ny);
  ScalarView<float> FH{phi, P.nx, P.ny, P.nz, P.zper}, FL{phi_lo, P.nx, P.ny, P.nz, P.zper};
  ScalarView<float> MH{mu, P.nx, P.ny, P.nz, P.zper}, ML{mu_lo, P.nx, P.ny, P.nz, P.zper};
  // raw central differences; (1/2h)^2 / eta is applied once to each
  // component of the cross product
  auto dd = [&](const ScalarView<float>& H, const ScalarView<float>& L, int i1, int j1, int k1, int i0,
                int j0, int k0) {
    const FF a{H(i1, j1, k1), L(i1, j1, k1)}, b{H(i0, j0, k0), L(i0, j0, k0)};
    return ff_add(a, ff_neg(b));
  };
  const FF ax = dd(FH, FL, i + 1, j, k, i - 1, j, k), ay = dd(FH, FL, i, j + 1, k, i, j - 1, k),
           az = dd(FH, FL, i, j, k + 1, i, j, k - 1);
  const FF bx = dd(MH, ML, i + 1, j, k, i - 1, j, k), by = dd(MH, ML, i, j + 1, k, i, j - 1, k),
           bz = dd(MH, ML, i, j, k + 1, i, j, k - 1);
  const FF ie{P.src_hi, P.src_lo};
  const long long jk = j + (long long)k * P.ny;
  const FF c0 = ff_add_f(ff_mul(ff_add(ff_mul(ay, bz), ff_neg(ff_mul(az, by))), ie), -s_omega.p[0][jk]);
  const FF c1 = ff_add_f(ff_mul(ff_add(ff_mul(az, bx), ff_neg(ff_mul(ax, bz))), ie), -s_omega.p[1][jk]);
  const FF c2 = ff_add_f(ff_mul(ff_add(ff_mul(ax, by), ff_neg(ff_mul(ay, bx))), ie), -s_omega.p[2][jk]);
  f.p[0][t] = c0.hi; f_lo.p[0][t] = c0.lo;
  f.p[1][t] = c1.hi; f_lo.p[1][t] = c1.lo;
  f.p[2][t] = c2.hi; f_lo.p[2][t] = c2.lo;
}

void launch_source_ff(Ctx& cx, const PhaseParams& P, const float* phi, const float* phi_lo,
                      const float* mu, const float* mu_lo, Comp3<float> s_omega, Comp3<float> f,
                      Comp3<float> f_lo) {
  cx.before(VSV_KCLASS_PHASE);
  if (use4(P))
    launch_k(cx, k_source_ff4, grid4(P), dim3(32, 8), 0, P, phi, phi_lo, mu, mu_lo, s_omega, f, f_lo);
  else
    k_source_ff<<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, phi_lo, mu, mu_lo,
                                                                         s_omega, f, f_lo);
  // phi, mu read, f (3) written, two words each
  cx.after(VSV_KCLASS_PHASE, 40.0 * (double)((long long)P.nx * P.ny * P.nz));
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }
static unsigned v4_blocks(const Ctx& cx, long long n) {
  const long long want = (n / 4 + kBlock - 1) / kBlock;
  return (unsigned)std::max<long long>(1, std::min<long long>(want, 16LL * cx.sms));
}

void launch_split_ff(Ctx& cx, const double* in, float* hi, float* lo, long long n) {
  cx.before(-1);
  if (aligned16(in) && aligned16(hi) && aligned16(lo))
    k_split_ff_v4<<<v4_blocks(cx, n), kBlock, 0, cx.stream>>>(in, hi, lo, n);
  else
    k_split_ff<<<nblk(n), kBlock, 0, cx.stream>>>(in, hi, lo, n);
  cx.after(-1);
}

void launch_merge_ff(Ctx& cx, const float* hi, const float* lo, double* out, long long n) {
  cx.before(-1);
  if (aligned16(out) && aligned16(hi) && aligned16(lo))
    k_merge_ff_v4<<<v4_blocks(cx, n), kBlock, 0, cx.stream>>>(hi, lo, out, n);
  else
    k_merge_ff<<<nblk(n), kBlock, 0, cx.stream>>>(hi, lo, out, n);
  cx.after(-1);
}

// ---------------------------------------------------------------- launchers
template <class T>
void launch_phi_update(Ctx& cx, const PhaseParams& P, const T* phi, const T* mu, Comp3<T> psi,
                       Comp3<T> v0, const Scalars* S, T dt, T* out) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  cx.before(VSV_KCLASS_PHASE);
  k_phi_update<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, mu, psi, v0, const_cast<Scalars*>(S),
                                                     dt, out);
  cx.after(VSV_KCLASS_PHASE, 6.0 * sizeof(T) * (double)n);   // phi, mu, psi' (3) read, phi written
}

template <class T>
bool launch_reduce_va(Ctx& cx, const PhaseParams& P, const T* phi, const T* phi_lo,
                      double* partials, int nblocks, Scalars* S, int init, float* g, float* g_lo) {
  bool with_g = false;
  const long long rows = (long long)P.ny * P.nz;
  cx.before(VSV_KCLASS_PHASE);
  if constexpr (std::is_same<T, float>::value) {
    if (use4(P)) {
      with_g = g && g_lo;
      const unsigned blocks = row_blocks(va4_lanes(P.nx), rows, nblocks);
      if (with_g)
        launch_k(cx, k_reduce_va_ff4<true>, blocks, kBlock, 0, P, phi, phi_lo, partials, g, g_lo, S,
                 init);
      else
        launch_k(cx, k_reduce_va_ff4<false>, blocks, kBlock, 0, P, phi, phi_lo, partials,
                 (float*)nullptr, (float*)nullptr, S, init);
    }
  }
  if (!std::is_same<T, float>::value || !use4(P)) {
    const unsigned blocks = row_blocks(row_lanes(P.nx), rows, nblocks);
    k_reduce_va<T><<<blocks, kBlock, 0, cx.stream>>>(P, phi, phi_lo, partials, S, init);
  }
  // phi read (two FP32 words, or one FP64); g written (two words)
  cx.after(VSV_KCLASS_PHASE, (with_g ? 16.0 : 8.0) * (double)((long long)P.nx * P.ny * P.nz));
  return with_g;
}

template <class T>
void launch_mu(Ctx& cx, const PhaseParams& P, const T* phi, T* g, T* mu, const Scalars* S) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  if (P.fe_kind == VSV_HELFRICH) {
    cx.before(VSV_KCLASS_PHASE);
    k_helfrich_g<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, g);
    cx.after(VSV_KCLASS_PHASE, 2.0 * sizeof(T) * (double)n);
  }
  cx.before(VSV_KCLASS_PHASE);
  k_mu<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, g, S, mu);
  cx.after(VSV_KCLASS_PHASE, (P.fe_kind == VSV_HELFRICH ? 3.0 : 2.0) * sizeof(T) * (double)n);
}

template <class T>
void launch_source(Ctx& cx, const PhaseParams& P, const T* phi, const T* mu, Comp3<T> s_omega,
                   Comp3<T> f) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  cx.before(VSV_KCLASS_PHASE);
  k_source<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, phi, mu, s_omega, f);
  cx.after(VSV_KCLASS_PHASE, 5.0 * sizeof(T) * (double)n);   // phi, mu read, f (3) written
}

template <class T>
void launch_velocity(Ctx& cx, const PhaseParams& P, Comp3<T> psi, const T* v0, int c, T* v) {
  cx.before(-1);
  k_velocity<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, psi, v0, c, v);
  cx.after(-1);
}

namespace {
template <int C, int OUT>
void velocity_dw(Ctx& cx, const PhaseParams& P, Comp3<float> psi, Comp3<float> psi_lo, const double* v0,
                 float* v, float* v_lo, double* vd) {
  constexpr int A = C == 0 ? 2 : C - 1, B = C == 2 ? 0 : C + 1;
  const double hih = 0.5 * P.inv_h;
  VelScale S;
  S.c1 = (float)hih;
  S.c2 = (float)(hih - (double)S.c1);
  S.c3 = (float)(hih - (double)S.c1 - (double)S.c2);
  const float *ah = psi.p[A], *al = psi_lo.p[A], *bh = psi.p[B], *bl = psi_lo.p[B];
  if (use4(P) && aligned16(v) && aligned16(v_lo) && aligned16(vd))
    k_velocity_dw4<C, OUT><<<grid4(P), dim3(32, 8), 0, cx.stream>>>(P, ah, al, bh, bl, v0, S, v, v_lo, vd);
  else
    k_velocity_dw<C, OUT><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, ah, al, bh, bl, v0, S,
                                                                               v, v_lo, vd);
}
template <int OUT>
void velocity_dw_c(Ctx& cx, const PhaseParams& P, Comp3<float> psi, Comp3<float> psi_lo, const double* v0,
                   int c, float* v, float* v_lo, double* vd) {
  if (c == 0) velocity_dw<0, OUT>(cx, P, psi, psi_lo, v0, v, v_lo, vd);
  else if (c == 1) velocity_dw<1, OUT>(cx, P, psi, psi_lo, v0, v, v_lo, vd);
  else velocity_dw<2, OUT>(cx, P, psi, psi_lo, v0, v, v_lo, vd);
}
}  // namespace

void launch_velocity_dw(Ctx& cx, const PhaseParams& P, Comp3<float> psi, Comp3<float> psi_lo,
                        const double* v0, int c, float* v, float* v_lo, double* v64) {
  cx.before(-1);
  if (v64) velocity_dw_c<kVelF64>(cx, P, psi, psi_lo, v0, c, nullptr, nullptr, v64);
  else if (v_lo) velocity_dw_c<kVelWords>(cx, P, psi, psi_lo, v0, c, v, v_lo, nullptr);
  else velocity_dw_c<kVelF32>(cx, P, psi, psi_lo, v0, c, v, nullptr, nullptr);
  cx.after(-1);
}

template <class T>
void launch_diag(Ctx& cx, const PhaseParams& P, const T* phi, const T* phi_lo, const T* g,
                 const T* g_lo, Comp3<T> vel, Comp3<T> vel_lo, Comp3<T> omega, Comp3<T> om_lo,
                 Comp3<T> psi, Comp3<T> ps_lo, Comp3<const double> psi0_ring,
                 Comp3<const double> v0d, double* partials, int nblocks, double* out) {
  cx.before(-1);
  k_diag_flow<T><<<nblocks, kBlock, 0, cx.stream>>>(P, vel, vel_lo, v0d, partials);
  cx.after(-1);
  cx.before(-1);
  k_diag_state<T><<<nblocks, kBlock, 0, cx.stream>>>(P, phi, phi_lo, g, g_lo, omega, om_lo, psi, ps_lo,
                                                     psi0_ring, partials);
  cx.after(-1);
  cx.before(-1);
  k_diag_finalize<<<13, kBlock, 0, cx.stream>>>(partials, nblocks, out);
  cx.after(-1);
}

template <class T>
void launch_sigma_t(Ctx& cx, const PhaseParams& P, Comp3<T> vel, Comp3<T> vel_lo, T* out) {
  const dim3 grid = grid3(P.nx, P.ny, P.nz, 1);
  const double f = 0.5 * P.inv_h / P.inv_eta;
  cx.before(-1);
  if constexpr (std::is_same<T, float>::value) {
    int fe = 1 << 20;   // out of every range: FP64
    FF fm{1.f, 0.f};
    if (f > 0.0 && std::isfinite(f)) {
      const double m = 2.0 * std::frexp(f, &fe);   // f = m 2^(fe - 1), 1 <= m < 2
      --fe;
      fm.hi = (float)m;
      fm.lo = (float)(m - (double)fm.hi);
    }
    k_sigma_t_dw<<<grid, block3(), 0, cx.stream>>>(P, vel, vel_lo, f, fm, fe, out);
  } else {
    k_sigma_t<<<grid, block3(), 0, cx.stream>>>(P, vel, vel_lo, f, out);
  }
  cx.after(-1);
}

template <class T>
void launch_stress_profile(Ctx& cx, const PhaseParams& P, const T* vx, const T* vx_lo, double* sums,
                           double* out) {
  // chunks of planes so that the rows fill the SMs, of at least 2,048 cells a row
  // (below, the second launch costs more than it saves); sums holds ny nz doubles
  const long long cells = (long long)P.nx * P.nz;
  const int want = (int)std::min<long long>(4 * cx.sms / std::max(1, P.ny), cells / 2048);
  const int chunks = std::max(1, std::min(P.nz, want));
  const int kchunk = (P.nz + chunks - 1) / chunks, n = (P.nz + kchunk - 1) / kchunk;
  const double scale = 0.5 * P.inv_h / P.inv_eta / (double)cells;
  cx.before(-1);
  k_stress_profile<T><<<dim3(P.ny, n), kBlock, 0, cx.stream>>>(P, vx, vx_lo, kchunk, n > 1 ? 1.0 : scale,
                                                               n > 1 ? sums : out);
  cx.after(-1);
  if (n == 1) return;
  cx.before(-1);
  k_profile_total<<<(P.ny + 127) / 128, 128, 0, cx.stream>>>(sums, P.ny, n, scale, out);
  cx.after(-1);
}

template <class Tin, class Tout>
void launch_convert(Ctx& cx, const Tin* in, Tout* out, long long n) {
  cx.before(-1);
  k_convert<Tin, Tout><<<nblk(n), kBlock, 0, cx.stream>>>(in, out, n);
  cx.after(-1);
}

template <class T>
void launch_full_field(Ctx& cx, const PhaseParams& P, const T* pert, const T* lo, const double* tab,
                       int ring, T* out) {
  cx.before(-1);
  k_full_field<T><<<grid3(P.nx, P.ny, P.nz, 1), block3(), 0, cx.stream>>>(P, pert, lo, tab, ring, out);
  cx.after(-1);
}

template <class T>
void launch_scale_copy(Ctx& cx, const T* in, T* out, long long n, double a) {
  cx.before(-1);
  k_scale_copy<T><<<nblk(n), kBlock, 0, cx.stream>>>(in, out, n, (T)a);
  cx.after(-1);
}

void launch_duct_ring(Ctx& cx, int ny, int nz, double h, const double* u0, const double* chi,
                      double* omy, double* omz, double* psy, double* psz) {
  const int m = ny > nz ? ny : nz;
  cx.before(-1);
  k_duct_ring<<<nblk(m), kBlock, 0, cx.stream>>>(ny, nz, h, u0, chi, omy, omz, psy, psz);
  cx.after(-1);
}

void launch_ring_boundary_rhs(Ctx& cx, int ny, int nz, double h, const double* ring, double scale,
                              const double* in, double* out) {
  cx.before(-1);
  k_ring_rhs<<<nblk((long long)ny * nz), kBlock, 0, cx.stream>>>(ny, nz, h, ring, scale, in, out);
  cx.after(-1);
}

void launch_ring_fill_interior(Ctx& cx, int ny, int nz, const double* interior, double* ring) {
  cx.before(-1);
  k_ring_fill<<<nblk((long long)ny * nz), kBlock, 0, cx.stream>>>(ny, nz, interior, ring);
  cx.after(-1);
}

void launch_base_derived(Ctx& cx, int ny, int nz, int zper, double h, const double* om[3],
                         const double* ps[3], double* v0[3], double* s_om[3], double* s_ps[3]) {
  Comp3<const double> O{{om[0], om[1], om[2]}}, Pp{{ps[0], ps[1], ps[2]}};
  Comp3<double> V{{v0[0], v0[1], v0[2]}}, SO{{s_om[0], s_om[1], s_om[2]}},
      SP{{s_ps[0], s_ps[1], s_ps[2]}};
  cx.before(-1);
  k_base_derived<<<nblk((long long)ny * nz), kBlock, 0, cx.stream>>>(ny, nz, zper, h, O, Pp, V, SO, SP);
  cx.after(-1);
}

double device_max_abs(Ctx& cx, const double* x, long long n, double* scratch) {
  cx.before(-1);
  k_max_abs<<<1, 1024, 0, cx.stream>>>(x, n, scratch);
  cx.after(-1);
  double h = 0.0;
  cudaMemcpyAsync(&h, scratch, sizeof(double), cudaMemcpyDeviceToHost, cx.stream);
  cudaStreamSynchronize(cx.stream);
  return h;
}

void launch_fill(Ctx& cx, double* x, long long n, double v) {
  cx.before(-1);
  k_fill<<<nblk(n), kBlock, 0, cx.stream>>>(x, n, v);
  cx.after(-1);
}

#define VSV_INST(T)                                                                               \
  template void launch_phi_update<T>(Ctx&, const PhaseParams&, const T*, const T*, Comp3<T>,      \
                                     Comp3<T>, const Scalars*, T, T*);                            \
  template bool launch_reduce_va<T>(Ctx&, const PhaseParams&, const T*, const T*, double*, int,   \
                                    Scalars*, int, float*, float*);                               \
  template void launch_mu<T>(Ctx&, const PhaseParams&, const T*, T*, T*, const Scalars*);         \
  template void launch_source<T>(Ctx&, const PhaseParams&, const T*, const T*, Comp3<T>,          \
                                 Comp3<T>);                                                       \
  template void launch_diag<T>(Ctx&, const PhaseParams&, const T*, const T*, const T*, const T*,  \
                               Comp3<T>, Comp3<T>, Comp3<T>, Comp3<T>, Comp3<T>, Comp3<T>,        \
                               Comp3<const double>, Comp3<const double>, double*, int, double*);  \
  template void launch_sigma_t<T>(Ctx&, const PhaseParams&, Comp3<T>, Comp3<T>, T*);              \
  template void launch_stress_profile<T>(Ctx&, const PhaseParams&, const T*, const T*, double*,   \
                                         double*);                                                \
  template void launch_full_field<T>(Ctx&, const PhaseParams&, const T*, const T*, const double*,  \
                                     int, T*);                                                    \
  template void launch_scale_copy<T>(Ctx&, const T*, T*, long long, double);
VSV_INST(float)
VSV_INST(double)
#undef VSV_INST
// (the mixed path's velocity is launch_velocity_dw's)
template void launch_velocity<double>(Ctx&, const PhaseParams&, Comp3<double>, const double*, int, double*);
template void launch_convert<float, double>(Ctx&, const float*, double*, long long);
template void launch_convert<double, float>(Ctx&, const double*, float*, long long);
template void launch_convert<float, float>(Ctx&, const float*, float*, long long);
template void launch_convert<double, double>(Ctx&, const double*, double*, long long);

}  // namespace vsv
