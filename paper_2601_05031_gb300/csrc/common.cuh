// Shared device/host definitions of the vorticity--stream-vector library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

namespace vsv {

constexpr int kMaxLevels = 16;
constexpr int kBlock = 256;

// One grid level of a Poisson problem (the fine grid is level 0).
// Dirichlet walls sit on the ghost nodes of the fine grid; on a coarse level
// l the wall lies between the ghost and the first cell, and the ghost value
// is the linear extrapolation through zero at the wall:
//   ghost = -alpha_l * (adjacent cell),  alpha_l = (2^l - 1) / (2^l + 1).
// A level may carry a diagonal shift: the operator is L_h - s (the
// backward-Euler vorticity step of the inertial variant), which adds
// sh2 = s h_l^2 to the diagonal coefficient 2 d + alpha * nwall.
struct Level {
  int n[3];          // nx, ny, nz
  int per[3];        // 1 = periodic axis
  int act[3];        // 0 for a periodic axis of extent 1 (no coupling)
  double alpha;      // Dirichlet closure coefficient (0 on the fine level)
  double inv_h2;     // 1 / h_l^2
  float alphaf;      // the same in FP32 (FP32 kernels never touch FP64 units)
  float inv_h2f;
  double sh2;        // s h_l^2 (0: plain Poisson)
  float sh2f;
  // 1 / (2 d + alpha * nwall + sh2) for nwall = 0..6 wall neighbours: the
  // smoothers multiply by these instead of dividing (same table in every
  // sweep kernel)
  float rcf[7];
  double rcd[7];
  // the diagonal coefficient 2 d + alpha * nwall + sh2 itself, rounded to
  // each type: every residual kernel reads it instead of forming it per cell
  // (on the FP64 path a conversion, an FMA and an addition on units that do
  // two operations per clock and SM)
  float cf[7];
  double cd[7];
  // the diagonal coefficient 2 d + alpha * nwall + sh2 as an FP32 pair
  // (hi + lo) for the exact defect
  float cdh[7], cdl[7];
  __host__ __device__ long long cells() const { return (long long)n[0] * n[1] * n[2]; }
};

template <class T> __host__ __device__ inline T lv_rc(const Level& L, int nwall);
template <> __host__ __device__ inline float lv_rc<float>(const Level& L, int nwall) { return L.rcf[nwall]; }
template <> __host__ __device__ inline double lv_rc<double>(const Level& L, int nwall) { return L.rcd[nwall]; }

template <class T> __host__ __device__ inline T lv_coef(const Level& L, int nwall);
template <> __host__ __device__ inline float lv_coef<float>(const Level& L, int nwall) { return L.cf[nwall]; }
template <> __host__ __device__ inline double lv_coef<double>(const Level& L, int nwall) { return L.cd[nwall]; }

template <class T> __host__ __device__ inline T lv_alpha(const Level& L);
template <> __host__ __device__ inline float lv_alpha<float>(const Level& L) { return L.alphaf; }
template <> __host__ __device__ inline double lv_alpha<double>(const Level& L) { return L.alpha; }
template <class T> __host__ __device__ inline T lv_sh2(const Level& L);
template <> __host__ __device__ inline float lv_sh2<float>(const Level& L) { return L.sh2f; }
template <> __host__ __device__ inline double lv_sh2<double>(const Level& L) { return L.sh2; }
template <class T> __host__ __device__ inline T lv_ih2(const Level& L);
template <> __host__ __device__ inline float lv_ih2<float>(const Level& L) { return L.inv_h2f; }
template <> __host__ __device__ inline double lv_ih2<double>(const Level& L) { return L.inv_h2; }

// Up to three components processed by one launch (gridDim.y = component).
template <class T>
struct Comp3 {
  T* p[3];
  // p[c] without a runtime index into the array (a kernel parameter indexed
  // at run time is copied to local memory first)
  __host__ __device__ __forceinline__ T* at(int c) const {
    return c == 0 ? p[0] : (c == 1 ? p[1] : p[2]);
  }
};

// Correctly rounded a b + c and a b in T, never contracted or split by the
// compiler: the kernels that must agree bit for bit share formulas written
// with these.
template <class T>
__device__ __forceinline__ T fma_t(T a, T b, T c) {
  if constexpr (sizeof(T) == 4) return __fmaf_rn(a, b, c);
  else return __fma_rn(a, b, c);
}
template <class T>
__device__ __forceinline__ T mul_t(T a, T b) {
  if constexpr (sizeof(T) == 4) return __fmul_rn(a, b);
  else return __dmul_rn(a, b);
}

// Prolongation increment of one fine cell (cell-centred trilinear, weights
// 3/4 and 1/4 per axis).  The arguments are the (x-centre, x-neighbour) pairs
// of coarse values, already multiplied by their boundary factors, for the
// (centre plane, centre row), (centre plane, neighbour row), (neighbour
// plane, centre row) and (neighbour plane, neighbour row).  Every
// prolongation kernel calls this, or its two parts where cells share the pairs,
// so they agree bit for bit.
template <class T>
__device__ __forceinline__ T prolong_pair(T c, T x) {   // 3/4 c + 1/4 x
  return fma_t((T)0.75, c, mul_t((T)0.25, x));
}
template <class T>
__device__ __forceinline__ T prolong_sum(T a, T b, T c, T d) {   // of the four pairs
  return fma_t((T)0.0625, d, fma_t((T)0.1875, c, fma_t((T)0.1875, b, mul_t((T)0.5625, a))));
}
template <class T>
__device__ __forceinline__ T prolong_value(T aC, T aX, T bC, T bX, T cC, T cX, T dC, T dX) {
  return prolong_sum(prolong_pair(aC, aX), prolong_pair(bC, bX), prolong_pair(cC, cX),
                     prolong_pair(dC, dX));
}

// b - L x of one cell: (neighbour sum s) - coef x, times 1 / h^2, from b;
// shared by every residual and restriction kernel.
template <class T>
__device__ __forceinline__ T resid_value(T b, T s, T coef, T x, T ih2) {
  return fma_t(-fma_t(-coef, x, s), ih2, b);
}

// Weighted red-black update of one cell (red-black SOR smoothing; an
// over-relaxed smoother contracts a multigrid V-cycle faster):
// x <- x + omega (gs - x) with the Gauss-Seidel value gs = t rc, where
// t = (neighbour sum) - b h^2 and rc = 1 / diagonal, evaluated as
// t (omega rc) + (1 - omega) x in one fused multiply-add.  Every sweep
// kernel forms t with nb_term and updates through relax, with the same
// rounded constants wrc = omega rc and c1 = 1 - omega, so the fused and
// per-colour sweeps agree bit for bit; omega = 1 (c1 = 0, wrc = rc) gives
// the Gauss-Seidel value t rc itself.
template <class T>
__device__ __forceinline__ T nb_term(T s, T b, T h2) {
  if constexpr (sizeof(T) == 4) return __fmaf_rn(-b, h2, s);
  else return __fma_rn(-b, h2, s);
}
template <class T>
__device__ __forceinline__ T relax(T x, T t, T wrc, T c1) {
  if constexpr (sizeof(T) == 4) return __fmaf_rn(t, wrc, __fmul_rn(c1, x));
  else return __fma_rn(t, wrc, __dmul_rn(c1, x));
}
template <class T>
__device__ __forceinline__ T wscale(T omega, T rc) {
  if constexpr (sizeof(T) == 4) return __fmul_rn(omega, rc);
  else return __dmul_rn(omega, rc);
}

// The GPU's global timer in nanoseconds (bounds of every wait on other
// threads, CTAs or copies).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// First statement of every kernel that launch_k() launches.  Under
// programmatic stream serialisation a kernel can be scheduled while the
// kernel before it in the stream is still running: griddepcontrol.wait
// blocks until every prerequisite grid has completed and its memory
// operations are visible (it returns at once for a plain launch), so nothing
// before it may touch global memory.  launch_dependents then lets the next
// kernel of the stream be scheduled once every CTA of this one has got here;
// its CTAs take SM slots that this kernel's last wave leaves free and wait
// in the same way.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Right-hand side b = beta * B[c] + S[j + k * ny] (beta 1 or -1; S may be null).
template <class T>
struct Rhs3 {
  const T* B[3];
  const T* S[3];
  T beta;
  __host__ __device__ __forceinline__ const T* b_at(int c) const {
    return c == 0 ? B[0] : (c == 1 ? B[1] : B[2]);
  }
  __host__ __device__ __forceinline__ const T* s_at(int c) const {
    return c == 0 ? S[0] : (c == 1 ? S[1] : S[2]);
  }
};

// Device scalars written by reductions and read by later kernels.
struct Scalars {
  double V, A, V0, A0;
  double lambda_v, gamma_a;
  double k_vol, k_area, eps;   // copies of the penalty parameters
  double h3;
  float lambda_vf, gamma_af;   // FP32 copies read by the FP32 kernels
  int nonfinite;
  unsigned ticket;             // CTAs of a norm reduction that have stored their sums
};

// ---------------------------------------------------------------- device helpers
__host__ __device__ inline long long lin(int i, int j, int k, int nx, int ny) {
  return ((long long)k * ny + j) * nx + i;
}

// Cell-parallel launches use a 3-D grid: x threads along a row, y blocks
// over rows, z blocks over (plane, component) -- no per-cell division.
constexpr int kBX = 64, kBY = 4;
inline dim3 grid3(int nx, int ny, int nz, int ncomp) {
  return dim3((unsigned)((nx + kBX - 1) / kBX), (unsigned)((ny + kBY - 1) / kBY),
              (unsigned)(nz * ncomp));
}
inline dim3 block3() { return dim3(kBX, kBY, 1); }
__device__ __forceinline__ bool cell3(int nx, int ny, int nz, int& i, int& j, int& k, int& comp) {
  i = blockIdx.x * blockDim.x + threadIdx.x;
  j = blockIdx.y * blockDim.y + threadIdx.y;
  comp = ((int)blockIdx.z >= nz) + ((int)blockIdx.z >= 2 * nz);   // at most three components
  k = (int)blockIdx.z - comp * nz;
  return i < nx && j < ny;
}

// Knuth's TwoSum: s + e == a + b exactly (round-to-nearest).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Double-word ("float-float") value hi + lo with |lo| <= ulp(hi) / 2, built
// from the error-free transforms TwoSum (Knuth), Fast2Sum (Dekker) and
// TwoProd by FMA; the sloppy add / multiply of Joldes, Muller and Popescu
// (2017) give a relative error of a few 2^-44.
struct FF {
  float hi, lo;
};

__device__ __forceinline__ FF fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_from(float a) { return FF{a, 0.f}; }
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return fast_two_sum(s, e);
}
__device__ __forceinline__ FF ff_add_f(FF a, float b) {
  float s, e;
  two_sum(a.hi, b, s, e);
  return fast_two_sum(s, __fadd_rn(e, a.lo));
}
__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.hi, -a.lo}; }
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
  return fast_two_sum(p, e);
}
__device__ __forceinline__ FF ff_mul_f(FF a, float b) {
  const float p = __fmul_rn(a.hi, b);
  const float e = __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p));
  return fast_two_sum(p, e);
}
__device__ __forceinline__ float ff_round(FF a) { return __fadd_rn(a.hi, a.lo); }

// (double)x, exactly, by integer operations: the conversion instruction runs on
// the FP64 units, which do two operations per clock and SM, and takes as long
// there as the addition it feeds.  A subnormal is scaled up first (exactly).
__device__ __forceinline__ double f2d(float x) {
  const bool tiny = (__float_as_uint(x) & 0x7f800000u) == 0u;
  const unsigned u = __float_as_uint(tiny ? x * 16777216.f : x), e = u & 0x7f800000u;
  const unsigned bias = e == 0x7f800000u ? 0x70000000u : (tiny ? 0x36800000u : 0x38000000u);
  return __hiloint2double((int)((u & 0x80000000u) | (e ? ((u & 0x7fffffffu) >> 3) + bias : 0u)),
                          (int)(u << 29));
}

// Cascaded (compensated) summation accumulator, Ogita-Rump-Oishi "Sum2":
// the running sum is kept as hi + lo with every rounding error of hi
// collected in lo.
struct CascadeSum {
  float hi, lo;
  __device__ __forceinline__ CascadeSum(float a) : hi(a), lo(0.f) {}
  __device__ __forceinline__ void add(float t) {
    float s, e;
    two_sum(hi, t, s, e);
    hi = s;
    lo = __fadd_rn(lo, e);
  }
  // exact product of a float by a small integer constant (error term by FMA)
  __device__ __forceinline__ void add_scaled(float c, float x) {
    float p = __fmul_rn(c, x);
    float pe = __fmaf_rn(c, x, -p);
    add(p);
    lo = __fadd_rn(lo, pe);
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(hi, lo); }
};

// Two FP32 numbers in one register pair.  The packed operations round each like
// the scalar one and take one issue slot for two results (the FP32 units' rate is
// the same: 37 T operations/s either way), which is what the double-word kernels
// run short of.  The functions below are the scalar ones above, term for term, on
// two cells at a time.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ void f2_get(F2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 neg2(F2 a) {
  float x, y;
  f2_get(a, x, y);
  return f2(-x, -y);
}
// Scalar products: a packed one is contracted with an addition that follows it
// (seen in the error words of a TwoSum), a scalar one is not.
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  float a0, a1, b0, b1;
  f2_get(a, a0, a1);
  f2_get(b, b0, b1);
  return f2(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}
__device__ __forceinline__ void two_sum(F2 a, F2 b, F2& s, F2& e) {
  s = add2(a, b);
  const F2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

struct CascadeSum2 {
  F2 hi, lo;
  __device__ __forceinline__ CascadeSum2(F2 a) : hi(a), lo(f2(0.f)) {}
  __device__ __forceinline__ void add(F2 t) {
    F2 s, e;
    two_sum(hi, t, s, e);
    hi = s;
    lo = add2(lo, e);
  }
  __device__ __forceinline__ void add_scaled(F2 c, F2 x) {
    const F2 p = mul2(c, x);
    const F2 pe = fma2(c, x, neg2(p));
    add(p);
    lo = add2(lo, pe);
  }
};

}  // namespace vsv
