// Two-sweep passes of the multigrid V-cycle (FP32 storage): the whole of a
// level's pre-smoothing (two red-black sweeps from e = 0, optionally the
// residual restricted to the next level) and the whole of its
// post-smoothing (prolongation, two red-black sweeps, optionally the update
// of the double-word iterate), each as one launch.
//
// What they replace: one launch per sweep (two per sweep on levels without
// tiles), one per transfer and one zero fill, eleven launches of a few
// microseconds each that the small levels are bound by.
//
// A CTA owns a block of 32 x 8 x 8 cells and works on a window with a
// four-cell halo around it, all of whose planes it holds in shared memory:
// every half-sweep runs over the whole window at once, with one barrier
// after it, so a launch has five or six dependent phases instead of the
// dozens a march along z has.  A half-sweep is valid one cell less far from
// the block's edge, so the halo of four serves two sweeps and the residual
// (or the prolonged values); it is recomputed, not exchanged, and CTAs share
// nothing.
//
// Colours.  A plane is split by colour ((i + j + k) & 1) into two arrays of
// half the row length, in which the six neighbours of a cell are all in the
// other colour's arrays: y and z neighbours at the cell's own index, the x
// neighbours at its own index and one beside it.  So every operand of four
// cells of a colour is one 128-bit load of consecutive words, and the offset
// of a thread's group is four times its index within the plane.
//
// Measured (three components, GB300): 64 x 32 x 32 cells 7 + 10 us instead of
// 27 + 25 us level by level, a step at 128 x 64 x 64 cells 852 -> 740 us.  Bound
// by instruction issue (0.35 per clock and scheduler; 14 k and 19 k warp
// instructions per block, 40 % of them in the halo) and, on a level of few
// blocks, by the latency of the five or six phases.  The same passes as a
// march along z (a ring of planes, four barriers a plane) took 12 + 20 us at
// 64 x 32 x 32; on 256 x 128 x 128 cells 79 + 166 us against the 88 + 107 us of
// the fused sweeps and tiled transfers, which large levels therefore keep.
//
// Arithmetic: rb updates, residuals and prolongation go through nb_term /
// relax / resid_value / prolong_pair / prolong_sum with the sums in the order of
// the per-colour kernels, so the results are theirs bit for bit.
#include <algorithm>

#include "tile.cuh"

namespace vsv {

namespace {

constexpr int kHalo = 4;
constexpr int kPX = 32, kPY = 8, kPZ = 8;            // the block
constexpr int kG = (kPX + 2 * kHalo) / 8;            // 8-column groups per window row
constexpr int kRows = kPY + 2 * kHalo, kPlanes = kPZ + 2 * kHalo;
constexpr int kHW = 4 * kG;                          // row length of one colour
constexpr int kItems = kG * kRows;                   // groups per window plane
constexpr int kThr = 8 * kItems;                     // threads: two planes' groups each
constexpr int kPS = kThr / kItems, kNP = kPlanes / kPS;
constexpr int kCol = kRows * kHW, kX = 2 * kCol;     // one colour of a plane, a plane (floats)
constexpr int kColR = (kRows - 2) * kHW, kR = 2 * kColR;   // rhs planes reach one cell less far
constexpr int kCRows = kPY / 2 + 6, kCPlanes = kPZ / 2 + 6;   // coarse rows and planes of the window
constexpr int kPW = 2 * kHW;                         // x-interpolated coarse row (fine columns)
constexpr int kPad = 4;                              // the left neighbour of the first word
static_assert(kCRows * kCPlanes * kG <= kThr, "one coarse item per thread");
constexpr size_t kSmemPre = sizeof(float) * (kPad + kPlanes * kX + (kPlanes - 2) * kR + kPad);
constexpr size_t kSmemRst = kSmemPre + sizeof(float) * 4 * 4 * (kPX / 4) * (kPY / 2) * (kPZ / 2);
constexpr size_t kSmemPost = kSmemPre + sizeof(float) * kCRows * kCPlanes * kPW;

struct PassGeom {
  int nx, ny, nz, per_y, per_z;
  int ntx;
  int cnx, cny, cnz;          // coarse extents
  float w0, w1, w2;           // omega / diagonal with 0, 1, 2 wall neighbours
  float d0, d1, d2;           // the diagonal itself
  float h2, c1, ih2, malpha;  // 1 - omega; 1 / h^2; - alpha of the coarse level
};

__device__ __forceinline__ float pick3(float a, float b, float c, int n) {
  return n == 0 ? a : (n == 1 ? b : c);
}
// i mod n: one step for all but extents shorter than a window (an integer
// division costs more than the rest of a group's set-up)
__device__ __forceinline__ int mod_(int i, int n) {
  if (i < 0) i += n;
  else if (i >= n) i -= n;
  if ((unsigned)i < (unsigned)n) return i;
  i %= n;
  return i < 0 ? i + n : i;
}
__device__ __forceinline__ float4 l4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float2 l2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void s4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// Half-sweep of four cells of one colour.  oc: the other colour at this
// group in the same plane, om / op in the planes below and above, par the column parity of this colour in the row.
__device__ __forceinline__ float4 half_sweep(const float* oc, const float* om, const float* op, float4 own,
                                             float4 b, int par, float w, float h2, float c1) {
  const float4 o = l4(oc), u = l4(oc - kHW), d = l4(oc + kHW), m = l4(om), p = l4(op);
  const float e = oc[par ? 4 : -1];
  float4 r;
  r.x = relax(own.x, nb_term(((o.x + (par ? o.y : e)) + (u.x + d.x)) + (m.x + p.x), b.x, h2), w, c1);
  r.y = relax(own.y, nb_term(((o.y + (par ? o.z : o.x)) + (u.y + d.y)) + (m.y + p.y), b.y, h2), w, c1);
  r.z = relax(own.z, nb_term(((o.z + (par ? o.w : o.y)) + (u.z + d.z)) + (m.z + p.z), b.z, h2), w, c1);
  r.w = relax(own.w, nb_term(((o.w + (par ? e : o.z)) + (u.w + d.w)) + (m.w + p.w), b.w, h2), w, c1);
  return r;
}

// first half-sweep from e = 0: the scaled rhs alone
__device__ __forceinline__ float4 half_sweep_zero(float4 b, float w, float h2, float c1) {
  return make_float4(relax(0.f, nb_term(0.f, b.x, h2), w, c1), relax(0.f, nb_term(0.f, b.y, h2), w, c1),
                     relax(0.f, nb_term(0.f, b.z, h2), w, c1), relax(0.f, nb_term(0.f, b.w, h2), w, c1));
}

// eight columns (a, b) <-> the two colours; par: column parity of `c`
__device__ __forceinline__ void split8(float4 a, float4 b, int par, float4& c, float4& other) {
  const float4 ev = make_float4(a.x, a.z, b.x, b.z), od = make_float4(a.y, a.w, b.y, b.w);
  c = par ? od : ev;
  other = par ? ev : od;
}
__device__ __forceinline__ void join8(float4 c, float4 other, int par, float4& a, float4& b) {
  const float4 ev = par ? other : c, od = par ? c : other;
  a = make_float4(ev.x, od.x, ev.y, od.y);
  b = make_float4(ev.z, od.z, ev.w, od.w);
}

// What a thread knows about its group of eight window columns (the same row
// and columns in each of its planes).
struct Item {
  int row, pl, off, j;       // window row, first window plane, float offset in a colour, global row
  bool in, st_a, st_b;       // row in the domain; stores its two float4
  int ga, gb;                // offsets of its two float4 within a global plane
  int yw;
  __device__ __forceinline__ void init(const PassGeom& G, int x0, int y0) {
    pl = threadIdx.x / kItems;
    const int t = threadIdx.x - pl * kItems;
    row = t / kG;
    const int g = t - row * kG;
    off = 4 * t;
    j = y0 - kHalo + row;
    in = G.per_y || (j >= 0 && j < G.ny);
    const int jw = G.per_y ? mod_(j, G.ny) : (in ? j : 0);
    const int xa = x0 - kHalo + 8 * g, xb = xa + 4;
    ga = jw * G.nx + mod_(xa, G.nx);
    gb = jw * G.nx + mod_(xb, G.nx);
    const bool own = in && row >= kHalo && row < kHalo + kPY && j < G.ny;
    st_a = own && g >= 1 && xa < G.nx;
    st_b = own && g < kG - 1 && xb < G.nx;
    yw = G.per_y ? 0 : (j == 0) + (j == G.ny - 1);
  }
  // in the domain and at least d rows inside the window
  __device__ __forceinline__ bool inner(int d) const { return in && row >= d && row < kRows - d; }
};

}  // namespace

// Pre-smoothing: E <- two red-black sweeps for L e = R from e = 0; RESTRICT:
// also RC <- the residual averaged onto the next level.
template <bool RESTRICT>
__global__ void __launch_bounds__(kThr, 2)
k_pre_pass(const __grid_constant__ PassGeom G, Comp3<float> R, Comp3<float> E, Comp3<float> RC) {
  pdl_begin();
  extern __shared__ float4 smem_pp[];
  float* const X = reinterpret_cast<float*>(smem_pp) + kPad;
  float* const B = X + kPlanes * kX - kR - kHW;   // rhs: window planes and rows from 1 on
  const int comp = blockIdx.z;
  const float* __restrict__ rhs = R.at(comp);
  float* __restrict__ e = E.at(comp);
  const int x0 = (blockIdx.x % G.ntx) * kPX, y0 = (blockIdx.x / G.ntx) * kPY, z0 = blockIdx.y * kPZ;
  Item I;
  I.init(G, x0, y0);
  const float w0 = pick3(G.w0, G.w1, G.w2, I.yw), w1 = pick3(G.w0, G.w1, G.w2, I.yw + 1);
  const float h2 = G.h2, c1 = G.c1;
  const long long plane_n = (long long)G.nx * G.ny;
  auto ghost = [&](int k) { return !G.per_z && (k < 0 || k >= G.nz); };
  auto wgt = [&](int k) { return !G.per_z && (k == 0 || k == G.nz - 1) ? w1 : w0; };
  {   // rhs in; red 1 (the scaled rhs); zeros on ghost cells
    float4 A[kNP], Bv[kNP];
#pragma unroll
    for (int m = 0; m < kNP; ++m) {
      const int k = z0 - kHalo + I.pl + kPS * m;
      A[m] = Bv[m] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (I.in && !ghost(k)) {
        const float* p = rhs + (long long)(G.per_z ? mod_(k, G.nz) : k) * plane_n;
        A[m] = l4(p + I.ga);
        Bv[m] = l4(p + I.gb);
      }
    }
#pragma unroll
    for (int m = 0; m < kNP; ++m) {
      const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
      float* x = X + pi * kX + I.off;
      float4 r, b;
      split8(A[m], Bv[m], (I.j + k) & 1, r, b);
      if (I.row >= 1 && I.row < kRows - 1 && pi >= 1 && pi < kPlanes - 1) {
        s4(B + pi * kR + I.off, r);
        s4(B + pi * kR + kColR + I.off, b);
      }
      if (I.in && !ghost(k)) {
        s4(x, half_sweep_zero(r, wgt(k), h2, c1));
      } else {
        s4(x, make_float4(0.f, 0.f, 0.f, 0.f));
        s4(x + kCol, make_float4(0.f, 0.f, 0.f, 0.f));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // black 1
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 1 && pi < kPlanes - 1 && I.inner(1) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      s4(x + kCol, half_sweep(x, x - kX, x + kX, make_float4(0.f, 0.f, 0.f, 0.f),
                              l4(B + pi * kR + kColR + I.off), 1 - ((I.j + k) & 1), wgt(k), h2, c1));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // red 2
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 2 && pi < kPlanes - 2 && I.inner(2) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      s4(x, half_sweep(x + kCol, x + kCol - kX, x + kCol + kX, l4(x), l4(B + pi * kR + I.off),
                       (I.j + k) & 1, wgt(k), h2, c1));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // black 2; the block's cells are then finished
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 3 && pi < kPlanes - 3 && I.inner(3) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      const int par = (I.j + k) & 1;
      const float4 v = half_sweep(x, x - kX, x + kX, l4(x + kCol), l4(B + pi * kR + kColR + I.off),
                                  1 - par, wgt(k), h2, c1);
      if (RESTRICT) s4(x + kCol, v);
      if (pi >= kHalo && pi < kHalo + kPZ && k < G.nz) {
        float4 a, b;
        join8(l4(x), v, par, a, b);
        float* dst = e + (long long)k * plane_n;
        if (I.st_a) s4(dst + I.ga, a);
        if (I.st_b) s4(dst + I.gb, b);
      }
    }
  }
  if constexpr (RESTRICT) {
    __syncthreads();
    // residuals of two coarse cells' children in one fine row each (window
    // half-columns i2, i2 + 1; all four planes-and-rows of a coarse row in
    // parallel), then their sums in the children's order: plane by plane, row
    // by row, in x order
    constexpr int kQ = kPX / 4, kRP = kPY / 2, kCoarse = kQ * kRP * (kPZ / 2);
    static_assert(4 * kCoarse <= kThr, "one residual item per thread");
    float4* const S = reinterpret_cast<float4*>(X + kPlanes * kX + (kPlanes - 2) * kR + kPad);
    {
      const int t = threadIdx.x % kCoarse, hk = threadIdx.x / kCoarse;
      const int kc = t / (kQ * kRP), rp = (t / kQ) % kRP, i2 = 2 + 2 * (t % kQ);
      if (hk < 4) {
        const int pi = kHalo + 2 * kc + (hk >> 1), row = kHalo + 2 * rp + (hk & 1);
        const int jj = y0 - kHalo + row, k = z0 - kHalo + pi, o = row * kHW + i2;
        const int par = (jj + k) & 1;      // column parity of the red cells
        const int nw = (G.per_y ? 0 : (jj == 0) + (jj == G.ny - 1)) +
                       (G.per_z ? 0 : (k == 0) + (k == G.nz - 1));
        const float dg = pick3(G.d0, G.d1, G.d2, nw);
        float res[2][2];   // [colour][cell]
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float* oc = X + pi * kX + (1 - c) * kCol + o;   // the other colour
          const int pc = c ? 1 - par : par;
          const float2 v = l2(oc), u = l2(oc - kHW), d = l2(oc + kHW), m = l2(oc - kX), p = l2(oc + kX);
          const float2 own = l2(X + pi * kX + c * kCol + o), b = l2(B + pi * kR + c * kColR + o);
          const float x = oc[pc ? 2 : -1];
          res[c][0] = resid_value(b.x, ((v.x + (pc ? v.y : x)) + (u.x + d.x)) + (m.x + p.x), dg, own.x,
                                  G.ih2);
          res[c][1] = resid_value(b.y, ((v.y + (pc ? x : v.x)) + (u.y + d.y)) + (m.y + p.y), dg, own.y,
                                  G.ih2);
        }
        S[hk * kCoarse + t] = par ? make_float4(res[1][0], res[0][0], res[1][1], res[0][1])
                                  : make_float4(res[0][0], res[1][0], res[0][1], res[1][1]);
      }
    }
    __syncthreads();
    const int t = threadIdx.x, kc = t / (kQ * kRP), rp = (t / kQ) % kRP;
    const int cK = (z0 >> 1) + kc, cJ = (y0 >> 1) + rp, cI = (x0 >> 1) + 2 * (t % kQ);
    if (t < kCoarse && cK < G.cnz && cJ < G.cny && cI < G.cnx) {
      float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
      for (int hk = 0; hk < 4; ++hk) {
        const float4 r = S[hk * kCoarse + t];
        acc0 += r.x; acc0 += r.y;
        acc1 += r.z; acc1 += r.w;
      }
      *reinterpret_cast<float2*>(RC.at(comp) + ((long long)cK * G.cny + cJ) * G.cnx + cI) =
          make_float2(acc0 * 0.125f, acc1 * 0.125f);
    }
  }
}

// Post-smoothing: two red-black sweeps for L x = R from x = E + P EC (the
// prolonged correction of the next level).  UPD: the result is added to the
// double-word iterate (XH, XL) with the arithmetic of k_update_dw; else it is
// stored to OUT.
template <bool UPD>
__global__ void __launch_bounds__(kThr, 2)
k_post_pass(const __grid_constant__ PassGeom G, Comp3<float> R, Comp3<float> E, Comp3<float> EC,
            Comp3<float> OUT, Comp3<float> XH, Comp3<float> XL) {
  pdl_begin();
  extern __shared__ float4 smem_qq[];
  float* const X = reinterpret_cast<float*>(smem_qq) + kPad;
  float* const B = X + kPlanes * kX - kR - kHW;   // rhs: window planes and rows from 1 on
  float* const P = X + kPlanes * kX + (kPlanes - 2) * kR + kPad;
  const int comp = blockIdx.z;
  const float* __restrict__ rhs = R.at(comp);
  const float* __restrict__ e = E.at(comp);
  const int x0 = (blockIdx.x % G.ntx) * kPX, y0 = (blockIdx.x / G.ntx) * kPY, z0 = blockIdx.y * kPZ;
  Item I;
  I.init(G, x0, y0);
  const float w0 = pick3(G.w0, G.w1, G.w2, I.yw), w1 = pick3(G.w0, G.w1, G.w2, I.yw + 1);
  const float h2 = G.h2, c1 = G.c1;
  const long long plane_n = (long long)G.nx * G.ny;
  auto ghost = [&](int k) { return !G.per_z && (k < 0 || k >= G.nz); };
  auto wgt = [&](int k) { return !G.per_z && (k == 0 || k == G.nz - 1) ? w1 : w0; };
  float4 A[kNP], Bv[kNP];
#pragma unroll
  for (int m = 0; m < kNP; ++m) {
    const int k = z0 - kHalo + I.pl + kPS * m;
    if (I.in && !ghost(k)) {
      const float* p = e + (long long)(G.per_z ? mod_(k, G.nz) : k) * plane_n;
      A[m] = l4(p + I.ga);
      Bv[m] = l4(p + I.gb);
    }
  }
  {   // the window's coarse rows, interpolated in x onto the fine columns; a row
      // or plane beyond a wall is -alpha times the one beside it
    const int t = threadIdx.x, ck = t / (kCRows * kG), cr = (t / kG) % kCRows, g = t % kG;
    if (ck < kCPlanes) {
      int K = (z0 >> 1) - 3 + ck, J = (y0 >> 1) - 3 + cr;
      float fy = 1.f, fz = 1.f;
      if (G.per_z) K = mod_(K, G.cnz);
      else if (K < 0 || K >= G.cnz) { fz = G.malpha; K = K < 0 ? 0 : G.cnz - 1; }
      if (G.per_y) J = mod_(J, G.cny);
      else if (J < 0 || J >= G.cny) { fy = G.malpha; J = J < 0 ? 0 : G.cny - 1; }
      const float f = fz * fy;
      const float* p = EC.at(comp) + ((long long)K * G.cny + J) * G.cnx;
      int c = mod_((x0 >> 1) - 3 + 4 * g, G.cnx);
      float n[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        n[i] = f * p[c];
        c = c + 1 == G.cnx ? 0 : c + 1;
      }
      float v[8];
#pragma unroll
      for (int o = 0; o < 8; ++o)
        v[o] = prolong_pair(n[1 + (o >> 1)], n[(o & 1) ? 2 + (o >> 1) : (o >> 1)]);
      float* d = P + (ck * kCRows + cr) * kPW + 8 * g;
      s4(d, make_float4(v[0], v[1], v[2], v[3]));
      s4(d + 4, make_float4(v[4], v[5], v[6], v[7]));
    }
  }
  // rhs in
#pragma unroll
  for (int m = 0; m < kNP; ++m) {
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 1 && pi < kPlanes - 1 && I.inner(1) && !ghost(k)) {
      const float* p = rhs + (long long)(G.per_z ? mod_(k, G.nz) : k) * plane_n;
      float4 r, b;
      split8(l4(p + I.ga), l4(p + I.gb), (I.j + k) & 1, r, b);
      s4(B + pi * kR + I.off, r);
      s4(B + pi * kR + kColR + I.off, b);
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // x = e + P e_c
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f), b = r;
    if (I.in && !ghost(k)) {
      const int J = (I.j >> 1) - (y0 >> 1) + 3, K = (k >> 1) - (z0 >> 1) + 3;
      const int g8 = 8 * (I.off / 4 - I.row * kG);
      const float* p00 = P + (K * kCRows + J) * kPW + g8;
      const int dj = (I.j & 1) ? kPW : -kPW, dk = (k & 1) ? kCRows * kPW : -kCRows * kPW;
      auto up = [](float v, float c, float y, float z, float q) { return v + prolong_sum(c, y, z, q); };
      auto up4 = [&](float4 v, const float* p) {
        const float4 c = l4(p), y = l4(p + dj), z = l4(p + dk), q = l4(p + dj + dk);
        return make_float4(up(v.x, c.x, y.x, z.x, q.x), up(v.y, c.y, y.y, z.y, q.y),
                           up(v.z, c.z, y.z, z.z, q.z), up(v.w, c.w, y.w, z.w, q.w));
      };
      split8(up4(A[m], p00), up4(Bv[m], p00 + 4), (I.j + k) & 1, r, b);
    }
    s4(X + pi * kX + I.off, r);
    s4(X + pi * kX + kCol + I.off, b);
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // red 1
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 1 && pi < kPlanes - 1 && I.inner(1) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      s4(x, half_sweep(x + kCol, x + kCol - kX, x + kCol + kX, l4(x), l4(B + pi * kR + I.off),
                       (I.j + k) & 1, wgt(k), h2, c1));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // black 1
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 2 && pi < kPlanes - 2 && I.inner(2) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      s4(x + kCol, half_sweep(x, x - kX, x + kX, l4(x + kCol), l4(B + pi * kR + kColR + I.off),
                              1 - ((I.j + k) & 1), wgt(k), h2, c1));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // red 2
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= 3 && pi < kPlanes - 3 && I.inner(3) && !ghost(k)) {
      float* x = X + pi * kX + I.off;
      s4(x, half_sweep(x + kCol, x + kCol - kX, x + kCol + kX, l4(x), l4(B + pi * kR + I.off),
                       (I.j + k) & 1, wgt(k), h2, c1));
    }
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kNP; ++m) {   // black 2 of the block itself, stored
    const int pi = I.pl + kPS * m, k = z0 - kHalo + pi;
    if (pi >= kHalo && pi < kHalo + kPZ && k < G.nz && (I.st_a || I.st_b)) {
      const float* x = X + pi * kX + I.off;
      const int par = (I.j + k) & 1;
      const float4 v = half_sweep(x, x - kX, x + kX, l4(x + kCol), l4(B + pi * kR + kColR + I.off),
                                  1 - par, wgt(k), h2, c1);
      float4 a, b;
      join8(l4(x), v, par, a, b);
      const long long p = (long long)k * plane_n;
      if constexpr (UPD) {
        float* __restrict__ uh = XH.at(comp);
        float* __restrict__ ul = XL.at(comp);
        auto add = [&](long long gi, float4 d) {
          const float4 h = l4(uh + gi), l = l4(ul + gi);
          const FF v0 = ff_add_f(FF{h.x, l.x}, d.x), v1 = ff_add_f(FF{h.y, l.y}, d.y);
          const FF v2 = ff_add_f(FF{h.z, l.z}, d.z), v3 = ff_add_f(FF{h.w, l.w}, d.w);
          s4(uh + gi, make_float4(v0.hi, v1.hi, v2.hi, v3.hi));
          s4(ul + gi, make_float4(v0.lo, v1.lo, v2.lo, v3.lo));
        };
        if (I.st_a) add(p + I.ga, a);
        if (I.st_b) add(p + I.gb, b);
      } else {
        float* __restrict__ out = OUT.at(comp);
        if (I.st_a) s4(out + p + I.ga, a);
        if (I.st_b) s4(out + p + I.gb, b);
      }
    }
  }
}

// ---------------------------------------------------------------- launchers
namespace {

PassGeom pass_geom(const Level& F, const Level& C, float omega) {
  PassGeom G{};
  G.nx = F.n[0]; G.ny = F.n[1]; G.nz = F.n[2];
  G.cnx = C.n[0]; G.cny = C.n[1]; G.cnz = C.n[2];
  G.per_y = F.per[1]; G.per_z = F.per[2];
  G.ntx = (F.n[0] + kPX - 1) / kPX;
  G.w0 = omega * F.rcf[0]; G.w1 = omega * F.rcf[1]; G.w2 = omega * F.rcf[2];
  G.d0 = F.cf[0]; G.d1 = F.cf[1]; G.d2 = F.cf[2];
  G.c1 = 1.f - omega;
  G.h2 = (float)(1.0 / F.inv_h2);
  G.ih2 = F.inv_h2f;
  G.malpha = -C.alphaf;
  return G;
}

dim3 pass_grid(const PassGeom& G, int ncomp) {
  return dim3((unsigned)(G.ntx * ((G.ny + kPY - 1) / kPY)), (unsigned)((G.nz + kPZ - 1) / kPZ),
              (unsigned)ncomp);
}

}  // namespace

// Levels the passes serve: every axis active and halved, x periodic in whole
// 16-byte vectors (a window's columns past the extent are wrapped copies), at
// least two cells along y and z (a cell meets at most one wall per axis).
bool two_sweep_pass_ok(const Level& F, const Level& C) {
  return tile::ragged_ok(F) && F.n[0] == 2 * C.n[0] && F.n[1] == 2 * C.n[1] &&
         F.n[2] == 2 * C.n[2] && (long long)F.n[0] * F.n[1] < (1LL << 31);
}

// Every pass kernel's shared memory on the current device; false: the separate
// kernels do the level's work.
bool two_sweep_pass_ready() {
  static DeviceOnce once;
  return once([] {
    return allow_smem(k_pre_pass<true>, kSmemRst) && allow_smem(k_pre_pass<false>, kSmemPre) &&
           allow_smem(k_post_pass<true>, kSmemPost) && allow_smem(k_post_pass<false>, kSmemPost);
  });
}

void launch_pre_pass(Ctx& cx, const Level& F, const Level& C, Comp3<float> R, Comp3<float> E,
                     Comp3<float> RC, int ncomp, float omega, bool restrict_, int kclass) {
  const PassGeom G = pass_geom(F, C, omega);
  cx.before(kclass);
  if (restrict_) launch_k(cx, k_pre_pass<true>, pass_grid(G, ncomp), kThr, kSmemRst, G, R, E, RC);
  else launch_k(cx, k_pre_pass<false>, pass_grid(G, ncomp), kThr, kSmemPre, G, R, E, RC);
  // rhs read, e (and the restricted residual) written
  cx.after(kclass, (restrict_ ? 8.5 : 8.0) * (double)F.cells() * ncomp);
}

void launch_post_pass(Ctx& cx, const Level& F, const Level& C, Comp3<float> R, Comp3<float> E,
                      Comp3<float> EC, Comp3<float> OUT, const Comp3<float>* upd_hi,
                      const Comp3<float>* upd_lo, int ncomp, float omega, int kclass) {
  const PassGeom G = pass_geom(F, C, omega);
  const Comp3<float> none{{nullptr, nullptr, nullptr}};
  cx.before(kclass);
  if (upd_hi && upd_lo)
    launch_k(cx, k_post_pass<true>, pass_grid(G, ncomp), kThr, kSmemPost, G, R, E, EC, OUT, *upd_hi,
             *upd_lo);
  else
    launch_k(cx, k_post_pass<false>, pass_grid(G, ncomp), kThr, kSmemPost, G, R, E, EC, OUT, none, none);
  // e, e_c and rhs read; the iterate's two words read and written, or x written
  cx.after(kclass, (upd_hi && upd_lo ? 24.5 : 12.5) * (double)F.cells() * ncomp);
}

}  // namespace vsv
