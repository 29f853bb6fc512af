// Shared pieces of the Cholesky solvers (chol.cu: fp32 systems of the primal
// fits; fit.cu: the fp64-grade systems of the dual fits): double-float
// arithmetic, 64 x 64 shared tiles and their products, the factor and inverse
// of a 64 x 64 diagonal block, cluster barriers.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace arckv {

constexpr int NB = kCholNB;
constexpr int kCT = 512;
// Shared tiles are [NB][NBP] with rows padded to a 16-byte multiple, so that
// mm64 can read them with vector loads.
template <typename R>
constexpr int NBP = NB + 16 / (int)sizeof(R);
template <typename R>
using Tile = R (*)[NBP<R>];
template <typename R>
constexpr int kTileF = NB * NBP<R>;

__device__ __forceinline__ float fma_r(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rcp_r(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_r(double x) { return __drcp_rn(x); }

// Double-float arithmetic: a value hi + lo of two fp32 numbers (|lo| <= ulp(hi) / 2),
// ~48 significant bits.  The GB300's fp64 pipe issues at a small fraction of its
// fp32 rate, so the fp64 64 x 64 diagonal blocks of the dual Cholesky are
// factored in this arithmetic (each operation a short chain of fp32 operations:
// the error-free sum and product transformations of Dekker and Knuth, and one
// Newton step for the reciprocal and the square root), with the block read
// from and written back to fp64 storage.
struct df64 {
  float hi, lo;
  df64() = default;
  __device__ __forceinline__ df64(float h, float l) : hi(h), lo(l) {}
  __device__ __forceinline__ explicit df64(int v) : hi((float)v), lo(0.f) {}
};
__device__ __forceinline__ df64 df_fast2(float a, float b) {   // |a| >= |b| (or a = 0)
  const float s = a + b;
  return df64(s, b - (s - a));
}
__device__ __forceinline__ df64 df_two(float a, float b) {
  const float s = a + b, bb = s - a;
  return df64(s, (a - (s - bb)) + (b - bb));
}
__device__ __forceinline__ df64 operator+(df64 x, df64 y) {
  df64 s = df_two(x.hi, y.hi);
  const df64 t = df_two(x.lo, y.lo);
  s.lo += t.hi;
  s = df_fast2(s.hi, s.lo);
  s.lo += t.lo;
  return df_fast2(s.hi, s.lo);
}
__device__ __forceinline__ df64 operator-(df64 x) { return df64(-x.hi, -x.lo); }
__device__ __forceinline__ df64 operator-(df64 x, df64 y) { return x + (-y); }
__device__ __forceinline__ df64 operator*(df64 x, df64 y) {
  const float p = x.hi * y.hi;
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return df_fast2(p, e);
}
__device__ __forceinline__ df64& operator*=(df64& x, df64 y) { return x = x * y; }
__device__ __forceinline__ bool operator>(df64 x, df64 y) { return x.hi > y.hi || (x.hi == y.hi && x.lo > y.lo); }
__device__ __forceinline__ bool finite_r(float x) { return isfinite(x); }
__device__ __forceinline__ bool finite_r(double x) { return isfinite(x); }
__device__ __forceinline__ bool finite_r(df64 x) { return isfinite(x.hi); }
__device__ __forceinline__ df64 fma_r(df64 a, df64 b, df64 c) { return a * b + c; }
__device__ __forceinline__ df64 rcp_r(df64 x) {   // r + r (1 - x r)
  const df64 r(__frcp_rn(x.hi), 0.f);
  return r + r * (df64(1) - x * r);
}
__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_r(double x) { return ::sqrt(x); }
__device__ __forceinline__ df64 sqrt_r(df64 x) {    // s + (x - s^2) / (2 s)
  if (!(x.hi > 0.f)) return df64(sqrtf(x.hi), 0.f);
  const float s = sqrtf(x.hi);
  const df64 r = x - df64(s, 0.f) * df64(s, 0.f);
  return df_fast2(s, r.hi * (0.5f / s));
}
// fp32 -> fp64 by moving the fields (IEEE 754: the exponent rebiased by 1023 -
// 127, the fraction padded; subnormals -- a fifth of Phi -- scaled by 2^64
// first): GB300 converts fewer than one value per clock and SM, which held the
// residual passes at 62 and 64 us for 27 MB of Phi (8 heads, n = 1024, t = 819);
// they take 37 and 27 us this way.
// Infinities and NaN take the conversion.
__device__ __forceinline__ double widen_bits(float x) {
  const bool small = (__float_as_uint(x) & 0x7f800000u) == 0u;
  const unsigned u = __float_as_uint(small ? x * 18446744073709551616.f : x), ex = u & 0x7f800000u;
  if (ex == 0x7f800000u) return (double)x;
  const unsigned hi = (u & 0x80000000u) | (ex ? ((u & 0x7fffffffu) >> 3) + (small ? 0x34000000u : 0x38000000u) : 0u);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// storage conversions (the block lives in fp64 in global memory), by fields for
// the same reason: hi = v rounded to nearest even at 24 bits, lo = the exact
// remainder (29 bits and sign) rounded likewise
template <typename R, typename G>
__device__ __forceinline__ R to_reg(G v) { return v; }
template <>
__device__ __forceinline__ df64 to_reg<df64, double>(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v), m = u & 0x7fffffffffffffffull;
  const int ex = (int)(m >> 52);
  if (ex < 1023 - 60 || ex > 1023 + 120) {   // lo or hi near the ends of fp32's range (and zero, infinities, NaN)
    const float h = __double2float_rn(v);
    return df64(h, __double2float_rn(v - (double)h));
  }
  const unsigned long long r = m + 0x0fffffffull + ((m >> 29) & 1);   // rounds at bit 29
  const unsigned hb = (unsigned)(r >> 29);
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  const int rem = (int)(unsigned)m - (int)(hb << 29);   // m - (hb << 29), below 2^29 in magnitude
  const float lo = __int2float_rn(rem) * __uint_as_float((unsigned)(ex - 1075 + 127) << 23);   // exact scaling
  return df64(__uint_as_float(sign | (hb - (896u << 23))), __uint_as_float(__float_as_uint(lo) ^ sign));
}
template <typename G, typename R>
__device__ __forceinline__ G to_mem(R v) { return v; }
template <>
__device__ __forceinline__ double to_mem<double, df64>(df64 v) { return widen_bits(v.hi) + widen_bits(v.lo); }
template <typename R>
__device__ __forceinline__ R warp_sum_r(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The .aligned forms want the warp's threads together.  They often follow a loop
// or a branch that lanes leave at different times, and reconvergence after one
// is not promised, so each begins with a __syncwarp().
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// S[r][c] = G[(r0 + r) * ld + c0 + c] (or S[c][r] with `trans`), zero outside
// rows < rmax, cols < cmax of the source block.  Split into a fetch (eight
// loads per thread into registers) and a put (the shared stores), so that a
// caller loading two tiles issues all sixteen loads before its first store and
// pays the L2 latency once.  The transposed form maps a warp to 4 rows x 8
// columns, so its shared stores hit 32 distinct banks.
template <typename R>
struct TileRegs {
  static constexpr int NE = NB * NB / kCT;
  R v[NE];
  bool trans;
};
// element q of this thread: (row, col) of the source block
__device__ __forceinline__ void tile_pos(int q, bool trans, int& r, int& c) {
  const int e = threadIdx.x + q * kCT;
  if (!trans) {
    r = e / NB;
    c = e % NB;
  } else {
    const int lane = e & 31, w = e >> 5;
    c = (w & 7) * 8 + (lane & 7);
    r = (w >> 3) * 4 + (lane >> 3);
  }
}
template <typename R>
__device__ __forceinline__ void tile_fetch(TileRegs<R>& f, const R* G, long long ld, int r0, int c0, int rmax,
                                           int cmax, bool trans) {
  f.trans = trans;
#pragma unroll
  for (int q = 0; q < TileRegs<R>::NE; ++q) {
    int r, c;
    tile_pos(q, trans, r, c);
    f.v[q] = (r < rmax && c < cmax) ? __ldcg(G + (long long)(r0 + r) * ld + c0 + c) : R(0);
  }
}
template <typename R>
__device__ __forceinline__ void tile_put(Tile<R> S, const TileRegs<R>& f) {
#pragma unroll
  for (int q = 0; q < TileRegs<R>::NE; ++q) {
    int r, c;
    tile_pos(q, f.trans, r, c);
    if (f.trans) S[c][r] = f.v[q];
    else S[r][c] = f.v[q];
  }
}
template <typename R>
__device__ __forceinline__ void ld_tile(Tile<R> S, const R* G, long long ld, int r0, int c0, int rmax, int cmax,
                                        bool trans) {
  TileRegs<R> f;
  tile_fetch(f, G, ld, r0, c0, rmax, cmax, trans);
  tile_put(S, f);
}
// two tiles, one L2 round trip
template <typename R>
__device__ __forceinline__ void ld_tiles(Tile<R> S1, const R* G1, long long ld1, int r1, int c1, int rm1, int cm1,
                                         bool tr1, Tile<R> S2, const R* G2, long long ld2, int r2, int c2, int rm2,
                                         int cm2, bool tr2) {
  TileRegs<R> f1, f2;
  tile_fetch(f1, G1, ld1, r1, c1, rm1, cm1, tr1);
  tile_fetch(f2, G2, ld2, r2, c2, rm2, cm2, tr2);
  tile_put(S1, f1);
  tile_put(S2, f2);
}

// Thread tile of the 64 x 64 products: kTP rows x kTQ columns at (tile_ry, tile_cx).
// A warp covers 16 rows x 16 columns, so each k step of mm64 costs it one
// 16-byte load of the transposed left operand (4 rows) and one 8-byte load of
// the right one (2 columns): two shared wavefronts for 8 FMAs per thread.
constexpr int kTP = 4, kTQ = 2;
__device__ __forceinline__ int tile_ry() { return (threadIdx.x >> 7) * 16 + ((threadIdx.x >> 3) & 3) * 4; }
__device__ __forceinline__ int tile_cx() { return ((threadIdx.x >> 5) & 3) * 16 + (threadIdx.x & 7) * 2; }

// P[p*ld + q] -= acc[p][q] for p < pn, q < qn (all loads issued before the stores)
template <typename R>
__device__ __forceinline__ void rmw_sub(R* P, long long ld, int pn, int qn, const R (&acc)[kTP][kTQ]) {
  R old[kTP][kTQ];
#pragma unroll
  for (int p = 0; p < kTP; ++p)
#pragma unroll
    for (int q = 0; q < kTQ; ++q) old[p][q] = (p < pn && q < qn) ? __ldcg(P + p * ld + q) : R(0);
#pragma unroll
  for (int p = 0; p < kTP; ++p)
#pragma unroll
    for (int q = 0; q < kTQ; ++q)
      if (p < pn && q < qn) P[p * ld + q] = old[p][q] - acc[p][q];
}

__device__ __forceinline__ void lds2(float (&a)[2], const float* p) {
  const float2 v = *(const float2*)p;
  a[0] = v.x; a[1] = v.y;
}
__device__ __forceinline__ void lds4(float (&a)[4], const float* p) {
  const float4 v = *(const float4*)p;
  a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
}
__device__ __forceinline__ void lds2(double (&a)[2], const double* p) {
  const double2 v = *(const double2*)p;
  a[0] = v.x; a[1] = v.y;
}
__device__ __forceinline__ void lds4(double (&a)[4], const double* p) {
  const double2 v = *(const double2*)p, u = *(const double2*)(p + 2);
  a[0] = v.x; a[1] = v.y; a[2] = u.x; a[3] = u.y;
}

// acc[p][q] = sum_l XT[l][ry+p] Y[l][cx+q] (ry = tile_ry(), cx = tile_cx()): the left
// operand is held transposed so that each l takes one 4-wide and one 2-wide
// shared load.
template <typename R>
__device__ __forceinline__ void mm64(Tile<R> XT, Tile<R> Y, R (&acc)[kTP][kTQ]) {
  const int ry = tile_ry(), cx = tile_cx();
#pragma unroll
  for (int p = 0; p < kTP; ++p)
#pragma unroll
    for (int q = 0; q < kTQ; ++q) acc[p][q] = R(0);
#pragma unroll 8
  for (int l = 0; l < NB; ++l) {
    R a[4], c[2];
    lds4(a, &XT[l][ry]);
    lds2(c, &Y[l][cx]);
#pragma unroll
    for (int p = 0; p < kTP; ++p)
#pragma unroll
      for (int q = 0; q < kTQ; ++q) acc[p][q] = fma_r(a[p], c[q], acc[p][q]);
  }
}

// Load the lower part of A_kk + lam I into the tile L (identity beyond the
// matrix when kb < NB; zero above the diagonal).
template <typename R, typename G>
__device__ __forceinline__ void load_diag(Tile<R> L, const G* Ab, int t, int k0, int kb, G lam) {
  constexpr int NE = NB * NB / kCT;
  R v[NE];
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const int e = threadIdx.x + q * kCT, r = e / NB, c = e % NB;
    v[q] = (r < kb && c <= r) ? to_reg<R>(__ldcg(Ab + (long long)(k0 + r) * t + k0 + c) + (r == c ? lam : G(0)))
                              : (r == c ? R(1) : R(0));
  }
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const int e = threadIdx.x + q * kCT;
    L[e / NB][e % NB] = v[q];
  }
}

// Write L_kk (lower part, rows < kb) into A and the full tile Li into Linv[k].
template <typename R, typename G>
__device__ __forceinline__ void store_diag(Tile<R> L, Tile<R> Li, G* Ab, G* Lb, int t, int k, int kb) {
  G* Lo = Lb + (long long)k * NB * NB;
  const int k0 = k * NB;
#pragma unroll
  for (int q = 0; q < NB * NB / kCT; ++q) {
    const int e = threadIdx.x + q * kCT, rr = e / NB, cc = e % NB;
    const bool low = cc <= rr;   // the inverse is lower triangular
    Lo[e] = low ? to_mem<G>(Li[rr][cc]) : G(0);
    if (rr < kb && low) Ab[(long long)(k0 + rr) * t + k0 + cc] = to_mem<G>(L[rr][cc]);
  }
}

// The 16 x 16 diagonal block at c0 of a 64 x 64 block: its update by the panel
// at c0 - 16 (`upd`), its factor (unscaled right-looking, then the column
// scaling by sqrt(a_cc)) and the factor's inverse.  Writes the block of L (pad
// column NB: 1 / l_cc) and of Li.
//
// One warp, in registers: lane (r, hf) holds the eight columns 2q + hf of row
// r, and a step's pivot, column and row reach the other lanes by shuffles (no
// barrier between the columns).  The shuffles of a step are issued before its
// reciprocal, the next pivot's column is updated first.
__device__ __forceinline__ void factor16_warp(Tile<float> L, Tile<float> Li, int c0, int kb, bool upd, int* bad) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 15, hf = lane >> 4;
  float a[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) a[q] = L[c0 + r][c0 + 2 * q + hf];
  if (upd) {
#pragma unroll
    for (int m4 = 0; m4 < 16; m4 += 4) {
      float x[4], y[4];
      lds4(x, &L[c0 + r][c0 - 16 + m4]);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        lds4(y, &L[c0 + 2 * q + hf][c0 - 16 + m4]);
#pragma unroll
        for (int m = 0; m < 4; ++m) a[q] = fmaf(-x[m], y[m], a[q]);
      }
    }
  }
  // entries above the diagonal hold values that nothing on or below it reads
  float pc = 0.f;   // a_rr after its last update
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int kj = j >> 1, hj = (j & 1) * 16;
    float piv = __shfl_sync(kAll, a[kj], hj + j);
    if (r == j) pc = piv;
    if (j == 15) break;
    const float lr = __shfl_sync(kAll, a[kj], hj + r);
    float cj[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (2 * q + 1 > j) cj[q] = __shfl_sync(kAll, a[kj], hj + 2 * q + hf);
    if (!(piv > 0.f) || !isfinite(piv)) piv = 1.f;
    const float f = -lr * __frcp_rn(piv);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (2 * q + 1 > j && 2 * q + hf > j) a[q] = fmaf(f, cj[q], a[q]);
  }
  if (!(pc > 0.f) || !isfinite(pc)) {
    if (c0 + r < kb && hf == 0) *bad = 1;
    pc = 1.f;
  }
  const float dl = sqrtf(pc), il = __frcp_rn(dl);   // column r's scaling
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int c = 2 * q + hf;
    const float d = __shfl_sync(kAll, dl, c), di = __shfl_sync(kAll, il, c);
    a[q] = (r == c) ? d : a[q] * di;
    if (r >= c) L[c0 + r][c0 + c] = a[q];
  }
  if (hf == 0) L[c0 + r][NB] = il;
  // Y = I; y_lj -= l_li y_ij / l_ii for l > i, j <= i; then X = diag(1 / l_rr) Y
  float y[8], g[15];
#pragma unroll
  for (int i = 0; i < 15; ++i) g[i] = -__shfl_sync(kAll, a[i >> 1], (i & 1) * 16 + r) * __shfl_sync(kAll, il, i);
#pragma unroll
  for (int q = 0; q < 8; ++q) y[q] = (2 * q + hf == r) ? 1.f : 0.f;
#pragma unroll
  for (int i = 0; i < 15; ++i) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (2 * q > i) continue;
      const float yi = __shfl_sync(kAll, y[q], hf * 16 + i);
      if (r > i && 2 * q + hf <= i) y[q] = fmaf(g[i], yi, y[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (2 * q + hf <= r) Li[c0 + r][c0 + 2 * q + hf] = y[q] * il;
}

// The same for the other number types, on the first 256 threads: one element
// per thread in shared memory, a barrier of these threads per column (a
// double-float step is ~60 instructions, more than one warp hides: 31 K
// cycles a block on one warp, 11 K here).
constexpr int kTeam = 256;
template <typename R>
__device__ __forceinline__ void factor16_team(Tile<R> L, Tile<R> Li, int c0, int kb, bool upd, int* bad) {
  const int er = threadIdx.x >> 4, ec = threadIdx.x & 15;
  auto sync = [&]() { asm volatile("bar.sync 2, %0;" ::"n"(kTeam) : "memory"); };
  if (upd) {
    if (er >= ec) {
      R a = L[c0 + er][c0 + ec];
#pragma unroll
      for (int m = 0; m < 16; ++m) a = fma_r(-L[c0 + er][c0 - 16 + m], L[c0 + ec][c0 - 16 + m], a);
      L[c0 + er][c0 + ec] = a;
    }
    sync();
  }
  for (int j = 0; j < 15; ++j) {
    if (ec > j && er >= ec) {
      R piv = L[c0 + j][c0 + j];
      if (!(piv > R(0)) || !finite_r(piv)) piv = R(1);
      L[c0 + er][c0 + ec] = fma_r(-L[c0 + er][c0 + j] * rcp_r(piv), L[c0 + ec][c0 + j], L[c0 + er][c0 + ec]);
    }
    sync();
  }
  R v = R(0);
  if (er >= ec) {   // column scaling
    R pc = L[c0 + ec][c0 + ec];
    if (!(pc > R(0)) || !finite_r(pc)) {
      if (er == ec && c0 + ec < kb) *bad = 1;
      pc = R(1);
    }
    const R d = sqrt_r(pc);
    v = (er == ec) ? d : L[c0 + er][c0 + ec] * rcp_r(d);
  }
  sync();
  if (er >= ec) {
    L[c0 + er][c0 + ec] = v;
    if (er == ec) {
      L[c0 + er][NB] = rcp_r(v);
      Li[c0 + er][c0 + er] = R(1);
    }
  }
  sync();
  for (int i = 0; i < 15; ++i) {   // Y = I; y_lj -= l_li y_ij / l_ii for l > i, j <= i
    if (er > i && ec <= i)
      Li[c0 + er][c0 + ec] = fma_r(-L[c0 + er][c0 + i] * L[c0 + i][NB], Li[c0 + i][c0 + ec], Li[c0 + er][c0 + ec]);
    sync();
  }
  if (ec <= er) Li[c0 + er][c0 + ec] *= L[c0 + er][NB];   // X = diag(1 / l_rr) Y
}

// Factor diagonal block k, given in the tile L (load_diag's form), and invert
// the factor: L_kk goes into A and L_kk^-1 into Linv[k].  Blocked in
// four 16-wide panels:
//   panel p: its 16 x 16 diagonal block is factored and inverted
//            (factor16_warp / factor16_team); L_panel = A_panel X_pp^T below
//            it on all warps; trailing update A -= L_panel L_panel^T;
//   inverse: off-diagonal 16 x 16 blocks X_ij = -X_ii sum_{m=j}^{i-1} L_im X_mj.
// The chain of the four 16-column factorisations is what bounds it, so its
// threads go from one diagonal block to the next and take that block's own
// update, while the other warps finish the trailing update and form the
// inverse's blocks as soon as their factors are there.  One element per
// thread with block barriers, one phase after the other, took 40 K cycles.
// Tiles: L (the block; pad column NB holds 1 / l_cc), Li (the inverse), T
// (scratch).  Pad rows beyond the matrix (kb < NB) are the identity.
template <typename R, typename G = R>
__device__ void factor_diag(G* Ab, G* Lb, int t, int k, Tile<R> L, Tile<R> Li, Tile<R> T, int* bad) {
  static_assert(kCT == 512 && NB == 64, "thread map of the 16-wide panels");
  constexpr bool kWarp = std::is_same<R, float>::value;
  constexpr int kFirst = kWarp ? 32 : kTeam, kRest = kCT - kFirst;   // the others: kRest threads
  const int tid = threadIdx.x, k0 = k * NB, kb = min(NB, t - k0);
  for (int e = tid; e < NB * NB; e += kCT) Li[e / NB][e % NB] = R(0);
  __syncthreads();
  const int wt = tid - kFirst;
  auto rest_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kRest) : "memory"); };
  // T_ij = sum_{m=j}^{i-1} L_im X_mj (element x of the block)
  auto inv_t = [&](int i, int j, int x) {
    const int r = x >> 4, c = x & 15;
    R a = R(0);
    for (int m = j; m < i; ++m)
#pragma unroll
      for (int q = 0; q < 16; ++q) a = fma_r(L[16 * i + r][16 * m + q], Li[16 * m + q][16 * j + c], a);
    T[16 * i + r][16 * j + c] = a;
  };
  // X_ij = -X_ii T_ij
  auto inv_x = [&](int i, int j, int x) {
    const int r = x >> 4, c = x & 15;
    R a = R(0);
    for (int q = 0; q <= r; ++q) a = fma_r(Li[16 * i + r][16 * i + q], T[16 * i + q][16 * j + c], a);
    Li[16 * i + r][16 * j + c] = -a;
  };
  for (int p = 0; p < 4; ++p) {
    const int c0 = 16 * p;
    if (wt < 0) {
      if constexpr (kWarp) factor16_warp(L, Li, c0, kb, p > 0, bad);
      else factor16_team<R>(L, Li, c0, kb, p > 0, bad);
    } else {
      if (p > 0) {
        // the rest of panel p - 1's trailing update: L[r][c] -= sum_m L[r][cp + m] L[c][cp + m], c0 <= c <= r, r >= c0 + 16
        const int wdt = NB - c0, ntri = wdt * (wdt + 1) / 2, cp = c0 - 16;
        for (int e = 136 + wt; e < ntri; e += kRest) {   // 136 = the diagonal block's lower triangle
          int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
          while (r * (r + 1) / 2 > e) --r;
          while ((r + 1) * (r + 2) / 2 <= e) ++r;
          const int c = e - r * (r + 1) / 2;
          R a = L[c0 + r][c0 + c];
#pragma unroll
          for (int m = 0; m < 16; ++m) a = fma_r(-L[c0 + r][cp + m], L[c0 + c][cp + m], a);
          L[c0 + r][c0 + c] = a;
        }
      }
      if (p == 2) {
        for (int e = wt; e < 256; e += kRest) inv_t(1, 0, e);
        rest_sync();
        for (int e = wt; e < 256; e += kRest) inv_x(1, 0, e);
      }
      if (p == 3) {
        for (int e = wt; e < 512; e += kRest) inv_t(2, e >> 8, e & 255);
        rest_sync();
        for (int e = wt; e < 512; e += kRest) inv_x(2, e >> 8, e & 255);
        rest_sync();
        for (int e = wt; e < 768; e += kRest) inv_t(3, e >> 8, e & 255);
      }
    }
    __syncthreads();
    if (p == 3) break;
    // panel below: L[r][c0 + c] = sum_m A[r][c0 + m] X_pp[c][m] (all reads before the writes)
    const int rows = NB - c0 - 16;
    R o[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + q * kCT, r = c0 + 16 + e / 16, c = e % 16;
      R a = R(0);
      if (e < rows * 16) {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const R s = fma_r(L[r][c0 + m], Li[c0 + c][c0 + m], a);
          if (m <= c) a = s;
        }
      }
      o[q] = a;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + q * kCT;
      if (e < rows * 16) L[c0 + 16 + e / 16][c0 + e % 16] = o[q];
    }
    __syncthreads();
  }
  for (int e = tid; e < 768; e += kCT) inv_x(3, e >> 8, e & 255);
  __syncthreads();
  store_diag(L, Li, Ab, Lb, t, k, kb);
  __syncthreads();
}

// S[r][c] = G1[(r0 + r) * ld + c0 + c] + G2[...] (zero outside rows < rmax, cols < cmax)
template <typename R>
__device__ __forceinline__ void ld_tile_sum(Tile<R> S, const R* G1, const R* G2, long long ld, int r0, int c0,
                                            int rmax, int cmax) {
  constexpr int NE = NB * NB / kCT;
  R v[NE], u[NE];
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const int e = threadIdx.x + q * kCT, r = e / NB, c = e % NB;
    const bool ok = r < rmax && c < cmax;
    const long long o = (long long)(r0 + r) * ld + c0 + c;
    v[q] = ok ? __ldcg(G1 + o) : R(0);
    u[q] = ok ? __ldcg(G2 + o) : R(0);
  }
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const int e = threadIdx.x + q * kCT;
    S[e / NB][e % NB] = v[q] + u[q];
  }
}

// P[p*ld + q] = acc[p][q] for p < pn, q < qn
template <typename R>
__device__ __forceinline__ void st_acc(R* P, long long ld, int pn, int qn, const R (&acc)[kTP][kTQ]) {
#pragma unroll
  for (int p = 0; p < kTP; ++p)
#pragma unroll
    for (int q = 0; q < kTQ; ++q)
      if (p < pn && q < qn) P[p * ld + q] = acc[p][q];
}

}  // namespace arckv
