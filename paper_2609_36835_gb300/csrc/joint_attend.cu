// Attention over a compact block followed by an uncompressed block (App. A.7
// Eq. concatenated_attention_preservation):
//
//   O_i = sum_j e^{a_ij} v_j / sum_j e^{a_ij},   a_ij = scale q_i.k_j + b_j,
//   k, v, b = [C_k; K_fixed], [C_v; V_fixed], [beta; 0_F]
//
// for H independent heads of n query rows (a decode batch folds into H).
// The operation streams every key and value once and does ~2 FMA per byte of
// bf16 cache: it is HBM-bound, so it runs on the SIMT pipes as a split-key
// ("flash-decoding") pass, not as a GEMM.
//   attend_warp_kernel: CTA (key split, 4-row block, head) of four warps that
//     never wait for one another: each has its own ring of 16-key tiles (K and
//     V rows by cp.async.bulk), its own running (max, sum) and accumulators;
//     the four are merged once, at the end of the split;
//   attend_combine_kernel: per (head, row) merges the splits' (m, l, o) and
//     checks the result (one split: the first kernel does both).
// A warp reads two keys per instruction; lane l holds query dims 8 (l % 16) ..
// +7 of the 4 rows in registers.  Its 32 partial dot products (8 keys x 4 rows)
// are summed over the 16 lanes of each half-warp by a transposing butterfly
// (30 shuffles), the weights go through 256 bytes of shared memory, and both
// products run as packed pairs (fma.rn.f32x2), without which the SIMT pipes
// would be as busy as the memory.
//
// t = 0 gives plain attention over the uncompressed block (the full-cache
// baseline of the decode measurement); F = 0 the compact operator of Sec. 3.1.
#include <algorithm>

#include "kernels.h"
#include "tc.cuh"

namespace arckv {

constexpr int kJR = 4;        // query rows per CTA
constexpr int kJKeys = 16;    // keys per tile of a warp
constexpr int kJWarps = 4;
constexpr int kJStages = 2;

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// eight consecutive elements of a row in shared memory as four pairs
__device__ __forceinline__ void lds8(const bf16* p, f32x2 (&x)[4]) {
  const uint4 u = *(const uint4*)p;
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) x[e] = pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
}
__device__ __forceinline__ void lds8(const float* p, f32x2 (&x)[4]) {
  const float4 a = *(const float4*)p, b = *(const float4*)(p + 4);
  x[0] = pack2(a.x, a.y);
  x[1] = pack2(a.z, a.w);
  x[2] = pack2(b.x, b.y);
  x[3] = pack2(b.z, b.w);
}

// Arguments of one pass over the keys.  kErr (App. B.1): all keys in the
// second block, and a second accumulator over the keys with inS != 0.
struct JointArgs {
  const bf16* Q;
  int n;
  const void* Ck;   // compact rows, TC
  const float* beta;
  const void* Cv;
  int t;
  const bf16 *Kf, *Vf;
  int F;
  const unsigned char* inS;
  float scale;
  int per_split, nsplit;
  float* Opart;     // [H][nsplit][n][128] (kErr: 256: all keys, keys in S)
  float2* ml;       // [H][nsplit][n] (running max, sum)
  float* O;         // one split: the result
  DevStatus* stt;
  float* err;       // kErr, one split: the rows' errors [H][n]
  float eps;
};

// ||o - o_S|| / (||o|| + eps) of a row, on lane 0: o and o_S at this lane's four
// dims, unnormalised, over the same sum of weights l (one warp per row).
__device__ __forceinline__ float row_error(const float (&o)[4], const float (&os)[4], float l, float eps) {
  const float inv = 1.0f / l;
  float dd = 0.f, oo = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float x = o[e] * inv, y = os[e] * inv;
    dd = fmaf(x - y, x - y, dd);
    oo = fmaf(x, x, oo);
  }
  dd = warp_sum(dd);
  oo = warp_sum(oo);
  return sqrtf(dd) / (sqrtf(oo) + eps);
}

template <typename TC>
constexpr int kJStageBytes = 2 * kJKeys * 128 * (int)sizeof(TC);   // K and V tile of one warp
template <typename TC>
constexpr int kJSmem = kJWarps * kJStages * kJStageBytes<TC>;

// kOne: kErr with one split, a kernel of its own (its shared rows and their norms
// in the other one cost a call of 160 us 4 of them).
template <typename TC, bool kErr, bool kOne = false>
__global__ void __launch_bounds__(32 * kJWarps, kErr ? 2 : 3) attend_warp_kernel(const JointArgs a) {
  chain_wait();
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar[kJWarps][kJStages];
  __shared__ __align__(16) float sP[kJWarps][kJKeys][kJR];
  __shared__ float sM[kJWarps][kJR], sL[kJWarps][kJR];
  __shared__ int abort_flag;
  const int h = blockIdx.z, r0 = blockIdx.y * kJR, sp = blockIdx.x, n = a.n, t = a.t;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, hl = lane & 15, hh = lane >> 4;
  const int L = t + a.F, jb = sp * a.per_split, je = min(L, jb + a.per_split);
  // tiles: the compact keys [jb, min(je, t)), then the uncompressed ones [max(jb, t), je)
  const int c_hi = min(je, t), f_lo = max(jb, t);
  const int n1 = c_hi > jb ? (c_hi - jb + kJKeys - 1) / kJKeys : 0;
  const int ntile = n1 + (je > f_lo ? (je - f_lo + kJKeys - 1) / kJKeys : 0);
  unsigned char* ring = smraw + w * kJStages * kJStageBytes<TC>;
  auto tile_of = [&](int i, int& j0, int& nk, bool& comp) {
    comp = i < n1;
    j0 = comp ? jb + i * kJKeys : f_lo + (i - n1) * kJKeys;
    nk = min(kJKeys, (comp ? c_hi : je) - j0);
  };
  auto issue = [&](int i, int s) {   // lane 0: K and V of tile i into stage s
    int j0, nk;
    bool comp;
    tile_of(i, j0, nk, comp);
    unsigned char* st = ring + s * kJStageBytes<TC>;
    const uint32_t bytes = (uint32_t)nk * 128u * (comp ? (uint32_t)sizeof(TC) : 2u);
    tc::mbar_arrive_expect_tx(&bar[w][s], 2 * bytes);
    const void *ks, *vs;
    if (comp) {
      const long long row = ((long long)h * t + j0) * 128;
      ks = (const TC*)a.Ck + row;
      vs = (const TC*)a.Cv + row;
    } else {
      const long long row = ((long long)h * a.F + j0 - t) * 128;
      ks = a.Kf + row;
      vs = a.Vf + row;
    }
    tc::bulk_load(st, ks, bytes, &bar[w][s]);
    tc::bulk_load(st + kJStageBytes<TC> / 2, vs, bytes, &bar[w][s]);
  };
  if (tid == 0) abort_flag = 0;
  if (lane == 0) {
    for (int s = 0; s < kJStages; ++s) tc::mbar_init(&bar[w][s], 1);
    tc::mbar_fence_init();
    for (int s = 0; s < kJStages; ++s)
      if (w + s * kJWarps < ntile) issue(w + s * kJWarps, s);
  }
  __syncthreads();
  // the 4 query rows at dims 8 hl .. 8 hl + 7, pre-scaled
  f32x2 q[kJR][4], acc[kJR][4], accs[kErr ? kJR : 1][4];
#pragma unroll
  for (int r = 0; r < kJR; ++r) {
    const bf16* qp = a.Q + ((long long)h * n + r0 + r) * 128 + hl * 8;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      q[r][e] = r0 + r < n ? pack2(a.scale * __bfloat162float(qp[2 * e]), a.scale * __bfloat162float(qp[2 * e + 1]))
                           : 0ull;
      acc[r][e] = 0ull;
      if (kErr) accs[r][e] = 0ull;
    }
  }
  // running max and sum of rows rp, rp + 1; the sum over this lane's keys only
  const int rp = (hl & 1) * 2, kq = 2 * (hl >> 1) + hh;   // this lane's rows and key of a tile after the butterfly
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  bool ok = true;
  int it = 0;
  for (int i = w; i < ntile; i += kJWarps, ++it) {
    int j0, nk;
    bool comp;
    tile_of(i, j0, nk, comp);
    const int s = it % kJStages;
    float b = 0.f;
    if (comp && kq < nk) b = __ldg(a.beta + (long long)h * t + j0 + kq);
    ok = tc::mbar_wait(&bar[w][s], (uint32_t)((it / kJStages) & 1), &abort_flag, a.stt);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) break;
    const unsigned char* st = ring + s * kJStageBytes<TC>;
    float v[32];   // partial dots: entry 4 q + r is key 2 q + hh, row r
    auto logits = [&](const auto* Kt) {
#pragma unroll
      for (int qq = 0; qq < 8; ++qq) {
        f32x2 k[4];
        lds8(Kt + (2 * qq + hh) * 128 + hl * 8, k);
#pragma unroll
        for (int r = 0; r < kJR; ++r) {
          f32x2 d = mul2(q[r][0], k[0]);
#pragma unroll
          for (int e = 1; e < 4; ++e) d = fma2(q[r][e], k[e], d);
          const float2 f = unpack2(d);
          v[4 * qq + r] = f.x + f.y;
        }
      }
    };
    if (sizeof(TC) == 4 && comp) logits((const TC*)st);
    else logits((const bf16*)st);
    // transposing butterfly over the 16 lanes of the half-warp: lane hl ends
    // with entries 2 hl and 2 hl + 1 (key kq, rows rp and rp + 1)
#pragma unroll
    for (int o = 8, c = 16; o >= 1; o >>= 1, c >>= 1) {
      const bool up = hl & o;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        if (e >= c) break;
        const float mine = up ? v[c + e] : v[e], other = up ? v[e] : v[c + e];
        v[e] = mine + __shfl_xor_sync(0xffffffffu, other, o);
      }
    }
    const float a0 = kq < nk ? v[0] + b : -INFINITY, a1 = kq < nk ? v[1] + b : -INFINITY;
    float n0 = a0, n1_ = a1;
#pragma unroll
    for (int o = 16; o >= 2; o >>= 1) {
      n0 = fmaxf(n0, __shfl_xor_sync(0xffffffffu, n0, o));
      n1_ = fmaxf(n1_, __shfl_xor_sync(0xffffffffu, n1_, o));
    }
    n0 = fmaxf(m0, n0);
    n1_ = fmaxf(m1, n1_);
    // rows whose keys so far all have logit -inf keep weight 0 (not exp(-inf + inf))
    const float s0 = n0 == -INFINITY ? 0.f : n0, s1 = n1_ == -INFINITY ? 0.f : n1_;
    const float p0 = expf(a0 - s0), p1 = expf(a1 - s1);
    *(float2*)&sP[w][kq][rp] = make_float2(p0, p1);
    if (__any_sync(0xffffffffu, n0 != m0 || n1_ != m1)) {   // a new maximum: rescale
      const float f0 = expf(m0 - s0), f1 = expf(m1 - s1);
      l0 *= f0;
      l1 *= f1;
      const float g0 = __shfl_xor_sync(0xffffffffu, f0, 1), g1 = __shfl_xor_sync(0xffffffffu, f1, 1);
      const float f[kJR] = {rp ? g0 : f0, rp ? g1 : f1, rp ? f0 : g0, rp ? f1 : g1};
#pragma unroll
      for (int r = 0; r < kJR; ++r) {
        const f32x2 ff = pack2(f[r], f[r]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[r][e] = mul2(acc[r][e], ff);
          if (kErr) accs[r][e] = mul2(accs[r][e], ff);
        }
      }
      m0 = n0;
      m1 = n1_;
    }
    l0 += p0;
    l1 += p1;
    __syncwarp();
    auto values = [&](const auto* Vt) {
#pragma unroll
      for (int qq = 0; qq < 8; ++qq) {
        const int kk = 2 * qq + hh;
        if (kk < nk) {   // rows past the tile's end hold whatever was there
          f32x2 x[4];
          lds8(Vt + kk * 128 + hl * 8, x);
          const float4 p = *(const float4*)sP[w][kk];
          const f32x2 pp[kJR] = {pack2(p.x, p.x), pack2(p.y, p.y), pack2(p.z, p.z), pack2(p.w, p.w)};
#pragma unroll
          for (int r = 0; r < kJR; ++r)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[r][e] = fma2(pp[r], x[e], acc[r][e]);
          if (kErr && a.inS[(long long)h * a.F + j0 + kk]) {
#pragma unroll
            for (int r = 0; r < kJR; ++r)
#pragma unroll
              for (int e = 0; e < 4; ++e) accs[r][e] = fma2(pp[r], x[e], accs[r][e]);
          }
        }
      }
    };
    if (sizeof(TC) == 4 && comp) values((const TC*)(st + kJStageBytes<TC> / 2));
    else values((const bf16*)(st + kJStageBytes<TC> / 2));
    __syncwarp();   // the stage and sP are free
    if (lane == 0 && i + kJStages * kJWarps < ntile) issue(i + kJStages * kJWarps, s);
  }
  if (!ok && lane == 0) {
    // a wait gave up (status recorded): let the copies already issued land
    // (bounded) before the CTA's shared memory goes away
    volatile int never = 0;
    for (int k = it; k < it + kJStages && w + k * kJWarps < ntile; ++k)
      tc::mbar_wait(&bar[w][k % kJStages], (uint32_t)((k / kJStages) & 1), &never, a.stt);
  }
  // merge the half-warps (same dims, other keys), then the warps
#pragma unroll
  for (int o = 16; o >= 2; o >>= 1) {
    l0 += __shfl_xor_sync(0xffffffffu, l0, o);
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  }
  if (lane < 2) {
    sM[w][rp] = m0;
    sM[w][rp + 1] = m1;
    sL[w][rp] = l0;
    sL[w][rp + 1] = l1;
  }
  constexpr int kA = kErr ? 2 : 1;
  float* sAcc = (float*)smraw;   // [warp][kA][kJR][128]: each warp over its own drained ring
  static_assert(kA * kJR * 128 * 4 <= kJStages * kJStageBytes<TC>, "a warp's accumulators fit its ring");
  float* mine = (float*)ring;
#pragma unroll
  for (int r = 0; r < kJR; ++r)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 x = unpack2(acc[r][e]);
      x.x += __shfl_xor_sync(0xffffffffu, x.x, 16);
      x.y += __shfl_xor_sync(0xffffffffu, x.y, 16);
      if (hh == 0) *(float2*)&mine[r * 128 + hl * 8 + 2 * e] = x;
      if (kErr) {
        float2 y = unpack2(accs[r][e]);
        y.x += __shfl_xor_sync(0xffffffffu, y.x, 16);
        y.y += __shfl_xor_sync(0xffffffffu, y.y, 16);
        if (hh == 0) *(float2*)&mine[(kJR + r) * 128 + hl * 8 + 2 * e] = y;
      }
    }
  __syncthreads();
  if (abort_flag) return;
  constexpr int kRing = kJStages * kJStageBytes<TC> / 4;   // floats between two warps' accumulators
  __shared__ float sOut[kOne ? kJR : 1][2][kOne ? 128 : 1], sSum[kJR];   // kOne: the merged rows
  bool bad = false;
#pragma unroll
  for (int r = 0; r < kJR; ++r) {
    if (r0 + r >= n) break;
    float M = sM[0][r];
#pragma unroll
    for (int k = 1; k < kJWarps; ++k) M = fmaxf(M, sM[k][r]);
    const float Ms = M == -INFINITY ? 0.f : M;
    float f[kJWarps], l = 0.f;
#pragma unroll
    for (int k = 0; k < kJWarps; ++k) {
      f[k] = expf(sM[k][r] - Ms);
      l = fmaf(sL[k][r], f[k], l);
    }
    const long long row = ((long long)h * a.nsplit + sp) * n + r0 + r;
#pragma unroll
    for (int c = 0; c < kA; ++c) {
      float o = 0.f;
#pragma unroll
      for (int k = 0; k < kJWarps; ++k) o = fmaf(sAcc[k * kRing + (c * kJR + r) * 128 + tid], f[k], o);
      if (!kErr && a.nsplit == 1) {
        o *= 1.0f / l;
        bad |= !isfinite(o);
        a.O[((long long)h * n + r0 + r) * 128 + tid] = o;
      } else if constexpr (kOne) {
        sOut[r][c][tid] = o;
      } else {
        a.Opart[(row * kA + c) * 128 + tid] = o;
      }
    }
    if (tid == 0) {
      if constexpr (kOne) sSum[r] = l;
      else a.ml[row] = make_float2(M, l);
    }
  }
  if (bad) set_status(a.stt, ARCKV_ERR_NONFINITE);
  if constexpr (kOne) {   // nothing to combine, warp w takes row r0 + w
    __syncthreads();
    if (r0 + w >= n) return;
    float o[4], os[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      o[e] = sOut[w][0][lane * 4 + e];
      os[e] = sOut[w][1][lane * 4 + e];
    }
    const float er = row_error(o, os, sSum[w], a.eps);
    if (lane == 0) a.err[(long long)h * n + r0 + w] = er;
  }
}

// O[h][i] = sum_s e^{m_s - m} Opart_s / sum_s e^{m_s - m} l_s (one warp per row, lane dims 4l..4l+3)
__global__ void __launch_bounds__(128) attend_combine_kernel(const float* Opart, const float2* ml, int n, int nsplit,
                                                             long long rows, float* O, DevStatus* stt) {
  chain_wait();
  const long long g = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (g >= rows) return;
  const long long h = g / n, i = g % n;
  const float2* mlh = ml + h * nsplit * n + i;
  float m = -INFINITY;
  for (int s = lane; s < nsplit; s += 32) m = fmaxf(m, mlh[(long long)s * n].x);
  m = warp_max(m);
  float l = 0.f, o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll 4
  for (int s = 0; s < nsplit; ++s) {
    const float2 v = mlh[(long long)s * n];
    const float4 op = *(const float4*)(Opart + ((h * nsplit + s) * n + i) * 128 + lane * 4);
    const float f = expf(v.x - m);
    l = fmaf(v.y, f, l);
    o0 = fmaf(f, op.x, o0);
    o1 = fmaf(f, op.y, o1);
    o2 = fmaf(f, op.z, o2);
    o3 = fmaf(f, op.w, o3);
  }
  const float inv = 1.0f / l;
  const float4 o = make_float4(o0 * inv, o1 * inv, o2 * inv, o3 * inv);
  *(float4*)(O + g * 128 + lane * 4) = o;
  if (!isfinite(o.x) || !isfinite(o.y) || !isfinite(o.z) || !isfinite(o.w)) set_status(stt, ARCKV_ERR_NONFINITE);
}

// ---------------------------------------------------------------------------
// Truncated-output error of an anchor set (App. B.1 Eq. background_truncated_error):
//   O_i = sum_j p_ij v_j, O~_i(S) = sum_{j in S} p_ij v_j (p over the full cache),
//   err_i = ||O_i - O~_i|| / (||O_i|| + eps).
// The split-key pass above with two value accumulators (all keys; keys in S);
// then one warp per row merges the splits and takes the norms (in the first kernel
// where there is one split, so that the partial rows, 1 KB each, are kept only
// where the rows are too few to fill the SMs).  8 heads, n = 64, T = 8192: 0.17 ms
// a call; one CTA per four rows over all keys took 0.88 ms.
__global__ void __launch_bounds__(128) trunc_combine_kernel(const float* Opart, const float2* ml, int n, int nsplit,
                                                            long long rows, float eps, float* err) {
  chain_wait();
  const long long g = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (g >= rows) return;
  const long long h = g / n, i = g % n;
  const float2* mlh = ml + h * nsplit * n + i;
  float m = -INFINITY;
  for (int s = lane; s < nsplit; s += 32) m = fmaxf(m, mlh[(long long)s * n].x);
  m = warp_max(m);
  float l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f}, os[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int s = 0; s < nsplit; ++s) {
    const float2 v = mlh[(long long)s * n];
    const float* op = Opart + ((h * nsplit + s) * n + i) * 256 + lane * 4;
    const float4 x = *(const float4*)op, y = *(const float4*)(op + 128);
    const float f = expf(v.x - m);
    l = fmaf(v.y, f, l);
    o[0] = fmaf(f, x.x, o[0]); o[1] = fmaf(f, x.y, o[1]); o[2] = fmaf(f, x.z, o[2]); o[3] = fmaf(f, x.w, o[3]);
    os[0] = fmaf(f, y.x, os[0]); os[1] = fmaf(f, y.y, os[1]); os[2] = fmaf(f, y.z, os[2]); os[3] = fmaf(f, y.w, os[3]);
  }
  const float er = row_error(o, os, l, eps);
  if (lane == 0) err[g] = er;
}

// inS[h][j] = 1 for the anchors S[h][:] (clamped into [0, T); out-of-range entries record INVALID_ARG)
__global__ void anchor_mask_kernel(const int* S, int t, int T, int H, unsigned char* inS, DevStatus* stt) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < (long long)H * t;
       k += (long long)gridDim.x * blockDim.x) {
    const long long h = k / t;
    int j = S[k];
    if (j < 0 || j >= T) {
      set_status(stt, ARCKV_ERR_INVALID_ARG);
      j = min(max(j, 0), T - 1);
    }
    inS[h * T + j] = 1;
  }
}

// E[h] = mean_i err[h][i] (fixed order: lane sums, then the butterfly), one warp per head
__global__ void __launch_bounds__(32) row_mean_kernel(const float* err, int n, float* E, DevStatus* stt) {
  chain_wait();
  const int h = blockIdx.x, lane = threadIdx.x;
  float a = 0.f;
  for (int i = lane; i < n; i += 32) a += err[(long long)h * n + i];
  a = warp_sum(a);
  if (lane == 0) {
    const float e = a / (float)n;
    E[h] = e;
    if (!isfinite(e)) set_status(stt, ARCKV_ERR_NONFINITE);
  }
}

// Key splits: the count that minimises waves x (tiles of a warp + start), a
// split's start (first loads, merge) costing about one and a half tiles and
// every split a little in the combine; `per_sm` CTAs fit an SM (of fp32 compact
// rows, whose rings are twice as large, one: they are split like bf16 rows, since
// the workspace's size does not depend on their type; 512 heads, n = 4, t = 1638, F
// = 200: 186 us, 102 with bf16 rows, of which HBM takes 137 and 73).
static JointSplit split_keys(long long ctas, int L, int per_sm) {
  const long long slots = (long long)tc_gemm_sm_count() * per_sm;
  // up to eight rounds of CTAs, no warp without a tile
  const int tiles = cdiv(L, kJKeys);
  const int most = (int)std::min<long long>(cdiv(tiles, kJWarps), std::min<long long>(256, (8 * slots + ctas - 1) / ctas));
  JointSplit best{tiles * kJKeys, 1};
  double cost = 1e300;
  for (int want = 1; want <= most; ++want) {
    const int per = cdiv(tiles, want), ns = cdiv(tiles, per);
    const double waves = std::max(1.0, (double)((ctas * ns + slots - 1) / slots));
    const double c = waves * (cdiv(per, kJWarps) + 1.5) + 0.05 * (ns > 1 ? ns + 8 : 0);
    if (c < cost) {
      cost = c;
      best = JointSplit{per * kJKeys, ns};
    }
  }
  return best;
}

JointSplit joint_split(int H, int n, int t, int F) { return split_keys((long long)H * cdiv(n, kJR), t + F, 3); }

JointSplit trunc_split(int H, int n, int T) { return split_keys((long long)H * cdiv(n, kJR), T, 2); }

int launch_truncated_error(int H, int n, int T, int t, float scale, float eps, const bf16* Q, const bf16* K,
                           const bf16* V, const int* S, float* E, unsigned char* inS, float* err, float* Opart,
                           float2* ml, DevStatus* stt, cudaStream_t st) {
  cudaMemsetAsync(inS, 0, (size_t)H * T, st);
  if (t > 0)
    launch_chained(anchor_mask_kernel, stride_grid((long long)H * t, 256, 4), 256, 0, st, S, t, T, H, inS, stt);
  const JointSplit s = trunc_split(H, n, T);
  const JointArgs a{Q, n, nullptr, nullptr, nullptr, 0, K, V, T, inS, scale, s.per_split, s.nsplit, Opart, ml, nullptr,
                    stt, err, eps};
  auto kern = s.nsplit > 1 ? attend_warp_kernel<bf16, true> : attend_warp_kernel<bf16, true, true>;
  set_dyn_smem((const void*)kern, kJSmem<bf16>);
  launch_chained(kern, dim3(s.nsplit, cdiv(n, kJR), H), 32 * kJWarps, kJSmem<bf16>, st, a);
  const long long rows = (long long)H * n;
  if (s.nsplit > 1)
    launch_chained(trunc_combine_kernel, (unsigned)cdiv(rows, 4), 128, 0, st, Opart, ml, n, s.nsplit, rows, eps, err);
  launch_chained(row_mean_kernel, H, 32, 0, st, err, n, E, stt);
  return 2 + (t > 0 ? 1 : 0) + (s.nsplit > 1 ? 1 : 0);
}

int launch_attend_joint(int H, int n, int t, int F, float scale, const bf16* Q, const void* Ck, const float* beta,
                        const void* Cv, bool compact_bf16, const bf16* Kf, const bf16* Vf, float* O, float* Opart,
                        float2* ml, DevStatus* stt, cudaStream_t st) {
  const JointSplit s = joint_split(H, n, t, F);
  const dim3 grid(s.nsplit, cdiv(n, kJR), H);
  const JointArgs a{Q, n, Ck, beta, Cv, t, Kf, Vf, F, nullptr, scale, s.per_split, s.nsplit, Opart, ml, O, stt, nullptr, 0.f};
  if (compact_bf16 || t == 0) {
    set_dyn_smem((const void*)attend_warp_kernel<bf16, false>, kJSmem<bf16>);
    launch_chained(attend_warp_kernel<bf16, false>, grid, 32 * kJWarps, kJSmem<bf16>, st, a);
  } else {
    set_dyn_smem((const void*)attend_warp_kernel<float, false>, kJSmem<float>);
    launch_chained(attend_warp_kernel<float, false>, grid, 32 * kJWarps, kJSmem<float>, st, a);
  }
  if (s.nsplit == 1) return 1;
  const long long rows = (long long)H * n;
  launch_chained(attend_combine_kernel, (unsigned)cdiv(rows, 4), 128, 0, st, Opart, ml, n, s.nsplit, rows, O, stt);
  return 2;
}

}  // namespace arckv
