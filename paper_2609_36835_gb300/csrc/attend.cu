// Compact attention (Sec. 3.1 Eq. compact_attention) on the tensor pipe:
//   X = scale Q C_k^T + 1 beta^T   exact bf16 queries against the bf16 triple of
//                                  C_k (kSplit3B), beta added in the epilogue;
//   O = softmax(X) C_v             attend_pv_kernel: the probabilities formed on
//                                  the fly as a bf16 triple against the triple
//                                  of C_v, eight products (fp32-grade).
// Four launches (a fifth sums key splits): the operands' split, X, its row
// statistics, the products.  8 heads, n = 1024, t = 819: 51 us of kernels (5 + 12
// + 10 + 24); 207 before, with beta and the statistics in a pass of 58 us and the
// products one part of C_v at a time from a probability triple in memory.
#include <algorithm>

#include "kernels.h"
#include "tc_gemm.cuh"

namespace arckv {

// The operands' bf16 triples: C_k as it stands (CTAs below `ncopy`, part p of
// element e at ck[p * count + e]), C_v transposed, [3][H][128][ldt] with the pad
// columns zero (32 x 32 tiles).
__global__ void __launch_bounds__(256) attend_operands_kernel(const float* Ck, const float* Cv, bf16* ck, bf16* vt,
                                                              int H, int t, int ldt, int ncopy) {
  chain_wait();
  if ((int)blockIdx.x < ncopy) {
    const long long count = (long long)H * t * 128;
    for (long long e = 4 * ((long long)blockIdx.x * 256 + threadIdx.x); e < count; e += 4LL * ncopy * 256) {
      float x[4];
      if ((((uintptr_t)Ck) & 15) == 0) {
        const float4 v = *(const float4*)(Ck + e);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = Ck[e + q];
      }
      __nv_bfloat162 h[2], m[2], l[2];
      split3_bf16x2(x[0], x[1], h[0], m[0], l[0]);
      split3_bf16x2(x[2], x[3], h[1], m[1], l[1]);
      *(uint2*)(ck + e) = *(const uint2*)h;
      *(uint2*)(ck + count + e) = *(const uint2*)m;
      *(uint2*)(ck + 2 * count + e) = *(const uint2*)l;
    }
    return;
  }
  __shared__ float tile[32][33];
  const int nr = (ldt + 31) / 32;
  int i = (int)blockIdx.x - ncopy;
  const int c0 = (i & 3) * 32;
  i >>= 2;
  const int b = i / nr, r0 = (i - b * nr) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float* sb = Cv + (long long)b * t * 128;
#pragma unroll
  for (int q = ty; q < 32; q += 8) tile[q][tx] = r0 + q < t ? sb[(long long)(r0 + q) * 128 + c0 + tx] : 0.f;
  __syncthreads();
  const long long part = (long long)H * 128 * ldt;
#pragma unroll
  for (int q = ty; q < 32; q += 8)
    if (r0 + tx < ldt) {
      const long long o = ((long long)b * 128 + c0 + q) * ldt + r0 + tx;
      split3_bf16(tile[tx][q], vt[o], vt[part + o], vt[2 * part + o]);
    }
}

// X[b][row][col] = scale acc + beta[b][col] through staged TMA stores, eight
// epilogue warps of 64 columns.
struct TcEpiBias {
  CUtensorMap map;   // box {32, 32, 1}, 128-byte swizzle
  const float* beta;
  float scale;
  int M, N;
  static constexpr int kEpiWarps = 8;
  static constexpr int kStageBytes = 32 * 128;
  struct State {
    uint8_t* stage;
    int* stores;
    const float* be;
    int b, y, n0;
  };
  __device__ __forceinline__ void init(State& s, int b, int row, int n0, int, int) const {
    s.b = b;
    s.y = row & ~31;
    s.n0 = n0;
    s.be = beta + (long long)b * N + n0;
  }
  __device__ __forceinline__ void attach(State& s, uint8_t* stage, int* stores) const {
    s.stage = stage;
    s.stores = stores;
  }
  __device__ __forceinline__ void consume(State& s, int, int j, float (&v)[32]) const {
    const int lane = threadIdx.x & 31;
    const float bl = s.n0 + 32 * j + lane < N ? __ldg(s.be + 32 * j + lane) : 0.f;
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = fmaf(scale, v[q], __shfl_sync(0xffffffffu, bl, q));
    staged_store_32x32<1>(&map, s.stage, s.stores, s.n0 + 32 * j, s.y, s.b, M, N, v, 1.f);
  }
  __device__ __forceinline__ void finish(State&, int, int, int, int, int) const {}
};

// shift = max, mul = 1 / sum exp(x - shift) of the rows of X (pitch ld), one
// warp per row, 16-byte loads (the columns of the last one past t are skipped).
__global__ void __launch_bounds__(256) row_stats_kernel(const float* X, float* shift, float* mul, long long rows, int t,
                                                        int ld) {
  chain_wait();
  const long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const float* x = X + row * ld;
  auto at = [&](int c) {
    float4 v = *(const float4*)(x + c);
    if (c + 4 > t) {
      v.y = c + 1 < t ? v.y : -INFINITY;
      v.z = c + 2 < t ? v.z : -INFINITY;
      v.w = -INFINITY;
    }
    return v;
  };
  float mx = -INFINITY;
#pragma unroll 4
  for (int c = 4 * lane; c < t; c += 128) {
    const float4 v = at(c);
    mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
  }
  mx = warp_max(mx);
  float sm = 0.f;
#pragma unroll 4
  for (int c = 4 * lane; c < t; c += 128) {
    const float4 v = at(c);
    sm += (expf(v.x - mx) + expf(v.y - mx)) + (expf(v.z - mx) + expf(v.w - mx));
  }
  sm = warp_sum(sm);
  if (lane == 0) {
    shift[row] = mx;
    mul[row] = 1.0f / sm;
  }
}

// O = P C_v with P = exp(X - shift) mul formed on the fly.  CTA = (kR query
// rows, key split): TMA streams kR x 64 slabs of X into a raw ring; sixteen
// converter warps form P and its bf16 triple in the K-major layout of an MMA
// operand; per 16-wide K step one thread issues the products of the two
// triples (all but l l, 2^-32 of the result), D [128 dims x kR rows] += C_v^T
// P^T: h h into one accumulator, the others, at most 2^-8 of it, into a second,
// so that the leading sum is rounded once per step.  The value side is M, so that
// a short row tile makes a narrow MMA instead of an idle half.  The products
// are bound by operand bytes (6 KB of shared memory per MMA at kR = 64), a CTA
// by them and the conversion about alike.
namespace {
constexpr int kAvVTile = 128 * 128;   // one part of C_v^T: 128 dims x 64 keys, bf16
constexpr int kAvRS = 3, kAvOS = 2;   // raw and operand ring depths
constexpr int kAvConv = 16;
constexpr int kAvThreads = 32 * (kAvConv + 3);
template <int kR>
constexpr int kAvStage = 3 * (kAvVTile + kR * 128);
template <int kR>
constexpr int kAvSmem = kAvRS * kR * 256 + kAvOS * kAvStage<kR> + 1024;
}  // namespace

template <int kR>
__global__ void __launch_bounds__(kAvThreads, 1)
    attend_pv_kernel(const __grid_constant__ CUtensorMap mX, const __grid_constant__ CUtensorMap mV, const float* shift,
                     const float* mul, float* O, float* parts, int H, int rows, int T, int splits, DevStatus* stt) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t rfull[kAvRS], rempty[kAvRS], vfull[kAvOS], ofull[kAvOS], oempty[kAvOS], accf, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t s0 = tc::smem_u32(smem_raw);
  uint8_t* obase = smem_raw + (((s0 + 1023u) & ~1023u) - s0);   // operand stages: V_h V_m V_l P_h P_m P_l
  uint8_t* rbase = obase + kAvOS * kAvStage<kR>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = (rows + kR - 1) / kR;
  const int tile = blockIdx.x / splits, sp = blockIdx.x - tile * splits;
  const int b = tile / mt, m0 = (tile - b * mt) * kR;
  const int nk = (T + 63) / 64;
  const int kb0 = (int)((long long)nk * sp / splits), nkb = (int)((long long)nk * (sp + 1) / splits) - kb0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kAvRS; ++s) {
      tc::mbar_init(&rfull[s], 1);
      tc::mbar_init(&rempty[s], kAvConv);
    }
    for (int s = 0; s < kAvOS; ++s) {
      tc::mbar_init(&vfull[s], 1);
      tc::mbar_init(&ofull[s], kAvConv);
      tc::mbar_init(&oempty[s], 1);
    }
    tc::mbar_init(&accf, 1);
    tc::mbar_init(&drain, 1);
    abort_flag = 0;
    tc::mbar_fence_init();
  }
  constexpr int kCols = 2 * kR;
  chain_wait();
  if (warp == 1) tc::tmem_alloc(&tmem_slot, kCols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    if (lane == 0) {   // X slabs
      tc::tma_prefetch(&mX);
      int g = 0;
      for (; g < nkb; ++g) {
        const int s = g % kAvRS;
        if (g >= kAvRS && !tc::mbar_wait(&rempty[s], ((g / kAvRS) - 1) & 1, abortp, stt)) break;
        tc::mbar_arrive_expect_tx(&rfull[s], kR * 256);
        tc::tma_load_3d(rbase + s * kR * 256, &mX, (kb0 + g) * 64, m0, b, &rfull[s]);
      }
      volatile int never = 0;
      for (int k = g > kAvRS ? g - kAvRS : 0; k < g; ++k) tc::mbar_wait(&rfull[k % kAvRS], (k / kAvRS) & 1, &never, stt);
    }
  } else if (warp == kAvConv + 2) {
    if (lane == 0) {   // the three parts of C_v^T
      tc::tma_prefetch(&mV);
      int g = 0;
      for (; g < nkb; ++g) {
        const int s = g % kAvOS;
        if (g >= kAvOS && !tc::mbar_wait(&oempty[s], ((g / kAvOS) - 1) & 1, abortp, stt)) break;
        tc::mbar_arrive_expect_tx(&vfull[s], 3 * kAvVTile);
        for (int p = 0; p < 3; ++p)
          tc::tma_load_3d(obase + s * kAvStage<kR> + p * kAvVTile, &mV, (kb0 + g) * 64, 0, p * H + b, &vfull[s]);
      }
      volatile int never = 0;
      for (int k = g > kAvOS ? g - kAvOS : 0; k < g; ++k) tc::mbar_wait(&vfull[k % kAvOS], (k / kAvOS) & 1, &never, stt);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16_f32(kR);
      bool ok = true;
      for (int g = 0; g < nkb && ok; ++g) {
        const int s = g % kAvOS;
        const uint32_t ph = (g / kAvOS) & 1;
        if (!tc::mbar_wait(&vfull[s], ph, abortp, stt) || !tc::mbar_wait(&ofull[s], ph, abortp, stt)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t v = tc::smem_u32(obase + s * kAvStage<kR>), p = v + 3 * kAvVTile;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
          for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j)
              if (i + j < 4)
                tc::mma_f16(tmem + (i + j > 0 ? kR : 0), tc::sdesc_k128(v + i * kAvVTile + ks * 32),
                            tc::sdesc_k128(p + j * kR * 128 + ks * 32), idesc,
                            (g > 0 || ks > 0 || i + j > 1 || (i == 1 && j == 0)) ? 1u : 0u);
        tc::mma_commit(&oempty[s]);
      }
      if (ok) tc::mma_commit(&accf);
      tc::mma_commit(&drain);
      volatile int never = 0;
      tc::mbar_wait(&drain, 0, &never, stt);
    }
  } else {
    // converters: warp cw owns kR / 16 rows, two at a time (lanes 0-15 the
    // first), four keys per lane
    constexpr int kSteps = kR / 32;
    const int cw = warp - 2, hl = lane >> 4, cl = lane & 15;
    float zl[kSteps], mu[kSteps];   // shift and scale (0, 0 past the end: P = 0)
#pragma unroll
    for (int u = 0; u < kSteps; ++u) {
      const int row = m0 + cw * (kR / 16) + 2 * u + hl;
      const bool in = row < rows;
      zl[u] = in ? shift[(long long)b * rows + row] : 0.f;
      mu[u] = in ? mul[(long long)b * rows + row] : 0.f;
    }
    bool ok = true;
    for (int g = 0; g < nkb; ++g) {
      const int rs = g % kAvRS, os = g % kAvOS;
      ok = tc::mbar_wait(&rfull[rs], (g / kAvRS) & 1, abortp, stt);
      if (ok && g >= kAvOS) ok = tc::mbar_wait(&oempty[os], ((g / kAvOS) - 1) & 1, abortp, stt);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const float* R = (const float*)(rbase + rs * kR * 256);
      uint8_t* P = obase + os * kAvStage<kR> + 3 * kAvVTile;
      const int c = (kb0 + g) * 64 + 4 * cl;
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int r = cw * (kR / 16) + 2 * u + hl;
        const float4 x = *(const float4*)(R + r * 64 + 4 * cl);
        float p[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) p[e] = c + e < T ? expf(p[e] - zl[u]) * mu[u] : 0.f;
        __nv_bfloat162 h[2], m[2], l[2];
        split3_bf16x2(p[0], p[1], h[0], m[0], l[0]);
        split3_bf16x2(p[2], p[3], h[1], m[1], l[1]);
        // 128-byte swizzle: 16-byte chunk cl / 2 of row r sits at chunk (cl / 2) ^ (r % 8)
        const uint32_t off = (uint32_t)r * 128u + ((((uint32_t)cl >> 1) ^ ((uint32_t)r & 7u)) << 4) +
                             (((uint32_t)cl & 1u) << 3);
        *(uint2*)(P + off) = *(const uint2*)h;
        *(uint2*)(P + kR * 128 + off) = *(const uint2*)m;
        *(uint2*)(P + 2 * kR * 128 + off) = *(const uint2*)l;
      }
      tc::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tc::mbar_arrive(&rempty[rs]);
        tc::mbar_arrive(&ofull[os]);
      }
    }
    if (ok) ok = tc::mbar_wait(&accf, 0, abortp, stt);
    ok = __all_sync(0xffffffffu, ok);
    const int qd = warp & 3, cg = cw >> 2;   // TMEM lane quarter (32 dims); 16-row group
    if (ok && cg * 16 < kR) {
      tc::fence_after_sync();
      bool bad = false;
      for (int g16 = cg * 16; g16 < kR; g16 += 64) {
        float v[16], u[16];
        tc::tmem_ld16(tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)g16, v);
        tc::tmem_ld16(tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(kR + g16), u);
        float* d = (splits > 1 ? parts + (long long)sp * H * rows * 128 : O) + ((long long)b * rows + m0 + g16) * 128 +
                   qd * 32 + lane;
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (m0 + g16 + e < rows) {
            const float o = v[e] + u[e];
            d[e * 128] = o;
            bad |= !isfinite(o);
          }
      }
      if (bad) set_status(stt, ARCKV_ERR_NONFINITE);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kCols);
  }
}

// O = the splits' products added in order; non-finite sums are recorded.
__global__ void __launch_bounds__(256) sum_parts_kernel(const float* P, float* O, long long count, int splits,
                                                        DevStatus* stt) {
  chain_wait();
  bool bad = false;
  for (long long k = blockIdx.x * 256LL + threadIdx.x; k < count; k += 256LL * gridDim.x) {
    float a = P[k];
    for (int s = 1; s < splits; ++s) a += P[s * count + k];
    O[k] = a;
    bad |= !isfinite(a);
  }
  if (bad) set_status(stt, ARCKV_ERR_NONFINITE);
}

constexpr int kAvMaxSplits = 3;

AttendLayout attend_layout(int H, int n, int t) {
  AttendLayout L{};
  const size_t h = H, ldt = (size_t)(t + 7) / 8 * 8;
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t r = o; o += (bytes + 255) / 256 * 256; return r; };
  L.status = take(256);
  L.X = take(h * n * (size_t)logit_ld(t) * 4);
  L.shift = take(h * n * 4);
  L.mul = take(h * n * 4);
  L.ck3 = take(3 * h * t * 128 * 2);
  L.vt3 = take(3 * h * 128 * ldt * 2);
  L.parts = take(kAvMaxSplits * h * n * 128 * 4);
  L.total = o;
  return L;
}

template <int kR>
static cudaError_t launch_attend_pv(int H, int n, int t, const float* X, const float* shift, const float* mul,
                                    const bf16* vt, float* O, float* parts, int splits, DevStatus* stt,
                                    cudaStream_t st) {
  const int ld = logit_ld(t), ldt = (t + 7) / 8 * 8;
  CUtensorMap mX, mV;
  if (!encode_f32_map_3d(&mX, X, t, n, H, 64, kR, ld, (uint64_t)n * ld) ||
      !encode_bf16_map_3d(&mV, vt, ldt, 128, 3ull * H, 128))
    return cudaErrorInvalidValue;
  auto kern = attend_pv_kernel<kR>;
  const cudaError_t e = set_dyn_smem((const void*)kern, kAvSmem<kR>);
  if (e != cudaSuccess) return e;
  launch_chained(kern, H * cdiv(n, kR) * splits, kAvThreads, kAvSmem<kR>, st, mX, mV, shift, mul, O, parts, H, n, t, splits, stt);
  return cudaGetLastError();
}

int launch_attend(int H, int n, int t, float scale, const bf16* Q, const float* C_k, const float* beta,
                  const float* C_v, float* O, char* ws, DevStatus* stt, cudaStream_t st) {
  const AttendLayout L = attend_layout(H, n, t);
  const long long htd = (long long)H * t * 128, rows = (long long)H * n;
  const int ldt = (t + 7) / 8 * 8, ld = logit_ld(t), sms = tc_gemm_sm_count();
  float* X = (float*)(ws + L.X);
  float* shift = (float*)(ws + L.shift);
  float* mul = (float*)(ws + L.mul);
  bf16* ck = (bf16*)(ws + L.ck3);
  bf16* vt = (bf16*)(ws + L.vt3);
  float* parts = (float*)(ws + L.parts);
  const int ncopy = stride_grid(htd, 4 * 256, 4);
  launch_chained(attend_operands_kernel, ncopy + 4 * H * cdiv(ldt, 32), 256, 0, st, C_k, C_v, ck, vt, H, t, ldt, ncopy);
  {
    CUtensorMap mA, mB, mB2, mB3;
    TcEpiBias epi{};
    epi.beta = beta;
    epi.scale = scale;
    epi.M = n;
    epi.N = t;
    if (!encode_bf16_map_3d(&mA, Q, 128, n, H, 128) || !encode_bf16_map_3d(&mB, ck, 128, t, H, 128) ||
        !encode_bf16_map_3d(&mB2, ck + htd, 128, t, H, 128) || !encode_bf16_map_3d(&mB3, ck + 2 * htd, 128, t, H, 128) ||
        !encode_f32_map_3d(&epi.map, X, t, n, H, 32, 32, ld, (uint64_t)n * ld, true))
      return -1;
    if (launch_tc_gemm<128, kSplit3B>(mA, mB, mA, mB2, epi, H, n, t, 128, 128, stt, st, 0, &mB3) != cudaSuccess)
      return -1;
  }
  launch_chained(row_stats_kernel, (unsigned)cdiv(rows, 8), 256, 0, st, X, shift, mul, rows, t, ld);
  // 64-row tiles where they fill the SMs, else 32-row ones, and key splits
  // (of four slabs or more) for what is still idle
  const int tiles64 = H * cdiv(n, 64), tiles32 = H * cdiv(n, 32), nk = cdiv(t, 64);
  const bool small = 4 * tiles64 < 3 * sms;
  const int splits = std::max(1, std::min({kAvMaxSplits, sms / (small ? tiles32 : tiles64), nk / 4}));
  const cudaError_t e = small ? launch_attend_pv<32>(H, n, t, X, shift, mul, vt, O, parts, splits, stt, st)
                              : launch_attend_pv<64>(H, n, t, X, shift, mul, vt, O, parts, splits, stt, st);
  if (e != cudaSuccess) return -1;
  if (splits == 1) return 4;
  launch_chained(sum_parts_kernel, stride_grid(rows * 128, 256, 8), 256, 0, st, parts, O, rows * 128, splits, stt);
  return 5;
}

}  // namespace arckv
