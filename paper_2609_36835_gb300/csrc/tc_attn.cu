// Softmax attention products on tcgen05 with fp32-grade accuracy:
//
//   value-attention logits (U_q q_i).(U_k k_j) = q''_i . k_j,
//       q''_i = U_k^T (U_q q_i)                       (Eq. value_context)
//   A V and softmax(l) V with A, softmax(l) row-stochastic and V the bf16 cache
//                                                     (Eq. value_context, Eq. value_lstsq's Y)
//
// In every product one operand is an exact bf16 input (K or V) and the other
// an fp32 value, which enters as a bf16 triple (h, m, l) summing to it within
// 2^-24; the kSplit3A GEMM issues h*B + m*B + l*B.
#include "kernels.h"
#include "tc_gemm.cuh"

namespace arckv {

__global__ void split3_kernel(const float* x, bf16* h, bf16* m, bf16* l, long long count) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
       k += (long long)gridDim.x * blockDim.x)
    split3_bf16(x[k], h[k], m[k], l[k]);
}

// VT[b][d][j] = V[b][j][d] (bf16), zero for T <= j < ldT.
__global__ void __launch_bounds__(256) transpose_v_kernel(const bf16* V, bf16* VT, int T, int ldT) {
  chain_wait();
  const int b = blockIdx.z, j0 = blockIdx.x * 32, d0 = blockIdx.y * 32;
  __shared__ bf16 tile[32][34];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const bf16 zero = __float2bfloat16_rn(0.f);
  for (int q = ty; q < 32; q += 8) {
    const int j = j0 + q;
    tile[q][tx] = (j < T) ? V[((long long)b * T + j) * 128 + d0 + tx] : zero;
  }
  __syncthreads();
  for (int q = ty; q < 32; q += 8) {
    const int j = j0 + tx;
    if (j < ldT) VT[((long long)b * 128 + d0 + q) * ldT + j] = tile[tx][q];
  }
}

int launch_value_logits_tc(const Dims& D, const bf16* q_h, const bf16* q_m, const bf16* q_l, const bf16* K,
                           float* logits, float2* part, DevStatus* stt, cudaStream_t st) {
  CUtensorMap mA, mA2, mA3, mB;
  if (!encode_bf16_map_3d(&mA, q_h, 128, D.n, D.H, 128) || !encode_bf16_map_3d(&mA2, q_m, 128, D.n, D.H, 128) ||
      !encode_bf16_map_3d(&mA3, q_l, 128, D.n, D.H, 128) || !encode_bf16_map_3d(&mB, K, 128, D.T, D.H, 128))
    return -1;
  if (launch_tc_logits_rowpart<kSplit3A>(mA, mB, mA2, mA, &mA3, logits, 1.f, part, D.H, D.n, D.T, 128, stt, st) !=
      cudaSuccess)
    return -1;
  return 1;
}

int launch_split3(const float* x, bf16* h, bf16* m, bf16* l, long long count, cudaStream_t st) {
  launch_chained(split3_kernel, stride_grid(count, 256, 8), 256, 0, st, x, h, m, l, count);
  return 1;
}

int launch_transpose_v(const Dims& D, const bf16* V, bf16* VT, cudaStream_t st) {
  const int ldT = (D.T + 7) / 8 * 8;
  launch_chained(transpose_v_kernel, dim3(cdiv(ldT, 32), 4, D.H), 256, 0, st, V, VT, D.T, ldT);
  return 1;
}

// ---------------------------------------------------------------------------
// Fused O = P V with P = exp(X - shift_row) * mul_row, X the fp32 logits
// [H][rows][T] and V the bf16 cache (as V^T [H][128][ldT]).  P never reaches
// memory: TMA streams 128 x 64 slabs of X into a raw ring; sixteen converter
// warps form P there (e^x as 2^(x log2 e), one MUFU op per element), split it into the bf16 triple (h, m, l) and write the
// three operand tiles straight into the 128-byte-swizzled K-major layout the
// MMA reads; one thread issues h V + m V + l V per 16-wide K step into a
// 128 x 128 fp32 TMEM accumulator; a fifth warp streams the V^T slabs.
//
// kExpf takes e^x by expf after the subtraction: the form that T % 4 != 0 has
// always had, kept so that its anchors stay what they were.
//
// CTA = (row tile, K split); with two K splits the halves are added into a
// zeroed output with fp32 atomics (two addends onto 0: the sum does not depend
// on their order).  A row tile has kRows = 128, 64 or 32 rows: a slab's time is
// the converters', so a call that leaves SMs idle takes shorter tiles, each
// still one M = 128 MMA whose other rows are ignored (the results keep their
// bits; 2 row tiles x 2 at n = 256, T = 1024: 20 us, as 8 x 2: 11).
namespace {
constexpr int kPvTile = 128 * 128;          // one bf16 128 x 64 operand tile
constexpr int kPvRS = 3;                    // raw ring depth
constexpr int kPvOS = 2;                    // operand ring depth (h, m, l, V^T)
constexpr int kPvOpBytes = 4 * kPvTile;
constexpr int kPvConv = 16;                 // converter warps 2..17, kRows / 16 rows each
constexpr int kPvThreads = 32 * (kPvConv + 3);
constexpr int kPvSmem = kPvRS * 128 * 64 * 4 + kPvOS * kPvOpBytes + 1024;
}  // namespace

template <bool kSkip, bool kExpf, int kRows>
__global__ void __launch_bounds__(kPvThreads, 1)
    probs_v_kernel(const __grid_constant__ CUtensorMap mX, const __grid_constant__ CUtensorMap mVT,
                   const float* shift, const float* mul, const int* skip, float* O, int rows, int T, int splits,
                   DevStatus* stt) {
  constexpr int kPvRawBytes = kRows * 64 * 4;   // one fp32 slab of X
  constexpr int kSteps = kRows / 32;            // two rows of a warp at a time
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t rfull[kPvRS], rempty[kPvRS], vfull[kPvOS], ofull[kPvOS], oempty[kPvOS], accf, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t r0 = tc::smem_u32(smem_raw);
  uint8_t* rbase = smem_raw + (((r0 + 1023u) & ~1023u) - r0);
  uint8_t* obase = rbase + kPvRS * kPvRawBytes;   // 1024-byte aligned: the ring is a multiple of 1 KB
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = (rows + kRows - 1) / kRows;
  const int tile = blockIdx.x / splits, sp = blockIdx.x - tile * splits;
  const int b = tile / mt, m0 = (tile - b * mt) * kRows;
  const int nk = (T + 63) / 64;
  const int kb0 = (int)((long long)nk * sp / splits), kb1 = (int)((long long)nk * (sp + 1) / splits);
  const int nkb = kb1 - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPvRS; ++s) {
      tc::mbar_init(&rfull[s], 1);
      tc::mbar_init(&rempty[s], kPvConv);
    }
    for (int s = 0; s < kPvOS; ++s) {
      tc::mbar_init(&vfull[s], 1);
      tc::mbar_init(&ofull[s], kPvConv);
      tc::mbar_init(&oempty[s], 1);
    }
    tc::mbar_init(&accf, 1);
    tc::mbar_init(&drain, 1);
    abort_flag = 0;
    tc::mbar_fence_init();
  }
  chain_wait();
  if (warp == 1) tc::tmem_alloc(&tmem_slot, 128);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // X slabs
    if (lane == 0) {
      tc::tma_prefetch(&mX);
      int g = 0;
      for (; g < nkb; ++g) {
        const int s = g % kPvRS;
        if (g >= kPvRS && !tc::mbar_wait(&rempty[s], ((g / kPvRS) - 1) & 1, abortp, stt)) break;
        tc::mbar_arrive_expect_tx(&rfull[s], kPvRawBytes);
        tc::tma_load_3d(rbase + s * kPvRawBytes, &mX, (kb0 + g) * 64, m0, b, &rfull[s]);
      }
      volatile int never = 0;
      for (int k = g > kPvRS ? g - kPvRS : 0; k < g; ++k) tc::mbar_wait(&rfull[k % kPvRS], (k / kPvRS) & 1, &never, stt);
    }
  } else if (warp == kPvConv + 2) {
    // V^T slabs
    if (lane == 0) {
      tc::tma_prefetch(&mVT);
      int g = 0;
      for (; g < nkb; ++g) {
        const int s = g % kPvOS;
        if (g >= kPvOS && !tc::mbar_wait(&oempty[s], ((g / kPvOS) - 1) & 1, abortp, stt)) break;
        tc::mbar_arrive_expect_tx(&vfull[s], kPvTile);
        tc::tma_load_3d(obase + s * kPvOpBytes + 3 * kPvTile, &mVT, (kb0 + g) * 64, 0, b, &vfull[s]);
      }
      volatile int never = 0;
      for (int k = g > kPvOS ? g - kPvOS : 0; k < g; ++k) tc::mbar_wait(&vfull[k % kPvOS], (k / kPvOS) & 1, &never, stt);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16_f32(128);
      bool ok = true;
      for (int g = 0; g < nkb && ok; ++g) {
        const int s = g % kPvOS;
        const uint32_t ph = (g / kPvOS) & 1;
        if (!tc::mbar_wait(&vfull[s], ph, abortp, stt) || !tc::mbar_wait(&ofull[s], ph, abortp, stt)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t a = tc::smem_u32(obase + s * kPvOpBytes), bv = a + 3 * kPvTile;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint64_t bd = tc::sdesc_k128(bv + ks * 32);
#pragma unroll
          for (int part = 0; part < 3; ++part)
            tc::mma_f16(tmem, tc::sdesc_k128(a + part * kPvTile + ks * 32), bd, idesc,
                        (g > 0 || ks > 0 || part > 0) ? 1u : 0u);
        }
        tc::mma_commit(&oempty[s]);
      }
      if (ok) tc::mma_commit(&accf);
      tc::mma_commit(&drain);
      volatile int never = 0;
      tc::mbar_wait(&drain, 0, &never, stt);
    }
  } else {
    // converters: warp cw owns kRows / 16 consecutive rows of the tile, two rows per
    // step (lanes 0-15 the first, 16-31 the second), four columns per lane
    const int cw = warp - 2, hl = lane >> 4, cl = lane & 15;
    float zl[kSteps], mu[kSteps];   // per step: shift * log2 e and scale of this lane's row (0, 0 past the end: P = 0)
    int sk[kSteps];
#pragma unroll
    for (int u = 0; u < kSteps; ++u) {
      const int row = m0 + cw * (kRows / 16) + 2 * u + hl;
      zl[u] = 0.f;
      mu[u] = 0.f;
      sk[u] = -1;
      if (row < rows) {
        const long long rr = (long long)b * rows + row;
        zl[u] = kExpf ? shift[rr] : shift[rr] * kLog2e;
        mu[u] = mul[rr];
        if (kSkip) sk[u] = skip[rr];
      }
    }
    bool ok = true;
    for (int g = 0; g < nkb; ++g) {
      const int rs = g % kPvRS, os = g % kPvOS;
      ok = tc::mbar_wait(&rfull[rs], (g / kPvRS) & 1, abortp, stt);
      if (ok && g >= kPvOS) ok = tc::mbar_wait(&oempty[os], ((g / kPvOS) - 1) & 1, abortp, stt);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const float* R = (const float*)(rbase + rs * kPvRawBytes);
      uint8_t* A = obase + os * kPvOpBytes;
      const int c = (kb0 + g) * 64 + 4 * cl;   // this lane's first column
      const bool edge = kSkip || c + 4 > T;
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int r = cw * (kRows / 16) + 2 * u + hl;
        const float4 x = *(const float4*)(R + r * 64 + 4 * cl);
        auto prob = [&](float v) {
          return (kExpf ? expf(v - zl[u]) : ex2_approx(fmaf(v, kLog2e, -zl[u]))) * mu[u];
        };
        float p[4] = {prob(x.x), prob(x.y), prob(x.z), prob(x.w)};
        if (edge) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (c + e >= T || c + e == sk[u]) p[e] = 0.f;
        }
        __nv_bfloat162 h0, m0_, l0, h1, m1, l1;
        split3_bf16x2(p[0], p[1], h0, m0_, l0);
        split3_bf16x2(p[2], p[3], h1, m1, l1);
        // 128-byte swizzle: 16-byte chunk cl / 2 of row r sits at chunk (cl / 2) ^ (r % 8)
        const uint32_t off = (uint32_t)r * 128u + ((((uint32_t)cl >> 1) ^ ((uint32_t)r & 7u)) << 4) +
                             (((uint32_t)cl & 1u) << 3);
        *(uint2*)(A + off) = make_uint2(*(uint32_t*)&h0, *(uint32_t*)&h1);
        *(uint2*)(A + kPvTile + off) = make_uint2(*(uint32_t*)&m0_, *(uint32_t*)&m1);
        *(uint2*)(A + 2 * kPvTile + off) = make_uint2(*(uint32_t*)&l0, *(uint32_t*)&l1);
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
    if (ok && (warp & 3) * 32 < kRows) {
      tc::fence_after_sync();
      const int qd = warp & 3, cg = cw >> 2;   // TMEM lane quarter; 32-column group
      const int row = m0 + qd * 32 + lane;
      float v[32];
      tc::tmem_ld32(tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cg * 32), v);
      if (row < rows) {
        float* d = O + ((long long)b * rows + row) * 128 + cg * 32;
        if (splits > 1) {
#pragma unroll
          for (int e = 0; e < 32; ++e) atomicAdd(d + e, v[e]);
        } else {
#pragma unroll
          for (int e = 0; e < 32; e += 4) *(float4*)(d + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 128);
  }
}

template <int kRows>
static cudaError_t launch_probs_v_rows(const Dims& D, const float* X, const float* shift, const float* mul,
                                       const CUtensorMap& mVT, float* out, int splits, DevStatus* stt, cudaStream_t st,
                                       const int* skip) {
  const int ld = logit_ld(D.T);
  CUtensorMap mX;
  if (!encode_f32_map_3d(&mX, X, D.T, D.n, D.H, 64, kRows, ld, (uint64_t)D.n * ld)) return cudaErrorInvalidValue;
  const bool odd = (D.T & 3) != 0;
  auto kern = skip ? (odd ? probs_v_kernel<true, true, kRows> : probs_v_kernel<true, false, kRows>)
                   : (odd ? probs_v_kernel<false, true, kRows> : probs_v_kernel<false, false, kRows>);
  const cudaError_t e = set_dyn_smem((const void*)kern, kPvSmem);
  if (e != cudaSuccess) return e;
  launch_chained(kern, D.H * cdiv(D.n, kRows) * splits, kPvThreads, kPvSmem, st, mX, mVT, shift, mul, skip, out, D.n, D.T, splits,
                                                                     stt);
  return cudaGetLastError();
}

int launch_probs_v_tc(const Dims& D, const float* X, const float* shift, const float* mul, const bf16* VT, float* out,
                      DevStatus* stt, cudaStream_t st, const int* skip) {
  if (((uintptr_t)X & 15u) != 0 || ((uintptr_t)out & 15u) != 0) return -1;
  const int ldT = (D.T + 7) / 8 * 8, sms = tc_gemm_sm_count();
  CUtensorMap mVT;
  if (!encode_bf16_map_3d(&mVT, VT, ldT, 128, D.H, 128)) return -1;
  const int tiles = D.H * cdiv(D.n, 128), nk = cdiv(D.T, 64);
  // (T % 4 != 0 never had its sums split, and the fits amplify their rounding a
  // hundredfold: it keeps one K range and takes shorter row tiles alone)
  const int splits = (2 * tiles <= sms && nk >= 2 && (D.T & 3) == 0) ? 2 : 1;
  if (splits > 1 && cudaMemsetAsync(out, 0, sizeof(float) * (size_t)D.H * D.n * 128, st) != cudaSuccess) return -1;
  const cudaError_t e =
      4 * tiles * splits <= sms   ? launch_probs_v_rows<32>(D, X, shift, mul, mVT, out, splits, stt, st, skip)
      : 2 * tiles * splits <= sms ? launch_probs_v_rows<64>(D, X, shift, mul, mVT, out, splits, stt, st, skip)
                                  : launch_probs_v_rows<128>(D, X, shift, mul, mVT, out, splits, stt, st, skip);
  return e == cudaSuccess ? 1 : -1;
}

}  // namespace arckv
