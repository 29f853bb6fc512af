// Tensor-core stages of Sec. 3.4:
//   * reference logits l = scale Q K^T (bf16 operands are exact, one MMA per
//     product, fp32 accumulation);
//   * the anchor assignment kappa(j) = argmax_r u_j . u_{s_r}
//     (Eq. anchor_assignment) as a split-bf16 GEMM of the transposed profiles
//     U^T [T x n] against the anchor rows U_S^T [t x n] whose epilogue keeps
//     the row maximum (lowest r on ties) and merges it across column tiles
//     with a 64-bit atomicMax; the T x t similarity is never stored.
#include <algorithm>

#include "kernels.h"
#include "tc_gemm.cuh"

namespace arckv {

struct TcEpiArgmax {
  unsigned long long* best;
  long long bbs;
  struct State {
    float bv;
    int bi, ncols, n0;
    bool row_ok;
  };
  __device__ __forceinline__ void init(State& s, int, int row, int n0, int M, int N) const {
    s.bv = -INFINITY;
    s.bi = -1;
    s.ncols = N - n0;
    s.n0 = n0;
    s.row_ok = row < M;
  }
  __device__ __forceinline__ void consume(State& s, int, int j, float (&v)[32]) const {
#pragma unroll
    for (int q = 0; q < 32; ++q)
      if (j * 32 + q < s.ncols && v[q] > s.bv) {
        s.bv = v[q];
        s.bi = s.n0 + j * 32 + q;
      }
  }
  __device__ __forceinline__ void finish(State& s, int b, int row, int, int, int) const {
    if (!s.row_ok || s.bi < 0) return;
    const unsigned long long key =
        ((unsigned long long)f32_ordered(s.bv) << 32) | (unsigned long long)(0xffffffffu - (unsigned int)s.bi);
    atomicMax(best + (long long)b * bbs + row, key);
  }
};

// The same with eight epilogue warps, two per TMEM lane quarter, for 256-wide
// tiles (each warp takes 128 columns).  gate (nullable): a non-zero word there
// closes the launch (the filter has taken the call).
struct TcEpiArgmax8 : TcEpiArgmax {
  static constexpr int kEpiWarps = 8;
  const int* gate;
  __device__ __forceinline__ bool closed() const { return gate != nullptr && __ldcg(gate) != 0; }
};

int launch_ref_logits_tc(const Dims& D, float scale, const bf16* Q, const bf16* K, float* L, float2* part,
                         DevStatus* stt, cudaStream_t st) {
  CUtensorMap mA, mB;
  if (!encode_bf16_map_3d(&mA, Q, D.d, D.n, D.H, 128) || !encode_bf16_map_3d(&mB, K, D.d, D.T, D.H, 128)) return -1;
  if (launch_tc_logits_rowpart<kPlain>(mA, mB, mA, mB, nullptr, L, scale, part, D.H, D.n, D.T, D.d, stt, st) !=
      cudaSuccess)
    return -1;
  return 1;
}

// Where key j's profile row goes.  An anchor's (anchors[r] == j) to row r of
// the anchor rows U_S^T; every other key to row j - #{anchors < j} of the
// compacted key rows, the T - t rows the assignment GEMM takes as M: the
// anchors' own assignment is fixed, kappa(s_r) = r, so their GEMM rows would
// only be discarded.  ab: the head's anchors, ascending (checked upstream).
// The element offset of that row (an anchor row as -1 - offset), or
// kNoRow when invalid anchors (a caller's, already flagged
// ARCKV_ERR_INVALID_ARG) leave no valid row.
constexpr long long kNoRow = -(1ll << 62);
__device__ __forceinline__ long long profile_row(const int* ab, int t, int T, int b, int j, int ldn, int* kmap) {
  int lo = 0, hi = t;   // first index with ab[index] >= j
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ab[mid] < j) lo = mid + 1;
    else hi = mid;
  }
  if (lo < t && ab[lo] == j) return -1 - ((long long)b * t + lo) * ldn;
  const int r = j - lo;
  if (r < 0 || r >= T - t) return kNoRow;
  kmap[(long long)b * T + r] = j;
  return ((long long)b * T + r) * ldn;
}

// Output rows of the profiles: key rows (Ut, compacted) or anchor rows (S),
// and the compacted row -> key map.
struct ProfileOut {
  bf16 *Ut_hi, *Ut_lo, *S_hi, *S_lo;
  int* kmap;           // [H][T]: key of compacted row c (c < T - t)
  const int* anchors;  // [H][t]
  int t;
  // filter (nullable): upper bounds of ||u - bf16(u)|| of the key rows [H][T]
  // (compacted like Ut) and of the anchor rows [H][ldr]
  float *rho_k, *rho_s;
  int ldr;
};

// The bound of one profile row (output offset ro) from its residual's sum of squares.
__device__ __forceinline__ void write_rho(const ProfileOut& po, int b, int T, int ldn, long long ro, float sq) {
  const float r = sqrtf(sq) * 1.001f;   // (the fp32 sum of squares is good to 1e-4)
  if (ro >= 0) po.rho_k[(long long)b * T + (ro / ldn - (long long)b * T)] = r;
  else po.rho_s[(long long)b * po.ldr + ((-1 - ro) / ldn - (long long)b * po.t)] = r;
}

// Column statistics of the reference logits and the transposed response
// profiles (Sec. 3.4, Eq. response_profile), one CTA per (32 columns, head):
//   pass 1: per column the online (M_j, s1, s2) over the n rows, the 16 row
//     slices (warps) combined in slice order,
//       M_j = max_i l_ij,  s1 = sum_i e^{l_ij - M_j},  s2 = sum_i e^{2(l_ij - M_j)},
//       log phi_j = M_j + log s1 - log n  (the mass of Eq. mass_centroid),
//       invN_j = 1 / sqrt(s2);
//   pass 2 (Ut_hi given): U_ij = e^{l_ij - M_j} invN_j, re-read from L2 (the
//     strip was just streamed in), split into bf16 (hi, lo) and written
//     transposed, Ut[b][j][i] (row stride ldn >= n, a multiple of 8; the pad
//     columns n..ldn-1 are written as zeros).
// e^x is taken as 2^(x log2 e) after the subtraction.
__global__ void __launch_bounds__(512) col_profiles_kernel(const float* L, float* logphi, ProfileOut po, int n, int T,
                                                           int ld, int ldn) {
  chain_wait();
  const int b = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j0 = blockIdx.x * 32, j = j0 + lane;
  __shared__ float red[3][16][32];
  __shared__ float cstat[2][32];
  __shared__ float tile[64][33];
  __shared__ long long orow[32];   // element offset of each column's output row
  if (po.Ut_hi != nullptr && w == 0 && j < T)
    orow[lane] = profile_row(po.anchors + (long long)b * po.t, po.t, T, b, j, ldn, po.kmap);
  const float* Lb = L + (long long)b * n * ld + j;
  float mx = -INFINITY, s1 = 0.f, s2 = 0.f;
  if (j < T) {
    int i = w;
    for (; i + 48 < n; i += 64) {   // rows i, i + 16, i + 32, i + 48: one rescale per step
      const float v0 = Lb[(long long)i * ld], v1 = Lb[(long long)(i + 16) * ld];
      const float v2 = Lb[(long long)(i + 32) * ld], v3 = Lb[(long long)(i + 48) * ld];
      const float m4 = fmaxf(fmaxf(v0, v1), fmaxf(v2, v3));
      if (m4 > mx) {
        const float r = (mx == -INFINITY) ? 0.f : ex2_approx((mx - m4) * kLog2e);
        s1 *= r;
        s2 *= r * r;
        mx = m4;
      }
      const float e0 = ex2_approx((v0 - mx) * kLog2e), e1 = ex2_approx((v1 - mx) * kLog2e);
      const float e2 = ex2_approx((v2 - mx) * kLog2e), e3 = ex2_approx((v3 - mx) * kLog2e);
      s1 += (e0 + e1) + (e2 + e3);
      s2 += (e0 * e0 + e1 * e1) + (e2 * e2 + e3 * e3);
    }
    for (; i < n; i += 16) {
      const float v = Lb[(long long)i * ld];
      if (v > mx) {
        const float r = (mx == -INFINITY) ? 0.f : ex2_approx((mx - v) * kLog2e);
        s1 = fmaf(s1, r, 1.f);
        s2 = fmaf(s2, r * r, 1.f);
        mx = v;
      } else {
        const float e = ex2_approx((v - mx) * kLog2e);
        s1 += e;
        s2 = fmaf(e, e, s2);
      }
    }
  }
  red[0][w][lane] = mx;
  red[1][w][lane] = s1;
  red[2][w][lane] = s2;
  __syncthreads();
  if (w == 0) {
    float M = -INFINITY;
    for (int q = 0; q < 16; ++q) M = fmaxf(M, red[0][q][lane]);
    float S1 = 0.f, S2 = 0.f;
    for (int q = 0; q < 16; ++q) {
      if (red[0][q][lane] == -INFINITY) continue;
      const float r = ex2_approx((red[0][q][lane] - M) * kLog2e);
      S1 = fmaf(red[1][q][lane], r, S1);
      S2 = fmaf(red[2][q][lane], r * r, S2);
    }
    if (j < T) logphi[(long long)b * T + j] = M + logf(S1) - logf((float)n);
    cstat[0][lane] = M;
    cstat[1][lane] = j < T ? 1.0f / sqrtf(S2) : 0.f;
  }
  __syncthreads();
  if (po.Ut_hi == nullptr) return;
  const float cm = cstat[0][lane], ci = cstat[1][lane];
  float rsq[2] = {0.f, 0.f};
  for (int i0 = 0; i0 < ldn; i0 += 64) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = w + 16 * k, i = i0 + r;
      tile[r][lane] = (i < n && j < T) ? ex2_approx((Lb[(long long)i * ld] - cm) * kLog2e) * ci : 0.f;
    }
    __syncthreads();
    // warp w writes columns 2w and 2w + 1, lane l rows i0 + 2l and i0 + 2l + 1 (ldn even)
#pragma unroll
    for (int c = 2 * w; c < 2 * w + 2; ++c) {
      const int jj = j0 + c, i = i0 + 2 * lane;
      if (jj < T && i < ldn && orow[c] != kNoRow) {
        bf16 h0, l0, h1, l1;
        split_bf16(tile[2 * lane][c], h0, l0);
        split_bf16(tile[2 * lane + 1][c], h1, l1);
        const float e0 = tile[2 * lane][c] - __bfloat162float(h0), e1 = tile[2 * lane + 1][c] - __bfloat162float(h1);
        rsq[c & 1] = fmaf(e0, e0, fmaf(e1, e1, rsq[c & 1]));
        const long long ro = orow[c];
        bf16* dh = ro >= 0 ? po.Ut_hi + ro : po.S_hi + (-1 - ro);
        bf16* dl = ro >= 0 ? po.Ut_lo + ro : po.S_lo + (-1 - ro);
        *(__nv_bfloat162*)(dh + i) = __halves2bfloat162(h0, h1);
        *(__nv_bfloat162*)(dl + i) = __halves2bfloat162(l0, l1);
      }
    }
    __syncthreads();
  }
  if (po.rho_k != nullptr) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float sq = warp_sum(rsq[k]);
      const int c = 2 * w + k;
      if (lane == 0 && j0 + c < T && orow[c] != kNoRow) write_rho(po, b, T, ldn, orow[c], sq);
    }
  }
}

// col_profiles_kernel with the n x W strip of l staged in shared memory by
// TMA (boxes of 256 rows x W columns, one mbarrier), so l crosses HBM once.
// Thread t owns column t % W and the rows congruent to t / W modulo 512 / W
// (the row phases are combined in order): pass 1 takes the column maxima,
// pass 2 overwrites the strip with e^{l - M_j} while summing s1 and s2, pass
// 3 scales by invN_j and writes the transposed split profiles.
template <int W>
__global__ void __launch_bounds__(512) col_profiles_tma_kernel(const __grid_constant__ CUtensorMap mL, float* logphi,
                                                               ProfileOut po, int n, int T, int ldn, int nbox,
                                                               DevStatus* stt) {
  chain_wait();
  constexpr int PH = 512 / W;   // row phases
  extern __shared__ uint8_t smem_raw[];
  const uint32_t r0 = tc::smem_u32(smem_raw);
  float* strip = (float*)(smem_raw + (((r0 + 127u) & ~127u) - r0));   // [nbox * 256][W], 128-byte aligned
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  __shared__ float red[3][PH][W];
  __shared__ float cstat[2][W];
  __shared__ float tile[64][W + 1];
  __shared__ long long orow[W];   // element offset of each column's output row (anchor rows: -1 - offset)
  const int b = blockIdx.y, j0 = blockIdx.x * W, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = tid % W, ph = tid / W, j = j0 + c;
  if (tid == 0) {
    tc::mbar_init(&bar, 1);
    abort_flag = 0;
    tc::mbar_fence_init();
  }
  __syncthreads();
  if (tid == 0) {
    tc::mbar_arrive_expect_tx(&bar, (uint32_t)(nbox * 256 * W * 4));
    for (int q = 0; q < nbox; ++q) tc::tma_load_3d(strip + q * 256 * W, &mL, j0, q * 256, b, &bar);
  }
  // the output rows of the CTA's keys (a binary search over the anchors)
  // while the strip is in flight
  if (po.Ut_hi != nullptr && tid >= 32 && tid < 32 + W && j0 + tid - 32 < T)
    orow[tid - 32] = profile_row(po.anchors + (long long)b * po.t, po.t, T, b, j0 + tid - 32, ldn, po.kmap);
  const bool ok = tc::mbar_wait(&bar, 0, &abort_flag, stt);
  if (!__syncthreads_and(ok)) {   // timed out: let the copies land (bounded) before leaving
    volatile int never = 0;
    if (tid == 0) tc::mbar_wait(&bar, 0, &never, stt);
    __syncthreads();
    return;
  }
  // pass 1: column maxima (four independent chains per thread)
  float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
  if (j < T) {
    int i = ph;
    for (; i + 3 * PH < n; i += 4 * PH) {
      m0 = fmaxf(m0, strip[i * W + c]);
      m1 = fmaxf(m1, strip[(i + PH) * W + c]);
      m2 = fmaxf(m2, strip[(i + 2 * PH) * W + c]);
      m3 = fmaxf(m3, strip[(i + 3 * PH) * W + c]);
    }
    for (; i < n; i += PH) m0 = fmaxf(m0, strip[i * W + c]);
  }
  red[0][ph][c] = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
  __syncthreads();
  if (tid < W) {
    float M = -INFINITY;
#pragma unroll 8
    for (int q = 0; q < PH; ++q) M = fmaxf(M, red[0][q][tid]);
    cstat[0][tid] = M;
  }
  __syncthreads();
  // pass 2: e_ij = e^{l_ij - M_j} replaces l in the strip; s1 = sum e, s2 = sum e^2
  {
    const float M = cstat[0][c];
    float a1 = 0.f, b1 = 0.f, a2 = 0.f, b2 = 0.f;
    if (j < T && M != -INFINITY) {
      int i = ph;
      for (; i + PH < n; i += 2 * PH) {
        const float e0 = ex2_approx((strip[i * W + c] - M) * kLog2e);
        const float e1 = ex2_approx((strip[(i + PH) * W + c] - M) * kLog2e);
        strip[i * W + c] = e0;
        strip[(i + PH) * W + c] = e1;
        a1 += e0;
        b1 += e1;
        a2 = fmaf(e0, e0, a2);
        b2 = fmaf(e1, e1, b2);
      }
      if (i < n) {
        const float e0 = ex2_approx((strip[i * W + c] - M) * kLog2e);
        strip[i * W + c] = e0;
        a1 += e0;
        a2 = fmaf(e0, e0, a2);
      }
    }
    red[1][ph][c] = a1 + b1;
    red[2][ph][c] = a2 + b2;
  }
  __syncthreads();
  if (tid < W) {
    float S1 = 0.f, S2 = 0.f;
#pragma unroll 8
    for (int q = 0; q < PH; ++q) {
      S1 += red[1][q][tid];
      S2 += red[2][q][tid];
    }
    if (j < T) logphi[(long long)b * T + j] = cstat[0][tid] + logf(S1) - logf((float)n);
    cstat[1][tid] = j < T ? 1.0f / sqrtf(S2) : 0.f;
  }
  __syncthreads();
  if (po.Ut_hi == nullptr) return;
  // pass 3: U_ij = e_ij invN_j, transposed through a padded tile 64 rows at a time
  constexpr int RPT = (64 + PH - 1) / PH;   // tile rows per thread: rows ph + k PH below 64
  const float inv = cstat[1][c];
  float rsq = 0.f;   // of column `warp` (W <= 16: one column per warp)
  for (int i0 = 0; i0 < ldn; i0 += 64) {
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int r = ph + k * PH, i = i0 + r;
      if (r < 64) tile[r][c] = (i < n) ? strip[i * W + c] * inv : 0.f;
    }
    __syncthreads();
    // warp w writes columns w, w + 16, ...: lane l rows i0 + 2l and i0 + 2l + 1 (ldn even)
    for (int cc = warp; cc < W; cc += 16) {
      const int jj = j0 + cc, i = i0 + 2 * lane;
      if (jj < T && i < ldn && orow[cc] != kNoRow) {
        const float x0 = tile[2 * lane][cc], x1 = tile[2 * lane + 1][cc];
        const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        const float2 hf = __bfloat1622float2(h);
        rsq = fmaf(x0 - hf.x, x0 - hf.x, fmaf(x1 - hf.y, x1 - hf.y, rsq));
        const long long ro = orow[cc];
        bf16* dh = ro >= 0 ? po.Ut_hi + ro : po.S_hi + (-1 - ro);
        bf16* dl = ro >= 0 ? po.Ut_lo + ro : po.S_lo + (-1 - ro);
        *(__nv_bfloat162*)(dh + i) = h;
        *(__nv_bfloat162*)(dl + i) = __floats2bfloat162_rn(x0 - hf.x, x1 - hf.y);
      }
    }
    __syncthreads();
  }
  static_assert(W <= 16, "one column per warp");
  if (po.rho_k != nullptr && warp < W) {
    rsq = warp_sum(rsq);
    if (lane == 0 && j0 + warp < T && orow[warp] != kNoRow) write_rho(po, b, T, ldn, orow[warp], rsq);
  }
}

template <int W>
static int launch_col_profiles_tma(const Dims& D, const float* L, float* logphi, const ProfileOut& po, int ldn,
                                   int nbox, DevStatus* stt, cudaStream_t st) {
  CUtensorMap m;
  if (!encode_f32_map_3d(&m, L, D.T, D.n, D.H, W, 256)) return -1;
  const int smem = nbox * 256 * W * 4 + 128;
  if (set_dyn_smem((const void*)col_profiles_tma_kernel<W>, smem) !=
      cudaSuccess)
    return -1;
  launch_chained(col_profiles_tma_kernel<W>, dim3(cdiv(D.T, W), D.H), 512, smem, st, m, logphi, po, D.n, D.T, ldn, nbox, stt);
  return 1;
}

static int col_profiles(const Dims& D, const float* L, float* logphi, const ProfileOut& po, DevStatus* stt,
                        cudaStream_t st) {
  const int ldn = (D.n + 7) / 8 * 8;
  // staged strips of at most 64 KB (three CTAs per SM) when l is TMA-tileable
  const int nbox = cdiv(D.n, 256);
  if ((D.T & 3) == 0 && ((uintptr_t)L & 15u) == 0 && nbox <= 16) {
    if (nbox <= 4) return launch_col_profiles_tma<16>(D, L, logphi, po, ldn, nbox, stt, st);
    if (nbox <= 8) return launch_col_profiles_tma<8>(D, L, logphi, po, ldn, nbox, stt, st);
    return launch_col_profiles_tma<4>(D, L, logphi, po, ldn, nbox, stt, st);
  }
  // each CTA re-reads its n x 32 strip from L2: with n > 1024 a shared-memory
  // reservation keeps at most two CTAs per SM so the live strips fit in L2
  const int smem = D.n > 1024 ? 80 * 1024 : 0;
  if (smem > 0 && set_dyn_smem((const void*)col_profiles_kernel, smem) !=
                      cudaSuccess)
    return -1;
  launch_chained(col_profiles_kernel, dim3(cdiv(D.T, 32), D.H), 512, smem, st, L, logphi, po, D.n, D.T, logit_ld(D.T), ldn);
  return 1;
}

int launch_col_profiles(const Dims& D, const float* L, float* logphi, DevStatus* stt, cudaStream_t st) {
  return col_profiles(D, L, logphi, ProfileOut{nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, D.t, nullptr, nullptr, 0}, stt, st);
}

// kappa of the non-anchor keys from the argmax of their compacted rows (rows c <
// Tm of head b; kmap gives the key), then the anchors' own, kappa(s_r) = r
__global__ void decode_assign_kernel(const unsigned long long* best, const int* kmap, const int* anchors, int* kappa,
                                     int T, int Tm, int t, long long keys, long long total) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    if (k < keys) {
      const long long b = k / Tm, o = b * T + (k - b * Tm);
      const unsigned long long v = best[o];
      const int j = kmap[o];
      if ((unsigned)j < (unsigned)T) kappa[b * T + j] = v ? (int)(0xffffffffu - (unsigned int)(v & 0xffffffffull)) : 0;
    } else {
      const long long a = k - keys, b = a / t;
      kappa[b * T + anchors[a]] = (int)(a - b * t);
    }
  }
}

// ---------------------------------------------------------------------------
// Filtered assignment, for many anchors.  The argmax needs the split products
// (three MMAs) only where two anchors are close: a first pass scores every
// (key, anchor) pair by one product of the leading parts, h_j . h_r, which
// misses the split product by at most
//     |rho_j| + |rho_r| + B0,   rho = u - h (Cauchy-Schwarz, ||u|| = ||h|| = 1),
// B0 covering what the split product itself leaves out and the fp32 sums of
// both.  Per key and 128 anchors its epilogue keeps the largest upper and lower
// bound; a tile of anchors whose upper bound reaches the key's largest lower
// bound may hold the argmax.  The second pass computes the split products of
// those (key, tile) pairs alone, with the MMA sequence of the full GEMM, so the
// scores it compares, and the result, have the same bits.
//   tc_gemm (kPlain, TcEpiFilter), share_kernel  the bounds of 128 keys a head, and
//                      whether few enough tiles are candidates for the rest to pay
//   tc_gemm (kPlain, TcEpiFilter)  bounds per (key, tile)
//   candidates_kernel  per (head, key chunk, tile): the list of its keys
//   items_kernel       lists -> work items of 256 keys
//   rescore_kernel     gathered keys x 128 anchors, argmax into `best`
//   tc_gemm (kSplit, TcEpiArgmax8)  the full product, where the share said so
// Keys go in chunks whose profiles stay in L2 while all anchor tiles pass them
// (a key is a candidate in 16 of 103 tiles on average at 128K).
// 128K layer (t = 13107, n = 2048, 8 heads): 26.6 + 0.5 + 22.6 ms (filter, lists,
// second pass); 75.1 ms for the full GEMM.
constexpr int kRsKeys = 256;   // keys per work item of the second pass
struct FilterDims {
  int Nt, Tp, CR, nch;   // anchor tiles, pitch of the bounds, keys per chunk, chunks
};
static FilterDims filter_dims(const Dims& D) {
  const int ldn = (D.n + 7) / 8 * 8, Tm = D.T - D.t;
  FilterDims f;
  f.Nt = 2 * cdiv(D.t, 256);   // the first pass takes anchors 256 at a time
  f.Tp = (Tm + 31) / 32 * 32;
  const long long rows = (48LL << 20) / (4LL * ldn) / 256 * 256;   // 48 MB of split profiles
  f.CR = (int)std::max<long long>(256, std::min<long long>(8192, rows));
  f.nch = cdiv(std::max(Tm, 1), f.CR);
  return f;
}
// byte offsets in the scratch (the index features' second half, free by then)
struct FilterLayout {
  size_t list, cnt, off, items, gate, rho_k, rho_s, total;
};
static FilterLayout filter_layout(const Dims& D, const FilterDims& f) {
  FilterLayout L;
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t r = o; o += (bytes + 255) / 256 * 256; return r; };
  const size_t E = (size_t)D.H * f.nch * f.Nt;
  L.list = take(E * f.CR * 4);
  L.cnt = take(E * 4);
  L.off = take((E + 1) * 4);
  L.items = take(E * (f.CR / kRsKeys) * 4);
  L.gate = take(4);
  L.rho_k = take((size_t)D.H * D.T * 4);
  L.rho_s = take((size_t)D.H * f.Nt * 128 * 4);
  L.total = o;
  return L;
}
// Where the filter is tried: from 24 tiles of 128 anchors, 512 reference rows
// and n t = 2.2 M up, when its bounds and lists fit the two halves of the index
// features' buffer.  Its passes over the bounds and lists do not shrink with n:
// time of the stage with the filter over without, 8 heads, random anchors, at
// n = 256, 512, 1024, 2048: t = 3000 1.25, 1.07, 0.98, 0.92 (768: 0.97); t = 6553
// 1.19, 0.96, 0.86, 0.76; t = 13107 1.12, 0.95, 0.76, 0.73.
bool assign_filtered(const Dims& D) {
  const FilterDims f = filter_dims(D);
  const size_t half = (size_t)D.H * D.T * D.HD * 2;
  return D.t > 23 * 128 && D.n >= 512 && (long long)D.n * D.t >= 2200000 && D.T - D.t >= 4096 && f.CR % kRsKeys == 0 &&
         (size_t)D.H * f.Nt * f.Tp * 8 <= half && filter_layout(D, f).total <= half;
}
// The time over the full GEMM's grows by 1.2 to 1.4 times the share of (key,
// tile) pairs that stay candidates, which is the data's: 0.2 to 0.4 for random
// anchors, 1 for keys that are all alike (1.6 to 1.9 times the full GEMM's time).
// The two take the same time at a share of about 0.35, 0.35 to 0.43 and 0.45 to
// 0.55 for n = 512, 1024, 2048, so the rest of the filter runs where a sample of
// kSampleKeys keys a head stays below the line here, else the full GEMM.  The stage
// then takes 0.71 to 0.99 of the full GEMM's time where the filter's passes run, up
// to 1.03 at a share near the line, and at most 1.02 where the sample turns it away.
constexpr int kSampleKeys = 128;
static float filter_share(int n) { return 0.5f - 80.f / n; }

// Bounds of a row over its warp's 128 anchors (eight warps, 256-wide tiles).
// rho_s is NaN past the last anchor: fmaxf skips those columns.
struct TcEpiFilter {
  static constexpr int kEpiWarps = 8;
  const float* rho_s;   // [H][Nt * 128]
  float2* bounds;       // [H][Nt][Tp] (upper, lower)
  int Nt, Tp;
  const int* gate;      // nullable: a zero word there closes the launch
  __device__ __forceinline__ bool closed() const { return gate != nullptr && __ldcg(gate) == 0; }
  struct State {
    float ub, lb;
    const float4* r;
  };
  __device__ __forceinline__ void init(State& s, int b, int, int n0, int, int) const {
    s.ub = s.lb = -INFINITY;
    s.r = (const float4*)(rho_s + (long long)b * Nt * 128 + n0);
  }
  __device__ __forceinline__ void consume(State& s, int, int j, float (&v)[32]) const {
    float u[4] = {s.ub, -INFINITY, -INFINITY, -INFINITY}, l[4] = {s.lb, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 r = s.r[j * 8 + q];
      u[0] = fmaxf(u[0], v[4 * q] + r.x);
      l[0] = fmaxf(l[0], v[4 * q] - r.x);
      u[1] = fmaxf(u[1], v[4 * q + 1] + r.y);
      l[1] = fmaxf(l[1], v[4 * q + 1] - r.y);
      u[2] = fmaxf(u[2], v[4 * q + 2] + r.z);
      l[2] = fmaxf(l[2], v[4 * q + 2] - r.z);
      u[3] = fmaxf(u[3], v[4 * q + 3] + r.w);
      l[3] = fmaxf(l[3], v[4 * q + 3] - r.w);
    }
    s.ub = fmaxf(fmaxf(u[0], u[1]), fmaxf(u[2], u[3]));
    s.lb = fmaxf(fmaxf(l[0], l[1]), fmaxf(l[2], l[3]));
  }
  __device__ __forceinline__ void finish(State& s, int b, int row, int n0, int M, int) const {
    if (row < M) bounds[((long long)b * Nt + n0 / 128) * Tp + row] = make_float2(s.ub, s.lb);
  }
};

// What a candidate's upper bound has to reach: upper + (rho_j + B0) >= lower -
// (rho_j + B0) for the largest lower bound lb of a key's tiles.
__device__ __forceinline__ float candidate_line(float lb, float rho, float B0) { return lb - 2.f * (rho + B0); }

// gate = 1 where at most a share `most` of the (key, tile) pairs of the sample are
// candidates: key k of a head is its compacted row k * step, its bounds at row k.
__global__ void __launch_bounds__(1024) share_kernel(const float2* bounds, const float* rho_k, float B0, int T, int H,
                                                     int step, int tiles, FilterDims f, float most, int* gate) {
  chain_wait();
  __shared__ int part[32];
  int count = 0;
  for (int k = threadIdx.x; k < H * kSampleKeys; k += 1024) {
    const int b = k / kSampleKeys, row = k % kSampleKeys;
    const float2* bd = bounds + (long long)b * f.Nt * f.Tp + row;
    float lb = -INFINITY;
#pragma unroll 8
    for (int i = 0; i < tiles; ++i) lb = fmaxf(lb, bd[(long long)i * f.Tp].y);
    const float thr = candidate_line(lb, rho_k[(long long)b * T + row * step], B0);
    if (!(lb > -INFINITY)) continue;
#pragma unroll 8
    for (int i = 0; i < tiles; ++i) count += bd[(long long)i * f.Tp].x >= thr;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = count;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < 32; ++w) sum += part[w];
    *gate = sum <= (double)most * H * kSampleKeys * tiles ? 1 : 0;
  }
}

// One thread per key: the tiles that may hold its argmax, appended to their
// lists (one atomic per warp and tile; the order within a list does not matter).
__global__ void __launch_bounds__(256) candidates_kernel(const float2* bounds, const float* rho_k, float B0, int T, int Tm,
                                                         FilterDims f, const int* gate, int* list, int* cnt) {
  chain_wait();
  if (__ldcg(gate) == 0) return;   // (the lists stay empty)
  const int b = blockIdx.y, row = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31;
  const int ch = blockIdx.x * 256 / f.CR;
  const float2* bd = bounds + (long long)b * f.Nt * f.Tp + row;
  const bool in = row < Tm;
  float lb = -INFINITY;
#pragma unroll 8
  for (int k = 0; k < f.Nt; ++k)
    if (in) lb = fmaxf(lb, bd[(long long)k * f.Tp].y);
  // (no finite bound, a NaN profile: no candidate)
  const float thr = in ? candidate_line(lb, rho_k[(long long)b * T + row], B0) : 0.f;
  const bool any = in && lb > -INFINITY;
  const long long e0 = ((long long)b * f.nch + ch) * f.Nt;
#pragma unroll 4
  for (int k = 0; k < f.Nt; ++k) {
    const bool c = any && bd[(long long)k * f.Tp].x >= thr;
    const unsigned m = __ballot_sync(0xffffffffu, c);
    if (m == 0) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(cnt + e0 + k, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (c) list[(e0 + k) * f.CR + base + __popc(m & ((1u << lane) - 1))] = row;
  }
}

// off = exclusive sums of the lists' kRsKeys-key blocks; items[i] = list * (CR / kRsKeys) + block.
__global__ void __launch_bounds__(1024) items_kernel(const int* cnt, int E, int per, int* off, int* items) {
  chain_wait();
  __shared__ int part[1024];
  const int tid = threadIdx.x, step = (E + 1023) / 1024, e0 = min(E, tid * step), e1 = min(E, e0 + step);
  int sum = 0;
  for (int e = e0; e < e1; ++e) sum += (cnt[e] + kRsKeys - 1) / kRsKeys;
  part[tid] = sum;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int v = tid >= o ? part[tid - o] : 0;
    __syncthreads();
    part[tid] += v;
    __syncthreads();
  }
  int at = part[tid] - sum;
  for (int e = e0; e < e1; ++e) {
    off[e] = at;
    const int nb = (cnt[e] + kRsKeys - 1) / kRsKeys;
    for (int k = 0; k < nb; ++k) items[at + k] = e * per + k;
    at += nb;
  }
  if (tid == 1023) off[E] = part[1023];
}

// 256 gathered keys x 128 anchors per work item (two M = 128 halves on the same
// anchor slab; the second is left out when its list has no key for it), split
// products over the whole K, row argmax (lowest index on ties) merged into
// `best`.  Persistent, one CTA per SM: warp 0 streams the anchor slabs by TMA,
// warps 6-9 gather the keys' (16-byte cp.async into the same swizzled layout; a
// thread serves one 16-byte chunk of eight rows), warp 1 issues the MMAs, warps
// 2-5 drain the accumulators.  What bounds it is the latency of the gathered
// rows against the 192 KB a CTA can have in flight, so an anchor slab serves as
// many keys as TMEM has accumulators for, in short slabs (32 of K, four stages, a
// slab handed over kRsLag later: 22.6 ms of the 128K layer; 1 later 23.8, 3
// later, when the gather waits for the MMAs, 37), and every role looks its next
// item up while it works on the current one.  With 128 keys an item (six stages)
// 26.6 ms.  86 GB of DRAM reads at 128K: the key chunks of 48 MB are read again
// by part, but chunks of 16 to 160 MB stay within 7 % of this time.
constexpr int kRsStages = 4, kRsLag = 2, kRsK = 32;
constexpr int kRsTile = 128 * kRsK * 2;          // 128 rows of one part
constexpr int kRsA = 2 * kRsTile;                // 256 keys of one part
constexpr int kRsLo = kRsA + kRsTile, kRsStage = 2 * kRsLo;   // [keys hi][anchors hi][keys lo][anchors lo]
constexpr int kRsThreads = 320;
struct RsItem {
  int e, b, n0, k0, nkeys;   // list, head, first anchor, first key of the list, keys
};
__global__ void __launch_bounds__(kRsThreads, 1)
    rescore_kernel(const __grid_constant__ CUtensorMap mB, const __grid_constant__ CUtensorMap mB2, const bf16* Ut_hi,
                   const bf16* Ut_lo, const int* list, const int* cnt, const int* off, const int* items, FilterDims f,
                   int H, int T, int t, int ldn, unsigned long long* best, DevStatus* stt) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[kRsStages], empty[kRsStages], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t raw = tc::smem_u32(smem_raw);
  uint8_t* base = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = 2 * ((ldn + 63) / 64), per = f.CR / kRsKeys, E = H * f.nch * f.Nt;   // whole 64-wide slabs, as the full GEMM
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRsStages; ++s) {
      tc::mbar_init(&full[s], 1 + 4);
      tc::mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&accf[i], 1);
      tc::mbar_init(&acce[i], 4);
    }
    tc::mbar_init(&drain, 1);
    abort_flag = 0;
    tc::mbar_fence_init();
  }
  chain_wait();
  if (warp == 1) tc::tmem_alloc(&tmem_slot, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  volatile int* abortp = &abort_flag;
  const int nitems = off[E];
  auto item = [&](int i) {
    RsItem x{};
    if (i < nitems) {
      const int v = items[i];
      x.e = v / per;
      x.k0 = (v - x.e * per) * kRsKeys;
      x.b = x.e / (f.nch * f.Nt);
      x.n0 = (x.e % f.Nt) * 128;
      x.nkeys = min(kRsKeys, cnt[x.e] - x.k0);
    }
    return x;
  };

  if (warp == 0) {
    if (lane == 0) {
      tc::tma_prefetch(&mB);
      tc::tma_prefetch(&mB2);
      int g = 0;
      bool ok = true;
      RsItem nx = item(blockIdx.x);
      for (int i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
        const RsItem x = nx;
        nx = item(i + gridDim.x);
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % kRsStages;
          if (g >= kRsStages && !tc::mbar_wait(&empty[s], ((g / kRsStages) - 1) & 1, abortp, stt)) {
            ok = false;
            break;
          }
          uint8_t* st = base + s * kRsStage;
          tc::mbar_arrive_expect_tx(&full[s], 2 * kRsTile);
          tc::tma_load_3d(st + kRsA, &mB, kb * kRsK, x.n0, x.b, &full[s]);
          tc::tma_load_3d(st + kRsLo + kRsA, &mB2, kb * kRsK, x.n0, x.b, &full[s]);
        }
      }
      // every issued copy lands before the CTA may exit: the last slabs' barriers
      // complete once the key gatherers have arrived too (they issue the same slabs)
      volatile int never = 0;
      for (int k = g > kRsStages ? g - kRsStages : 0; k < g; ++k)
        tc::mbar_wait(&full[k % kRsStages], (k / kRsStages) & 1, &never, stt);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int g = 0, c = 0;
      RsItem nx = item(blockIdx.x);
      for (int i = blockIdx.x; i < nitems && ok; i += gridDim.x, ++c) {
        const RsItem x = nx;
        nx = item(i + gridDim.x);
        const uint32_t idesc = tc::idesc_bf16_f32(min(128, (t - x.n0 + 15) & ~15));
        const int buf = c & 1;
        if (c >= 2 && !tc::mbar_wait(&acce[buf], ((c >> 1) - 1) & 1, abortp, stt)) break;
        tc::fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(buf * 256);
        const int halves = x.nkeys > 128 ? 2 : 1;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % kRsStages;
          if (!tc::mbar_wait(&full[s], (g / kRsStages) & 1, abortp, stt)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t bb = tc::smem_u32(base + s * kRsStage) + kRsA;
          for (int h = 0; h < halves; ++h) {
            const uint32_t a = bb - kRsA + h * kRsTile, dh = d + h * 128;
#pragma unroll
            for (int ks = 0; ks < kRsK / 16; ++ks) {   // the sequence of tc_gemm's kSplit
              const uint64_t ad = tc::sdesc_k64(a + ks * 32), bd = tc::sdesc_k64(bb + ks * 32);
              tc::mma_f16(dh, ad, bd, idesc, (kb > 0 || ks > 0) ? 1u : 0u);
              tc::mma_f16(dh, ad, tc::sdesc_k64(bb + kRsLo + ks * 32), idesc, 1u);
              tc::mma_f16(dh, tc::sdesc_k64(a + kRsLo + ks * 32), bd, idesc, 1u);
            }
          }
          tc::mma_commit(&empty[s]);
        }
        if (ok) tc::mma_commit(&accf[buf]);
      }
      tc::mma_commit(&drain);
      volatile int never = 0;
      tc::mbar_wait(&drain, 0, &never, stt);
    }
  } else if (warp < 6) {
    const int q = warp & 3;
    bool ok = true;
    int c = 0;
    for (int i = blockIdx.x; i < nitems; i += gridDim.x, ++c) {
      const RsItem x = item(i);   // (in the shadow of the item's MMAs)
      const int r = q * 32 + lane, n0 = x.n0, b = x.b;
      const int* lk = list + (long long)x.e * f.CR + x.k0;
      const int key[2] = {r < x.nkeys ? lk[r] : -1, r + 128 < x.nkeys ? lk[r + 128] : -1};
      ok = tc::mbar_wait(&accf[c & 1], (c >> 1) & 1, abortp, stt);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc::fence_after_sync();
      float bv[2] = {-INFINITY, -INFINITY};
      int bi[2] = {-1, -1};
      const int ncols = t - n0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h * 128 >= x.nkeys) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float v[32];
          tc::tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((c & 1) * 256 + h * 128 + j * 32), v);
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (j * 32 + k < ncols && v[k] > bv[h]) {
              bv[h] = v[k];
              bi[h] = n0 + j * 32 + k;
            }
        }
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acce[c & 1]);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (key[h] >= 0 && bi[h] >= 0)
          atomicMax(best + (long long)b * T + key[h], ((unsigned long long)f32_ordered(bv[h]) << 32) |
                                                          (unsigned long long)(0xffffffffu - (unsigned int)bi[h]));
    }
  } else {
    // gather: 16-byte chunk `ch` of rows rr, rr + 32, .. of the key tiles; a
    // slab is handed over kRsLag slabs later, when its copies have landed
    const int p = threadIdx.x - 192, ch = p & 3, rr = p >> 2;
    const long long lo = Ut_lo - Ut_hi;
    // 64-byte swizzle: chunk ch of row r at ch ^ (r / 2 % 4); rows rr + 32 u keep rr's
    const uint32_t dst = (uint32_t)(rr * 64 + ((ch ^ ((rr >> 1) & 3)) << 4));
    int g = 0;
    bool ok = true;
    auto hand_over = [&](int q) {   // slab q's copies are complete
      tc::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&full[q % kRsStages]);
    };
    // rows past the list's end repeat its first (their results are dropped)
    auto keys_of = [&](const RsItem& x, int (&key)[8]) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = rr + 32 * u;
        key[u] = x.nkeys > 0 ? list[(long long)x.e * f.CR + x.k0 + (r < x.nkeys ? r : 0)] : 0;
      }
    };
    RsItem x = item(blockIdx.x);
    int key[8];
    keys_of(x, key);
    for (int i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
      const bf16* src[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) src[u] = Ut_hi + ((long long)x.b * T + key[u]) * ldn + ch * 8;
      RsItem nx = item(i + gridDim.x);
      const bool both = x.nkeys > 128;
      for (int kb = 0; kb < nk; ++kb, ++g) {
        if (kb == nk / 2) keys_of(nx, key);
        const int s = g % kRsStages;
        if (g >= kRsStages) {
          ok = tc::mbar_wait(&empty[s], ((g / kRsStages) - 1) & 1, abortp, stt);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        const uint32_t st = tc::smem_u32(base + s * kRsStage);
        const int n16 = kb * kRsK + ch * 8 < ldn ? 16 : 0;   // past the row's end: zeros
        auto copy = [&](int u) {
          const bf16* y = src[u] + (n16 ? kb * kRsK : 0);
          const uint32_t to = st + dst + u * 2048;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(y), "r"(n16) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + kRsLo), "l"(y + lo), "r"(n16)
                       : "memory");
        };
#pragma unroll
        for (int u = 0; u < 4; ++u) copy(u);
        if (both) {
#pragma unroll
          for (int u = 4; u < 8; ++u) copy(u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (g >= kRsLag) {
          asm volatile("cp.async.wait_group %0;" ::"n"(kRsLag) : "memory");
          hand_over(g - kRsLag);
        }
      }
      x = nx;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    for (int q = g > kRsLag ? g - kRsLag : 0; q < g; ++q) hand_over(q);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 512);
  }
}

int launch_assign_prep(const Dims& D, const float* L, float* logphi, const int* anchors, bf16* Ut_hi, bf16* Ut_lo,
                       bf16* S_hi, bf16* S_lo, int* kmap, char* filter_scratch, DevStatus* stt, cudaStream_t st) {
  ProfileOut po{Ut_hi, Ut_lo, S_hi, S_lo, kmap, anchors, D.t, nullptr, nullptr, 0};
  if (filter_scratch) {
    const FilterDims f = filter_dims(D);
    const FilterLayout L2 = filter_layout(D, f);
    po.rho_k = (float*)(filter_scratch + L2.rho_k);
    po.rho_s = (float*)(filter_scratch + L2.rho_s);
    po.ldr = f.Nt * 128;
    // NaN past the anchors (TcEpiFilter)
    if (cudaMemsetAsync(po.rho_s, 0xff, (size_t)D.H * po.ldr * 4, st) != cudaSuccess) return -1;
  }
  return col_profiles(D, L, logphi, po, stt, st);
}

// The full product: 128 keys x 256 anchors per tile (M = 128, N = 256 MMAs): half
// the key-side operand bytes per flop of a 128-wide tile.  The key map spans all T
// rows of a head (its plane stride); the GEMM takes the first Tm.
static int full_argmax(const Dims& D, const bf16* Ut_hi, const bf16* Ut_lo, const bf16* S_hi, const bf16* S_lo,
                       unsigned long long* best, const int* gate, DevStatus* stt, cudaStream_t st) {
  constexpr int BN = 256;
  const int ldn = (D.n + 7) / 8 * 8, Tm = D.T - D.t;
  CUtensorMap mA, mA2, mB, mB2;
  if (!encode_bf16_map_3d(&mA, Ut_hi, ldn, D.T, D.H, 128) || !encode_bf16_map_3d(&mA2, Ut_lo, ldn, D.T, D.H, 128) ||
      !encode_bf16_map_3d(&mB, S_hi, ldn, D.t, D.H, BN) || !encode_bf16_map_3d(&mB2, S_lo, ldn, D.t, D.H, BN))
    return -1;
  TcEpiArgmax8 epi;
  epi.best = best;
  epi.bbs = D.T;
  epi.gate = gate;
  const int kfull = (ldn + 63) / 64 * 64;
  // anchor tiles in groups whose split profiles (BN rows x ldn x 4 bytes per
  // tile) take about 40 MB, so each group stays in L2 while the key profiles
  // stream past it (one pass over them per group instead of one per wave)
  const long long tile_bytes = (long long)BN * ldn * 4;
  const int group = (int)std::max<long long>(1, (40LL << 20) / tile_bytes);
  return launch_tc_gemm<BN, kSplit>(mA, mB, mA2, mB2, epi, D.H, Tm, D.t, ldn, kfull, stt, st, 0, nullptr, group) ==
                 cudaSuccess
             ? 1
             : -1;
}

// The filtered assignment: `best` of every compacted row, by its two passes or,
// where the sample says so, by the full product.
static int filtered_argmax(const Dims& D, const bf16* Ut_hi, const bf16* Ut_lo, const bf16* S_hi, const bf16* S_lo,
                           float2* bounds, char* scratch, unsigned long long* best, DevStatus* stt, cudaStream_t st) {
  const FilterDims f = filter_dims(D);
  const FilterLayout L = filter_layout(D, f);
  const int ldn = (D.n + 7) / 8 * 8, Tm = D.T - D.t, E = D.H * f.nch * f.Nt, step = Tm / kSampleKeys;
  const float* rho_k = (const float*)(scratch + L.rho_k);
  const float* rho_s = (const float*)(scratch + L.rho_s);
  int* list = (int*)(scratch + L.list);
  int* cnt = (int*)(scratch + L.cnt);
  int* off = (int*)(scratch + L.off);
  int* items = (int*)(scratch + L.items);
  int* gate = (int*)(scratch + L.gate);
  CUtensorMap mS, mA, mB, mC, mC2;
  // mS: every step-th compacted row of a head
  if (!encode_bf16_map_3d(&mS, Ut_hi, ldn, kSampleKeys, D.H, 128, (uint64_t)step * ldn, (uint64_t)D.T * ldn) ||
      !encode_bf16_map_3d(&mA, Ut_hi, ldn, D.T, D.H, 128) || !encode_bf16_map_3d(&mB, S_hi, ldn, D.t, D.H, 256) ||
      !encode_bf16_map_3d_sw64(&mC, S_hi, ldn, D.t, D.H, ldn, 128) ||
      !encode_bf16_map_3d_sw64(&mC2, S_lo, ldn, D.t, D.H, ldn, 128))
    return -1;
  if (cudaMemsetAsync(cnt, 0, (size_t)E * 4, st) != cudaSuccess) return -1;
  const int kfull = (ldn + 63) / 64 * 64;
  const int group = (int)std::max<long long>(1, (40LL << 20) / (512LL * ldn));   // 40 MB of anchor rows stay in L2
  // B0: the split product drops lo lo and the lo parts' own rounding (2^-15 in
  // all); an fp32 accumulation step errs by at most 2^-20 of a sum below 1, and
  // the two passes take 4 n / 16 of them
  const float B0 = 0x1p-15f + (float)D.n * 0x1p-22f;
  TcEpiFilter epi{rho_s, bounds, f.Nt, f.Tp, nullptr};
  if (launch_tc_gemm<256, kPlain>(mS, mB, mS, mB, epi, D.H, kSampleKeys, D.t, ldn, kfull, stt, st) != cudaSuccess)
    return -1;
  launch_chained(share_kernel, 1, 1024, 0, st, bounds, rho_k, B0, D.T, D.H, step, cdiv(D.t, 128), f, filter_share(D.n),
                 gate);
  epi.gate = gate;
  if (launch_tc_gemm<256, kPlain>(mA, mB, mA, mB, epi, D.H, Tm, D.t, ldn, kfull, stt, st, 0, nullptr, group) !=
      cudaSuccess)
    return -1;
  launch_chained(candidates_kernel, dim3(cdiv(Tm, 256), D.H), 256, 0, st, bounds, rho_k, B0, D.T, Tm, f, gate, list, cnt);
  launch_chained(items_kernel, 1, 1024, 0, st, cnt, E, f.CR / kRsKeys, off, items);
  const int smem = kRsStages * kRsStage + 1024;
  if (set_dyn_smem((const void*)rescore_kernel, smem) != cudaSuccess) return -1;
  if (launch_chained(rescore_kernel, tc_gemm_sm_count(), kRsThreads, smem, st, mC, mC2, Ut_hi, Ut_lo, list, cnt, off,
                     items, f, D.H, D.T, D.t, ldn, best, stt) != cudaSuccess)
    return -1;
  return full_argmax(D, Ut_hi, Ut_lo, S_hi, S_lo, best, gate, stt, st) < 0 ? -1 : 7;
}

int launch_assign_gemm(const Dims& D, const int* anchors, const bf16* Ut_hi, const bf16* Ut_lo, const bf16* S_hi,
                       const bf16* S_lo, const int* kmap, unsigned long long* best, int* kappa, float2* filter_bounds,
                       char* filter_scratch, DevStatus* stt, cudaStream_t st) {
  const int Tm = D.T - D.t;   // the non-anchor keys, compacted (none when t = T)
  int nl = 1;
  // every key gets an assignment in [0, t) even when invalid caller anchors
  // (flagged upstream) leave some compacted rows without a key
  cudaMemsetAsync(kappa, 0, sizeof(int) * (size_t)D.H * D.T, st);
  if (Tm > 0) {
    cudaMemsetAsync(best, 0, sizeof(unsigned long long) * (size_t)D.H * D.T, st);
    const int r = filter_scratch
                      ? filtered_argmax(D, Ut_hi, Ut_lo, S_hi, S_lo, filter_bounds, filter_scratch, best, stt, st)
                      : full_argmax(D, Ut_hi, Ut_lo, S_hi, S_lo, best, nullptr, stt, st);
    if (r < 0) return -1;
    nl += r;
  }
  const long long keys = (long long)D.H * Tm, total = keys + (long long)D.H * D.t;
  launch_chained(decode_assign_kernel, stride_grid(total, 256, 8), 256, 0, st, best, kmap, anchors, kappa, D.T,
                 std::max(Tm, 1), D.t, keys, total);
  return nl;
}

}  // namespace arckv
