// Closed-form attention-mass and compact-value fits (App. A.9).
//
// beta:  Phi_C = exp(scale Q C_k^T - z), z_i = max_j scale q_i.k_j;
//        (Phi_C^T Phi_C + lam_w I) w = Phi_C^T (Phi_K 1);  w* = max(w, 0);
//        beta = clip(log max(w*, eps_w), b_min, b_max)          (Eq. mass_fit)
// C_v:   P^ = softmax(scale Q C_k^T + 1 beta^T);
//        (P^T P^ + lam_v I) C_v = P^T Y, Y = softmax(scale Q K^T) V   (Eq. value_lstsq)
// with lam = ridge * trace(Gram) / t.  Both systems are solved by a blocked
// right-looking Cholesky factorisation (64 x 64 blocks; each diagonal block
// is factored and inverted in shared memory) with the forward substitution
// fused into the trailing updates, then blocked back substitution, all in one
// cluster launch per system (chol.cu).
#include <cooperative_groups.h>
#include <map>
#include <mutex>
#include <type_traits>

#include "chol.cuh"
#include "kernels.h"
#include "tc_gemm.cuh"

namespace arckv {

__global__ void phi_kernel(const float* LC, const float* z, float* Phi, int n, int t, long long count) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
       k += (long long)gridDim.x * blockDim.x) {
    const long long row = k / t;  // = b * n + i
    Phi[k] = expf(LC[k] - z[row]);
  }
}

// rhs[b][r] = sum_i Phi[b][i][r] m[b][i]   (Phi_C^T Phi_K 1).  A CTA owns 32
// columns; warp w sums the rows i = w, w+8, ... (four partial sums) and the
// eight warp sums are added in warp order.
__global__ void __launch_bounds__(1024) mass_rhs_kernel(const float* Phi, const float* m, float* rhs, int n, int t) {
  chain_wait();
  // 32 columns per CTA, the rows split over 32 warps (four loads in flight each)
  const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane;
  __shared__ float red[32][33];
  const float* P = Phi + (long long)b * n * t + r;
  const float* mb = m + (long long)b * n;
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
  if (r < t) {
    int i = warp;
    for (; i + 96 < n; i += 128) {
      a0 = fmaf(P[(long long)i * t], mb[i], a0);
      a1 = fmaf(P[(long long)(i + 32) * t], mb[i + 32], a1);
      a2 = fmaf(P[(long long)(i + 64) * t], mb[i + 64], a2);
      a3 = fmaf(P[(long long)(i + 96) * t], mb[i + 96], a3);
    }
    for (; i < n; i += 32) a0 = fmaf(P[(long long)i * t], mb[i], a0);
  }
  red[warp][lane] = (a0 + a1) + (a2 + a3);
  __syncthreads();
  if (warp == 0 && r < t) {
    float a = 0.f;
    for (int w = 0; w < 32; ++w) a += red[w][lane];
    rhs[(long long)b * t + r] = a;
  }
}

// ---------------------------------------------------------------------------
// Cluster Cholesky solver: (Gram + lam I) X = B for every head in ONE launch.
// One cluster of kCL CTAs per head; the matrix, its factor and the right-hand
// sides live in global memory (L2-resident at these sizes) and are read with
// ld.global.cg so that no CTA sees a stale L1 line of another CTA's writes.
// Phases of each 64-wide block step k are separated by hardware cluster
// barriers (release / acquire at cluster scope):
//   trsm    L_ik = A_ik Linv_kk^T for block rows i > k (round robin);
//   update  A_ij -= L_ik L_jk^T (k < j <= i) and B_i -= L_ik (Linv_kk B_k);
//           the CTA that owns block k+1 updates the diagonal block first and
//           factors it at once, overlapping the serial factorisation with the
//           other CTAs' updates;
// then block back substitution X_k = Linv_kk^T (Linv_kk B_k + Z_k),
// Z_i -= L_ki^T X_k (i < k).  lam = ridge * trace(Gram) / tdiv is added to the
// diagonal as each diagonal block is factored (tdiv = t, or the primal size
// when the dual system is solved).
// SIMT tile products throughout: the fp64 dual systems beyond kSlicedMaxK (the
// fp32 systems run in chol.cu).
template <typename R, int kCL>
__global__ void __cluster_dims__(kCL, 1, 1) __launch_bounds__(kCT, 1)
    chol_cluster_kernel(R* A, R* Linv, R* B, R* Z, R* X, int t, int nrhs, int ldb, long long bbs, R ridge, R tdiv,
                        DevStatus* stt) {
  chain_wait();
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smraw[];
  R* sm = (R*)smraw;
  Tile<R> S1 = (Tile<R>)sm;
  Tile<R> S2 = (Tile<R>)(sm + kTileF<R>);
  Tile<R> S3 = (Tile<R>)(sm + 2 * kTileF<R>);
  Tile<R> S4 = (Tile<R>)(sm + 3 * kTileF<R>);
  __shared__ R red[kCT / 32];
  __shared__ int bad, grab;
  __shared__ int ctr[2];   // rank 0's pair deals the tiles of alternate dynamic phases
  const int head = blockIdx.x / kCL;
  const int rank = (int)cluster_rank();
  const int tid = threadIdx.x;
  const int nblk = (t + NB - 1) / NB, nct = (nrhs + NB - 1) / NB;
  R* Ab = A + (long long)head * t * t;
  R* Lb = Linv + (long long)head * nblk * NB * NB;
  R* Bb = B + (long long)head * bbs;
  R* Zb = Z + (long long)head * bbs;
  R* Xb = X + (long long)head * bbs;
  const int ry = tile_ry(), cx = tile_cx();
  R acc[kTP][kTQ];
  int* ctr0 = cg::this_cluster().map_shared_rank(ctr, 0);
  int ep = 0;   // dynamic phase number; phase ep draws from ctr0[ep & 1]
  // next tile of the current dynamic phase (block-uniform)
  auto next_tile = [&]() -> int {
    __syncthreads();
    if (tid == 0) grab = atomicAdd(ctr0 + (ep & 1), 1);
    __syncthreads();
    return grab;
  };
  // lam = ridge * trace / t (every CTA forms it; the trace precedes all writes)
  R tr = R(0);
  for (int r = tid; r < t; r += kCT) tr += __ldcg(Ab + (long long)r * t + r);
  tr = warp_sum_r(tr);
  if ((tid & 31) == 0) red[tid >> 5] = tr;
  if (tid == 0) {
    bad = 0;
    ctr[0] = 0;
    ctr[1] = 0;
  }
  __syncthreads();
  if (tid < 32) {
    R v = tid < kCT / 32 ? red[tid] : R(0);
    v = warp_sum_r(v);
    if (tid == 0) red[0] = v;
  }
  __syncthreads();
  const R trace = red[0];
  const R lam = ridge * trace / tdiv;
  if (rank == 0 && tid == 0 && !isfinite(trace)) set_status(stt, ARCKV_ERR_NONFINITE);
  // zero Z (rows split over the cluster) and factor the first diagonal block
  for (long long e = (long long)rank * kCT + tid; e < (long long)t * ldb; e += (long long)kCL * kCT) Zb[e] = R(0);
  cluster_sync_all();   // everyone has read the unmodified diagonal for the trace; counters are set

  // trailing-update tiles of step k: x < ntri is the syrk tile (ii >= jj) of
  // the m trailing blocks, A_ij -= L_ik L_jk^T; the rest are rhs tiles
  // B_i -= L_ik Y_k with Y_k = Linv_kk B_k formed in the trsm phase
  // where tile x of step k reads its operands and writes its result
  struct UpdDesc {
    const R* Ga;   // L_ik (rows i0.., cols k0..), loaded transposed
    const R* Gb;   // L_jk (transposed) or Y_k (as is)
    R* dst;        // A_ij or B_i at the thread's first row / column
    long long ldb_, ldd;
    int i0, rb, br0, bc0, brm, bcm, pn, qn;
    bool btrans;
  };
  auto describe = [&](int k, int x, int ntri, UpdDesc& u) {
    const int k0 = k * NB;
    u.Ga = Ab;
    if (x < ntri) {
      int ii = (int)((sqrtf(8.f * x + 1.f) - 1.f) * 0.5f);
      while (ii * (ii + 1) / 2 > x) --ii;
      while ((ii + 1) * (ii + 2) / 2 <= x) ++ii;
      const int jj = x - ii * (ii + 1) / 2;
      const int i0 = (k + 1 + ii) * NB, j0 = (k + 1 + jj) * NB;
      u.i0 = i0;
      u.rb = min(NB, t - i0);
      const int cb = min(NB, t - j0);
      u.Gb = Ab; u.ldb_ = t; u.br0 = j0; u.bc0 = k0; u.brm = cb; u.bcm = NB; u.btrans = true;
      u.dst = Ab + (long long)(i0 + ry) * t + j0 + cx; u.ldd = t; u.pn = u.rb - ry; u.qn = cb - cx;
    } else {
      const int y = x - ntri, i = k + 1 + y / nct, c0 = (y % nct) * NB;
      const int i0 = i * NB, nc = min(NB, nrhs - c0);
      u.i0 = i0;
      u.rb = min(NB, t - i0);
      u.Gb = Bb; u.ldb_ = ldb; u.br0 = k0; u.bc0 = c0; u.brm = NB; u.bcm = nc; u.btrans = false;   // block k is full
      u.dst = Bb + (long long)(i0 + ry) * ldb + c0 + cx; u.ldd = ldb; u.pn = u.rb - ry; u.qn = nc - cx;
    }
  };
  // trailing-update tiles x0 and (when x1 < ntot) x1 of step k: all operand
  // loads in one L2 round trip, both products, both read-modify-writes
  auto update_tiles = [&](int k, int x0, int x1, int ntot, int ntri) {
    const int k0 = k * NB;
    const bool two = x1 < ntot;
    UpdDesc u0, u1;
    describe(k, x0, ntri, u0);
    if (two) describe(k, x1, ntri, u1);
    {
      TileRegs<R> fa0, fb0, fa1, fb1;
      tile_fetch(fa0, u0.Ga, t, u0.i0, k0, u0.rb, NB, true);
      tile_fetch(fb0, u0.Gb, u0.ldb_, u0.br0, u0.bc0, u0.brm, u0.bcm, u0.btrans);
      if (two) {
        tile_fetch(fa1, u1.Ga, t, u1.i0, k0, u1.rb, NB, true);
        tile_fetch(fb1, u1.Gb, u1.ldb_, u1.br0, u1.bc0, u1.brm, u1.bcm, u1.btrans);
      }
      tile_put(S1, fa0);
      tile_put(S2, fb0);
      if (two) {
        tile_put(S3, fa1);
        tile_put(S4, fb1);
      }
    }
    __syncthreads();
    mm64(S1, S2, acc);
    if (two) {
      R acc1[kTP][kTQ];
      mm64(S3, S4, acc1);
      rmw_sub(u0.dst, u0.ldd, u0.pn, u0.qn, acc);
      rmw_sub(u1.dst, u1.ldd, u1.pn, u1.qn, acc1);
    } else {
      rmw_sub(u0.dst, u0.ldd, u0.pn, u0.qn, acc);
    }
    __syncthreads();
  };


  // step k = -1 only factors the first diagonal block (one call site keeps the
  // register-resident factorisation inlined once)
  for (int k = -1; k < nblk; ++k) {
    const int m = nblk - k - 1, k0 = k * NB, kb = min(NB, t - k0);
    const R* Lk = Lb + (long long)k * NB * NB;
    // trsm phase: L_ik = A_ik Linv_kk^T (x < m) and Y_k = Linv_kk B_k, written over B_k
    for (int x = rank; k >= 0 && x < m + nct; x += kCL) {
      if (x < m) {
        const int i0 = (k + 1 + x) * NB, rb = min(NB, t - i0);
        ld_tiles(S1, Ab, t, i0, k0, rb, NB, true,                    // S1[l][r] = A_ik[r][l]
                 S2, Lk, (long long)NB, 0, 0, NB, NB, true);         // S2[l][c] = Linv[c][l]
        __syncthreads();
        mm64(S1, S2, acc);
        st_acc(Ab + (long long)(i0 + ry) * t + k0 + cx, t, rb - ry, NB, acc);
      } else {
        const int c0 = (x - m) * NB, nc = min(NB, nrhs - c0);
        ld_tiles(S1, Lk, (long long)NB, 0, 0, NB, NB, true,          // S1[l][r] = Linv[r][l]
                 S2, Bb, ldb, k0, c0, kb, nc, false);
        __syncthreads();
        mm64(S1, S2, acc);
        st_acc(Bb + (long long)(k0 + ry) * ldb + c0 + cx, ldb, kb - ry, nc - cx, acc);
      }
      __syncthreads();
    }
    if (k >= 0) {
      cluster_sync_all();
      if (m == 0) break;
    }
    // update phase: the owner of block k+1 updates and factors the diagonal
    // block first (overlapping the serial factorisation with the other CTAs'
    // updates); every CTA then draws the remaining tiles from the counter
    const int ntri = k >= 0 ? m * (m + 1) / 2 : 0, ntot = k >= 0 ? ntri + m * nct : 0;
    if (rank == 0 && tid == 0) ctr[(ep + 1) & 1] = 0;
    if (rank == (k + 1) % kCL) {
      if (k >= 0) update_tiles(k, 0, ntot, ntot, ntri);
      load_diag(S1, Ab, t, (k + 1) * NB, min(NB, t - (k + 1) * NB), lam);
      factor_diag<R>(Ab, Lb, t, k + 1, S1, S2, S3, &bad);
    }
    for (;;) {   // tiles are drawn two at a time
      const int x = 1 + 2 * next_tile();
      if (x >= ntot) break;
      update_tiles(k, x, x + 1, ntot, ntri);
    }
    ++ep;
    cluster_sync_all();
  }

  // back substitution: X_k = Linv_kk^T (Y_k + Z_k) and Z_i -= L_ki^T X_k (i < k).
  // The owner of block k-1 applies X_k to Z_{k-1} first and forms X_{k-1} at
  // once; the other Z tiles are drawn from the counter.
  auto form_x = [&](int k) {
    const int k0 = k * NB, kb = min(NB, t - k0);
    for (int c0 = 0; c0 < nrhs; c0 += NB) {
      const int nc = min(NB, nrhs - c0);
      ld_tile(S1, Lb + (long long)k * NB * NB, NB, 0, 0, NB, NB, false);   // S1[l][r] = Linv[l][r]
      ld_tile_sum(S2, Bb, Zb, ldb, k0, c0, kb, nc);                        // Y_k + Z_k
      __syncthreads();
      mm64(S1, S2, acc);
      st_acc(Xb + (long long)(k0 + ry) * ldb + c0 + cx, ldb, kb - ry, nc - cx, acc);
      __syncthreads();
    }
  };
  auto z_tile = [&](int k, int i, int c0) {
    const int k0 = k * NB, kb = min(NB, t - k0), i0 = i * NB, nc = min(NB, nrhs - c0);
    ld_tiles(S1, Ab, t, k0, i0, kb, NB, false,     // S1[l][r] = L_ki[l][r]
             S2, Xb, ldb, k0, c0, kb, nc, false);  // X_k
    __syncthreads();
    mm64(S1, S2, acc);
    rmw_sub(Zb + (long long)(i0 + ry) * ldb + c0 + cx, ldb, NB - ry, nc - cx, acc);   // block i < k is full
    __syncthreads();
  };
  if (rank == (nblk - 1) % kCL) form_x(nblk - 1);
  cluster_sync_all();
  for (int k = nblk - 1; k >= 1; --k) {
    if (rank == 0 && tid == 0) ctr[(ep + 1) & 1] = 0;
    if (rank == (k - 1) % kCL) {
      for (int c0 = 0; c0 < nrhs; c0 += NB) z_tile(k, k - 1, c0);
      form_x(k - 1);
    }
    const int ntz = (k - 1) * nct;
    for (;;) {
      const int g = next_tile();
      if (g >= ntz) break;
      z_tile(k, g / nct, (g % nct) * NB);
    }
    ++ep;
    cluster_sync_all();
  }
  if (tid == 0 && bad) set_status(stt, ARCKV_ERR_NOT_SPD);
}

// The fp64 system on SIMT tile products (dual fits beyond kSlicedMaxK).
static int cholesky_solve64(int H, int n, double* A, double* Linv, double* B, double* Z, double* X, int nrhs,
                            long long bbs, double ridge, double tdiv, DevStatus* stt, cudaStream_t st) {
  const int smem = 4 * kTileF<double> * (int)sizeof(double);
  if (set_dyn_smem((const void*)chol_cluster_kernel<double, 8>, smem) != cudaSuccess) return -1;
  launch_chained(chol_cluster_kernel<double, 8>, 8 * H, kCT, smem, st, A, Linv, B, Z, X, n, nrhs, nrhs, bbs, ridge, tdiv, stt);
  return 1;
}

__global__ void beta_kernel(const float* w, float* beta, long long count, float eps_w, float b_min, float b_max) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
       k += (long long)gridDim.x * blockDim.x) {
    const float ws = fmaxf(w[k], 0.f);
    beta[k] = fminf(fmaxf(logf(fmaxf(ws, eps_w)), b_min), b_max);
  }
}

// P[row] = softmax(LC[row] + beta), one warp per row (rows = H * n).
__global__ void softmax_bias_kernel(const float* LC, const float* beta, float* P, int n, int t) {
  chain_wait();
  const int b = blockIdx.y, row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  const float* x = LC + ((long long)b * n + row) * t;
  const float* be = beta + (long long)b * t;
  float* o = P + ((long long)b * n + row) * t;
  float mx = -INFINITY;
  for (int c = lane; c < t; c += 32) mx = fmaxf(mx, x[c] + be[c]);
  mx = warp_max(mx);
  float sm = 0.f;
  for (int c = lane; c < t; c += 32) sm += expf(x[c] + be[c] - mx);
  sm = warp_sum(sm);
  const float inv = 1.0f / sm;
  for (int c = lane; c < t; c += 32) o[c] = expf(x[c] + be[c] - mx) * inv;
}

// dst_hi/lo[b][c][r] = split(src[b][r][c]) for r < rows, zero for rows <= r < ldr:
// the transposed, K-major split-bf16 operand of the Gram GEMMs.
__global__ void __launch_bounds__(256) transpose_split_kernel(const float* src, int rows, int cols, bf16* dst_hi,
                                                              bf16* dst_lo, int ldr) {
  chain_wait();
  const int b = blockIdx.z, c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  __shared__ float tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float* sb = src + (long long)b * rows * cols;
  for (int q = ty; q < 32; q += 8) {
    const int r = r0 + q, c = c0 + tx;
    tile[q][tx] = (r < rows && c < cols) ? sb[(long long)r * cols + c] : 0.f;
  }
  __syncthreads();
  for (int q = ty; q < 32; q += 8) {
    const int c = c0 + q, r = r0 + tx;
    if (c < cols && r < ldr) {
      bf16 hi, lo;
      split_bf16(tile[tx][q], hi, lo);
      const long long o = ((long long)b * cols + c) * ldr + r;
      dst_hi[o] = hi;
      dst_lo[o] = lo;
    }
  }
}

// Transposed bf16 triple of src [rows][cols] (fp32): dst_{h,m,l}[b][c][r]
// (row stride ldr >= rows; the pad r in [rows, ldr) is written as zeros).
__global__ void __launch_bounds__(256) transpose_split3_kernel(const float* src, int rows, int cols, bf16* dh, bf16* dm,
                                                               bf16* dl, int ldr) {
  chain_wait();
  const int b = blockIdx.z, c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  __shared__ float tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float* sb = src + (long long)b * rows * cols;
  for (int q = ty; q < 32; q += 8) {
    const int r = r0 + q, c = c0 + tx;
    tile[q][tx] = (r < rows && c < cols) ? sb[(long long)r * cols + c] : 0.f;
  }
  __syncthreads();
  for (int q = ty; q < 32; q += 8) {
    const int c = c0 + q, r = r0 + tx;
    if (c < cols && r < ldr) {
      const long long o = ((long long)b * cols + c) * ldr + r;
      split3_bf16(tile[tx][q], dh[o], dm[o], dl[o]);
    }
  }
}

// C[b] (t x t, row stride t) = X^T X over the n reference rows, X^T given as a
// transposed bf16 triple [t][ldn]: the kSplit3S tensor-core Gram.
static int gram3_tc(int H, int t, int ldn, const bf16* Xh, const bf16* Xm, const bf16* Xl, float* C, DevStatus* stt,
                    cudaStream_t st) {
  CUtensorMap mA, mA2, mA3;
  if (!encode_bf16_map_3d(&mA, Xh, ldn, t, H, 128) || !encode_bf16_map_3d(&mA2, Xm, ldn, t, H, 128) ||
      !encode_bf16_map_3d(&mA3, Xl, ldn, t, H, 128))
    return -1;
  TcEpiStore epi{C, (long long)t * t, t, 1.f};
  const int kfull = (ldn + 63) / 64 * 64;
  if (launch_tc_gemm<128, kSplit3S>(mA, mA, mA2, mA2, epi, H, t, t, ldn, kfull, stt, st, 0, &mA3) != cudaSuccess)
    return -1;
  return 1;
}

// C[b] (M x N, row stride ldc) = X^T Z over the n reference rows, with X^T and
// Z^T given as transposed split-bf16 operands [M][ldn] and [N][ldn].
static int gram_tc(int H, int M, int N, int ldn, const bf16* Xh, const bf16* Xl, const bf16* Zh, const bf16* Zl,
                   float* C, int ldc, DevStatus* stt, cudaStream_t st) {
  CUtensorMap mA, mA2, mB, mB2;
  if (!encode_bf16_map_3d(&mA, Xh, ldn, M, H, 128) || !encode_bf16_map_3d(&mA2, Xl, ldn, M, H, 128) ||
      !encode_bf16_map_3d(&mB, Zh, ldn, N, H, 128) || !encode_bf16_map_3d(&mB2, Zl, ldn, N, H, 128))
    return -1;
  TcEpiStore epi{C, (long long)M * ldc, ldc, 1.f};
  const int kfull = (ldn + 63) / 64 * 64;
  if (launch_tc_gemm<128, kSplit>(mA, mB, mA2, mB2, epi, H, M, N, ldn, kfull, stt, st) != cudaSuccess) return -1;
  return 1;
}

// C[b] = X X^T in fp64 (X fp32 [rows][K]); 64 x 64 lower tiles, mirrored.
__global__ void __launch_bounds__(256) syrk64_kernel(const float* X, double* C, int rows, int K) {
  chain_wait();
  const int b = blockIdx.z, i0 = blockIdx.y * 64, j0 = blockIdx.x * 64;
  if (j0 > i0) return;
  const float* Xb = X + (long long)b * rows * K;
  double* Cb = C + (long long)b * rows * rows;
  __shared__ double As[16][65], Bs[16][65];
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0.0;
  for (int k0 = 0; k0 < K; k0 += 16) {
    for (int e = threadIdx.x; e < 64 * 16; e += 256) {
      const int r = e >> 4, kk = e & 15, k = k0 + kk;
      As[kk][r] = (i0 + r < rows && k < K) ? (double)Xb[(long long)(i0 + r) * K + k] : 0.0;
      Bs[kk][r] = (j0 + r < rows && k < K) ? (double)Xb[(long long)(j0 + r) * K + k] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      double a[4], c[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) { a[p] = As[kk][ty * 4 + p]; c[p] = Bs[kk][tx * 4 + p]; }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma(a[p], c[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ty * 4 + p, j = j0 + tx * 4 + q;
      if (i < rows && j < rows) {
        Cb[(long long)i * rows + j] = acc[p][q];
        Cb[(long long)j * rows + i] = acc[p][q];
      }
    }
}

__global__ void widen_kernel(const float* x, double* y, long long count) {
  chain_wait();
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < count;
       k += (long long)gridDim.x * blockDim.x)
    y[k] = (double)x[k];
}

// out[b][r][c] = sum_i X[b][i][r] Y[b][i][c] accumulated in fp64 (X fp32 [n][t],
// Y fp64 [n][ncol], out fp32 [t][ncol]); 64 x 32 output tiles.
__global__ void __launch_bounds__(256) xty64_kernel(const float* X, const double* Y, float* out, int n, int t,
                                                    int ncol) {
  chain_wait();
  const int b = blockIdx.z, r0 = blockIdx.x * 64, c0 = blockIdx.y * 32;
  const float* Xb = X + (long long)b * n * t;
  const double* Yb = Y + (long long)b * n * ncol;
  __shared__ double Xs[16][64], Ys[16][33];
  const int tr = threadIdx.x & 63, tc = threadIdx.x >> 6;   // 64 rows x 4 column groups of 8
  double acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0.0;
  for (int i0 = 0; i0 < n; i0 += 16) {
    for (int e = threadIdx.x; e < 16 * 64; e += 256) {
      const int ii = e >> 6, r = e & 63;
      Xs[ii][r] = (i0 + ii < n && r0 + r < t) ? (double)Xb[(long long)(i0 + ii) * t + r0 + r] : 0.0;
    }
    for (int e = threadIdx.x; e < 16 * 32; e += 256) {
      const int ii = e >> 5, c = e & 31;
      Ys[ii][c] = (i0 + ii < n && c0 + c < ncol) ? Yb[(long long)(i0 + ii) * ncol + c0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < 16; ++ii) {
      const double xv = Xs[ii][tr];
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] = fma(xv, Ys[ii][tc * 8 + q], acc[q]);
    }
    __syncthreads();
  }
  const int r = r0 + tr;
  if (r >= t) return;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int c = c0 + tc * 8 + q;
    if (c < ncol) out[((long long)b * t + r) * ncol + c] = (float)acc[q];
  }
}

// ---------------------------------------------------------------------------
// Blocked Cholesky solve of the fp64 dual systems, (A + lam I) X = B with
// lam = ridge * trace(A) / tdiv, A [H][n][n] (lower part read, overwritten
// by L), B [H][n][nrhs] (overwritten by the forward solution Y = L^-1 B),
// X [H][n][nrhs].  Right-looking over 64-wide block columns; every block
// product runs on the tensor pipe as an exact product of 5-slice operands
// (2^-40 of each row's largest entry per operand, the same backward error as
// an fp64 factorisation to ~1e-12), and only the 64 x 64 diagonal factors
// and inverses (double-float, ~48 bits, from fp64 storage) and the block
// back substitution run on the SIMT pipes:
//   for k:  L_kk = chol(A_kk + lam I), Linv_kk = L_kk^-1        (double-float)
//           L_ik = A_ik Linv_kk^T                        i > k  (sliced)
//           A_ij -= L_ik L_jk^T                    j <= i, i > k  (sliced, lower tiles)
//           Y_k = Linv_kk B_k;  B_i -= L_ik Y_k         i > k  (sliced)
//   for k descending:  Z_k = sum_{i>k} L_ik^T X_i            (sliced)
//           X_k = Linv_kk^T (Y_k - Z_k)                         (fp64 SIMT)
// With one right-hand side both substitutions run in tri_solve_cluster_kernel.

constexpr int kCholSlices = 5;

__global__ void chol_lambda_kernel(const double* A, int n, double ridge, double tdiv, double* lam, DevStatus* stt) {
  chain_wait();
  __shared__ double red[8];
  const int b = blockIdx.x;
  const double* Ab = A + (long long)b * n * n;
  double a = 0.0;
  for (int r = threadIdx.x; r < n; r += 256) a += Ab[(long long)r * n + r];
  a = warp_sum_r(a);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tr = 0.0;
    for (int w = 0; w < 8; ++w) tr += red[w];
    if (!isfinite(tr)) set_status(stt, ARCKV_ERR_NONFINITE);
    lam[b] = ridge * tr / tdiv;
  }
}

// Factor diagonal block k of every head (one CTA per head) in double-float
// arithmetic: L_kk into A, L_kk^-1 into Linv[k] (fp64 storage); a
// non-positive pivot records ARCKV_ERR_NOT_SPD.
__global__ void __launch_bounds__(kCT, 1) chol_diag_kernel(double* A, double* Linv, int n, int k, const double* lam,
                                                           DevStatus* stt) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  df64* sm = (df64*)smraw;
  Tile<df64> S1 = (Tile<df64>)sm;
  Tile<df64> S2 = (Tile<df64>)(sm + kTileF<df64>);
  Tile<df64> S3 = (Tile<df64>)(sm + 2 * kTileF<df64>);
  __shared__ int bad;
  const int b = blockIdx.x, nblk = (n + NB - 1) / NB;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  load_diag(S1, A + (long long)b * n * n, n, k * NB, min(NB, n - k * NB), lam[b]);
  factor_diag<df64, double>(A + (long long)b * n * n, Linv + (long long)b * nblk * NB * NB, n, k, S1, S2, S3, &bad);
  if (threadIdx.x == 0 && bad) set_status(stt, ARCKV_ERR_NOT_SPD);
}

// X_k = Linv_kk^T (Y_k - Z_k) for block k of every head, kBackCols right-hand
// sides per CTA (grid: head x column group): V = Y_k - Z_k and Linv_kk go through
// shared memory, X[k0 + c][j] = sum_{l >= c} Linv_k[l][c] V[l][j].  Bound by the
// fp64 pipe (two multiply-adds per clock and SM): 8 columns a CTA spread 8 heads
// x 128 columns over 128 SMs, 32 left three quarters of them idle (30 us a block).
constexpr int kBackCols = 8;
__global__ void __launch_bounds__(256) chol_back_block_kernel(const double* Linv, const double* Y, const double* Z,
                                                              double* X, int n, int k, int nrhs, int useZ) {
  chain_wait();
  __shared__ double Ls[NB][NB + 1];
  __shared__ double Vs[NB][kBackCols + 1];
  const int b = blockIdx.x, j0 = blockIdx.y * kBackCols, nblk = (n + NB - 1) / NB, k0 = k * NB, kb = min(NB, n - k0);
  const int nj = min(kBackCols, nrhs - j0);
  const double* Li = Linv + ((long long)b * nblk + k) * NB * NB;
  const double* Yb = Y + ((long long)b * n + k0) * nrhs + j0;
  const double* Zb = Z + (long long)b * NB * nrhs + j0;
  double* Xb = X + ((long long)b * n + k0) * nrhs + j0;
  for (int e = threadIdx.x; e < NB * NB; e += 256) Ls[e / NB][e % NB] = Li[e];
  for (int e = threadIdx.x; e < NB * kBackCols; e += 256) {
    const int l = e / kBackCols, j = e % kBackCols;
    Vs[l][j] = (l < kb && j < nj) ? Yb[(long long)l * nrhs + j] - (useZ ? Zb[(long long)l * nrhs + j] : 0.0) : 0.0;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kb * kBackCols; e += 256) {
    const int c = e / kBackCols, j = e % kBackCols;
    double a = 0.0;
    for (int l = c; l < kb; ++l) a = fma(Ls[l][c], Vs[l][j], a);
    if (j < nj) Xb[(long long)c * nrhs + j] = a;
  }
}

// w[b][r] = sum_i Phi[b][i][r] a[b][i] (Phi fp32 [n][t], a fp64): one thread
// per column r, the rows of the column read coalesced across the warp.  The
// terms cancel heavily (|a| |Phi| exceeds |w| by ~1e4 on 128K caches), so the
// sum runs in double-float arithmetic: each product Phi a_hi + Phi a_lo is
// formed exactly up to the lo part's rounding and added with an error-free
// sum; a is split into fp32 (hi, lo) pairs in shared memory, 1024 rows at a time,
// and sixteen rows of Phi are in flight per thread (128 threads a CTA: at t = 2001
// the columns fill the SMs).
constexpr int kPtThreads = 128;
__global__ void __launch_bounds__(kPtThreads) phi_t_vec_kernel(const float* Phi, const double* a,
                                                        float* __restrict__ w, int n, int t) {
  chain_wait();
  __shared__ float ah[1024], al[1024];
  const int b = blockIdx.y, r = blockIdx.x * kPtThreads + threadIdx.x;
  const float* p = Phi + (long long)b * n * t + min(r, t - 1);
  const double* ab = a + (long long)b * n;
  df64 sum(0.f, 0.f);
  for (int i0 = 0; i0 < n; i0 += 1024) {
    const int cnt = min(1024, n - i0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kPtThreads) {
      const double v = ab[i0 + i];
      const float h = __double2float_rn(v);
      ah[i] = h;
      al[i] = __double2float_rn(v - (double)h);
    }
    __syncthreads();
    if (r < t) {
      auto add = [&](float x, int i) {
        const float ph = x * ah[i];
        const float pl = fmaf(x, al[i], fmaf(x, ah[i], -ph));
        df64 s2 = df_two(sum.hi, ph);
        s2.lo += sum.lo + pl;
        sum = df_fast2(s2.hi, s2.lo);
      };
      int i = 0;
      for (; i + 16 <= cnt; i += 16) {
        float x[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = p[(long long)(i0 + i + e) * t];
#pragma unroll
        for (int e = 0; e < 16; ++e) add(x[e], i + e);
      }
      for (; i < cnt; ++i) add(p[(long long)(i0 + i) * t], i);
    }
  }
  if (r < t) w[(long long)b * t + r] = sum.hi + sum.lo;
}

// Both substitutions of the single-right-hand-side dual beta system
// L L^T x = r (the fp64 factor in A's lower triangle, Linv the inverses of its
// 64 x 64 diagonal blocks) by a cluster of kTsCL CTAs per head: in each block
// step every rank sums its share of the off-diagonal blocks (block index
// j = rank mod kTsCL) into rank 0's shared memory, and rank 0 applies the
// diagonal block's inverse and publishes the block of the solution.  The fp64
// multiply-adds (n^2 per head) are spread over the cluster's SMs.  Every rank
// runs the same fixed trip counts, so every cluster barrier is reached by all.
constexpr int kTsCL = 8;
__global__ void __cluster_dims__(kTsCL, 1, 1) __launch_bounds__(256, 1)
    tri_solve_cluster_kernel(const double* A, const double* Linv,
                             const double* r, double* __restrict__ yd, double* __restrict__ x, int n) {
  chain_wait();
  namespace cg = cooperative_groups;
  __shared__ double red[kTsCL][NB];   // rank 0: the ranks' partial sums
  __shared__ double part[4][NB];
  __shared__ double v[NB];
  const int head = blockIdx.x / kTsCL, rank = (int)cluster_rank(), tid = threadIdx.x;
  const int nblk = (n + NB - 1) / NB;
  const double* Ab = A + (long long)head * n * n;
  const double* Lb = Linv + (long long)head * nblk * NB * NB;
  const double* rb = r + (long long)head * n;
  double* y = yd + (long long)head * n;
  double* xb = x + (long long)head * n;
  double* red0 = cg::this_cluster().map_shared_rank(&red[0][0], 0);
  // forward: y_k = Linv_kk (r_k - sum_{j<k} L_kj y_j)
  for (int k = 0; k < nblk; ++k) {
    const int k0 = k * NB, kb = min(NB, n - k0);
    {  // four threads per row of block k
      const int rr = tid >> 2, pt = tid & 3;
      double a0 = 0.0, a1 = 0.0;
      if (rr < kb) {
        const double* row = Ab + (long long)(k0 + rr) * n;
        for (int j = rank; j < k; j += kTsCL)
          for (int c = j * NB + pt; c < j * NB + NB; c += 8) {
            a0 = fma(__ldcg(row + c), __ldcg(y + c), a0);
            a1 = fma(__ldcg(row + c + 4), __ldcg(y + c + 4), a1);
          }
      }
      double a = a0 + a1;
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      if (pt == 0) red0[rank * NB + rr] = a;
    }
    cluster_sync_all();
    if (rank == 0) {
      if (tid < NB) {
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < kTsCL; ++q) sum += red[q][tid];
        v[tid] = tid < kb ? rb[k0 + tid] - sum : 0.0;
      }
      __syncthreads();
      const int c = tid >> 2, pt = tid & 3;   // y_k[c] = sum_{l <= c} Linv_k[c][l] v[l]
      const double* Li = Lb + (long long)k * NB * NB + c * NB;
      double a = 0.0;
      for (int l = pt; l <= c; l += 4) a = fma(__ldcg(Li + l), v[l], a);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      if (pt == 0 && c < kb) y[k0 + c] = a;
    }
    cluster_sync_all();
  }
  // backward: x_k = Linv_kk^T (y_k - sum_{j>k} L_jk^T x_j)
  for (int k = nblk - 1; k >= 0; --k) {
    const int k0 = k * NB, kb = min(NB, n - k0);
    {  // column c of block k, four row groups
      const int c = tid & (NB - 1), pt = tid >> 6;
      double a0 = 0.0, a1 = 0.0;
      if (c < kb)
        for (int j = k + 1 + rank; j < nblk; j += kTsCL) {
          const int i1 = min(n, j * NB + NB);
          for (int i = j * NB + pt; i < i1; i += 8) {
            a0 = fma(__ldcg(Ab + (long long)i * n + k0 + c), __ldcg(xb + i), a0);
            if (i + 4 < i1) a1 = fma(__ldcg(Ab + (long long)(i + 4) * n + k0 + c), __ldcg(xb + i + 4), a1);
          }
        }
      part[pt][c] = a0 + a1;
    }
    __syncthreads();
    if (tid < NB) red0[rank * NB + tid] = (part[0][tid] + part[1][tid]) + (part[2][tid] + part[3][tid]);
    cluster_sync_all();
    if (rank == 0) {
      if (tid < NB) {
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < kTsCL; ++q) sum += red[q][tid];
        v[tid] = tid < kb ? y[k0 + tid] - sum : 0.0;
      }
      __syncthreads();
      const int c = tid >> 2, pt = tid & 3;   // x_k[c] = sum_{l >= c} Linv_k[l][c] v[l]
      const double* Li = Lb + (long long)k * NB * NB;
      double a = 0.0;
      for (int l = c + pt; l < NB; l += 4) a = fma(__ldcg(Li + (long long)l * NB + c), v[l], a);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      if (pt == 0 && c < kb) xb[k0 + c] = a;
    }
    cluster_sync_all();
  }
}

struct CholSlicedBufs {
  bf16 *sA, *sB, *sC;   // 5-slice operands: panel rows / columns, Linv_kk rows, right-hand-side columns
  int *eA, *eB, *eC;
  double *lam, *Z;      // [H], [H][64][nrhs]
};

// A second stream per calling stream (created on first use, kept for the
// process) and two events, for the look-ahead of the blocked dual Cholesky.
struct SideStream {
  cudaStream_t s;
  cudaEvent_t fork, join;
};
static bool side_stream(cudaStream_t main, SideStream& out) {
  static std::mutex mu;
  static std::map<std::pair<int, cudaStream_t>, SideStream> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> g(mu);
  auto it = cache.find({dev, main});
  if (it != cache.end()) {
    out = it->second;
    return true;
  }
  SideStream ss{};
  if (cudaStreamCreateWithFlags(&ss.s, cudaStreamNonBlocking) != cudaSuccess) return false;
  if (cudaEventCreateWithFlags(&ss.fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&ss.join, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cache[{dev, main}] = ss;
  out = ss;
  return true;
}

// Blocked right-looking Cholesky of the n x n systems with a look-ahead of
// one block: after step k's panel the trailing matrix is updated in two
// launches, first its leading 64-column block (block k + 1, all rows), then
// the rest of its lower triangle; the second runs on the calling stream
// while a side stream factors block k + 1, slices its inverse and forms and
// slices the panel below it, so the diagonal factor and the panel leave the
// critical path: the second update leaves kAheadSMs SMs free (its
// persistent grid is capped) and the side stream's panel product takes at
// most that many CTAs.  Slices of consecutive steps alternate between two
// buffers.
// The operations and their order per element are those of the plain blocked
// algorithm.
static int chol_solve_sliced(int H, int n, double* A, double* Linv, double* B, double* X, int nrhs, double ridge,
                             double tdiv, const CholSlicedBufs& W, DevStatus* stt, cudaStream_t st) {
  constexpr int S = kCholSlices;
  const int nblk = (n + NB - 1) / NB;
  const long long nn = (long long)n * n, nr = (long long)n * nrhs, lb = (long long)nblk * NB * NB;
  const int dsm = 3 * kTileF<df64> * (int)sizeof(df64);
  if (set_dyn_smem((const void*)chol_diag_kernel, dsm) != cudaSuccess)
    return -1;
  int nl = 0;
  auto ok = [&](int r) {
    if (r < 0) return false;
    nl += r;
    return true;
  };
  SideStream ss{};
  const bool ahead = nblk > 1 && side_stream(st, ss);
  constexpr int kAheadSMs = 16;
  const int main_ctas = ahead ? std::max(1, tc_gemm_sm_count() - kAheadSMs) : 0, side_ctas = ahead ? kAheadSMs : 0;
  const cudaStream_t sd = ahead ? ss.s : st;
  const long long sa_stride = (long long)S * H * n * NB, sb_stride = (long long)S * H * NB * NB;
  auto SA = [&](int k) { return W.sA + (k & 1) * sa_stride; };
  auto EA = [&](int k) { return W.eA + (k & 1) * (long long)H * n; };
  auto SB = [&](int k) { return W.sB + (k & 1) * sb_stride; };
  auto EB = [&](int k) { return W.eB + (k & 1) * (long long)H * NB; };
  // block k: its diagonal factor and inverse, the inverse's slices, the panel
  // L_ik = A_ik Linv_kk^T below it and the panel's slices (on stream s)
  auto diag_panel = [&](int k, cudaStream_t s) -> bool {
    const int k0 = k * NB, kb = std::min(NB, n - k0), m = n - k0 - kb;
    launch_chained(chol_diag_kernel, H, kCT, dsm, s, A, Linv, n, k, W.lam, stt);
    ++nl;
    if (!ok(launch_slice_rows(S, Linv + (long long)k * NB * NB, kb, kb, NB, lb, H, SB(k), EB(k), s))) return false;
    if (m > 0) {
      double* panel = A + (long long)(k0 + kb) * n + k0;
      if (!ok(launch_slice_rows(S, panel, m, kb, n, nn, H, SA(k), EA(k), s))) return false;
      if (!ok(launch_sliced_f64(S, SA(k), EA(k), m, SB(k), EB(k), kb, kb, H, panel, nn, n, false, false, stt, s, 0,
                                1 << 30, s == st ? 0 : side_ctas)))
        return false;
      if (!ok(launch_slice_rows(S, panel, m, kb, n, nn, H, SA(k), EA(k), s))) return false;
    }
    return true;
  };
  launch_chained(chol_lambda_kernel, H, 256, 0, st, A, n, ridge, tdiv, W.lam, stt);
  ++nl;
  if (!diag_panel(0, st)) return -1;
  for (int k = 0; k < nblk; ++k) {
    const int k0 = k * NB, kb = std::min(NB, n - k0), m = n - k0 - kb;
    if (m > 0) {
      // A_ij -= L_ik L_jk^T on the trailing lower triangle: block k + 1 first
      double* trail = A + (long long)(k0 + kb) * n + k0 + kb;
      if (!ok(launch_sliced_f64(S, SA(k), EA(k), m, SA(k), EA(k), m, kb, H, trail, nn, n, true, true, stt, st, 0, 1)))
        return -1;
      if (ahead) {
        cudaEventRecord(ss.fork, st);
        cudaStreamWaitEvent(sd, ss.fork, 0);
      }
      if (!diag_panel(k + 1, sd)) return -1;
      if (!ok(launch_sliced_f64(S, SA(k), EA(k), m, SA(k), EA(k), m, kb, H, trail, nn, n, true, true, stt, st, 1,
                                1 << 30, main_ctas)))
        return -1;
    }
    if (nrhs > 1) {
      // Y_k = Linv_kk B_k over B_k; B_i -= L_ik Y_k
      double* Bk = B + (long long)k0 * nrhs;
      if (!ok(launch_slice_cols(S, Bk, kb, nrhs, nrhs, nr, H, W.sC, W.eC, st))) return -1;
      if (!ok(launch_sliced_f64(S, SB(k), EB(k), kb, W.sC, W.eC, nrhs, kb, H, Bk, nr, nrhs, false, false, stt, st)))
        return -1;
      if (m > 0) {
        if (!ok(launch_slice_cols(S, Bk, kb, nrhs, nrhs, nr, H, W.sC, W.eC, st))) return -1;
        if (!ok(launch_sliced_f64(S, SA(k), EA(k), m, W.sC, W.eC, nrhs, kb, H, Bk + (long long)kb * nrhs, nr, nrhs,
                                  false, true, stt, st)))
          return -1;
      }
    }
    if (ahead && m > 0) {
      cudaEventRecord(ss.join, sd);
      cudaStreamWaitEvent(st, ss.join, 0);
    }
  }
  if (nrhs == 1) {
    // one right-hand side: both substitutions by a cluster per head (fp64,
    // n^2 multiply-adds spread over its SMs), the forward result left in W.Z
    launch_chained(tri_solve_cluster_kernel, H * kTsCL, 256, 0, st, A, Linv, B, W.Z, X, n);
    return nl + 1;
  }
  for (int k = nblk - 1; k >= 0; --k) {
    const int k0 = k * NB, kb = std::min(NB, n - k0), m = n - k0 - kb;
    if (m > 0) {
      // Z_k = sum_{i>k} L_ik^T X_i: the columns of the panel against the columns of X below block k
      const double* panel = A + (long long)(k0 + kb) * n + k0;
      if (!ok(launch_slice_cols(S, panel, m, kb, n, nn, H, W.sA, W.eA, st))) return -1;
      if (!ok(launch_slice_cols(S, X + (long long)(k0 + kb) * nrhs, m, nrhs, nrhs, nr, H, W.sC, W.eC, st))) return -1;
      if (!ok(launch_sliced_f64(S, W.sA, W.eA, kb, W.sC, W.eC, nrhs, m, H, W.Z, (long long)NB * nrhs, nrhs, false,
                                false, stt, st)))
        return -1;
    }
    launch_chained(chol_back_block_kernel, dim3(H, cdiv(nrhs, kBackCols)), 256, 0, st, Linv, B, W.Z, X, n, k, nrhs, m > 0 ? 1 : 0);
    ++nl;
  }
  return nl;
}

// Dual (push-through) form of both ridge fits for t > n, where the primal
// t x t normal matrices have rank <= n:
//   (Phi^T Phi + lam I) w = Phi^T m   <=>   w = Phi^T a,  (Phi Phi^T + lam I) a = m
//   (P^T P + lam I) C_v = P^T Y       <=>   C_v = P^T A,  (P P^T + lam I) A = Y
// with the same lam = ridge * trace / t (trace(Phi^T Phi) = trace(Phi Phi^T)),
// so the solutions equal the primal ones; the systems are n x n.  These
// systems reach condition numbers ~1e8 on 128K caches (lam relative to t
// diagonal entries, n of them carrying the mass), and a Gram error that does
// not keep the Gram structure moves beta by up to cond x error: the n x n
// Grams are exact products of row-sliced Phi / P^ on the tensor cores (4
// slices: 32 bits of each row relative to its largest entry, a perturbation
// of the operand itself), the solves are fp64-grade (chol_solve_sliced),
// w = Phi^T a is summed in double-float and C_v = P^T A is a 4-slice
// tensor-core product (with 3 slices for P^ the held-out outputs of a 128K
// head drift by ~7e-3).  Beyond kSlicedMaxK the fp64 SIMT products serve.
static int fits_dual(const Dims& D, float ridge_w, float ridge_v, float eps_w, float b_min, float b_max,
                     const float* m, const float* Y, const FitBufs& B, float* beta, float* C_v, DevStatus* stt,
                     cudaStream_t st, cudaEvent_t const* ev) {
  auto mark = [&](int s) {
    if (ev) cudaEventRecord(ev[s], st);
  };
  const long long nt = (long long)D.n * D.t, nd = (long long)D.n * D.d;
  const bool sliced = sliced_supported(D.t) && sliced_supported(D.n);
  const dim3 sgrid(cdiv(D.n, 64), cdiv(D.n, 64), D.H);
  int nl = 0;
  auto gram = [&](int S) -> int {   // B.G64 = X X^T for X = B.Phi [n][t]
    if (!sliced) {
      launch_chained(syrk64_kernel, sgrid, 256, 0, st, B.Phi, B.G64, D.n, D.t);
      return 1;
    }
    const int a = launch_slice_rows(S, B.Phi, D.n, D.t, D.t, nt, D.H, B.Sl, B.eR, st);
    const int g = launch_sliced_gram_lower(S, B.Sl, B.eR, D.n, D.t, D.H, B.G64, stt, st);
    return (a < 0 || g < 0) ? -1 : a + g;
  };
  // beta system
  int r = gram(4);
  if (r < 0) return -1;
  nl += r;
  const CholSlicedBufs CW{B.Sl, B.Sl2, B.Sl3, B.eR, B.eC, B.eC2, B.cl_lam, B.Z64};
  auto solve = [&](int nrhs, long long nrow, float ridge) -> int {
    if (sliced) return chol_solve_sliced(D.H, D.n, B.G64, B.L64, B.B64, B.X64, nrhs, ridge, D.t, CW, stt, st);
    return cholesky_solve64(D.H, D.n, B.G64, B.L64, B.B64, B.Z64, B.X64, nrhs, nrow, ridge, D.t, stt, st);
  };
  mark(8);
  launch_chained(widen_kernel, cdiv((long long)D.H * D.n, 256), 256, 0, st, m, B.B64, (long long)D.H * D.n);
  r = solve(1, D.n, ridge_w);
  if (r < 0) return -1;
  nl += 1 + r;
  launch_chained(phi_t_vec_kernel, dim3(cdiv(D.t, kPtThreads), D.H), kPtThreads, 0, st, B.Phi, B.X64, B.rhs, D.n, D.t);   // w = Phi^T a
  const long long ht = (long long)D.H * D.t;
  launch_chained(beta_kernel, cdiv(ht, 256), 256, 0, st, B.rhs, beta, ht, eps_w, b_min, b_max);
  launch_chained(softmax_bias_kernel, dim3(cdiv(D.n, 8), D.H), 256, 0, st, B.LC, beta, B.Phi, D.n, D.t);
  nl += 3;
  // value system
  mark(9);
  r = gram(4);
  if (r < 0) return -1;
  nl += r;
  mark(10);
  launch_chained(widen_kernel, cdiv((long long)D.H * nd, 256), 256, 0, st, Y, B.B64, (long long)D.H * nd);
  r = solve(D.d, nd, ridge_v);
  if (r < 0) return -1;
  nl += 1 + r;
  if (!sliced) {
    launch_chained(xty64_kernel, dim3(cdiv(D.t, 64), cdiv(D.d, 32), D.H), 256, 0, st, B.Phi, B.X64, C_v, D.n, D.t, D.d);
    return nl + 1;
  }
  // C_v = P^T A: the rows of P^T (columns of P) and of A^T, 4 slices each
  const int a = launch_slice_cols(4, B.Phi, D.n, D.t, D.t, nt, D.H, B.Sl, B.eR, st);
  const int b = launch_slice_cols(4, B.X64, D.n, D.d, D.d, nd, D.H, B.Sl2, B.eC, st);
  const int c = launch_sliced_product_f32(4, B.Sl, B.eR, D.t, B.Sl2, B.eC, D.d, D.n, D.H, C_v, D.d, stt, st);
  if (a < 0 || b < 0 || c < 0) return -1;
  return nl + a + b + c;
}

// ---------------------------------------------------------------------------
// Iterative refinement of the beta system (t <= n; App. A.9 Eq. mass_fit).
// The tensor-core Gram and factor are fp32-grade; with condition numbers up to
// ~1e7 that leaves beta a few 1e-3 off on long caches.  Each step forms the
// residual of the normal equations against Phi itself in fp64,
//     r = Phi^T (m - Phi x) - lam x,   lam = ridge * sum_ir Phi_ir^2 / t,
// (the exact normal matrix of the fp32 Phi, no Gram rounding) and corrects
// x += (L L^T)^-1 r with the factor the solver left behind: L_kk and the
// off-diagonal blocks in the Gram's lower part, L_kk^-1 in Linv.

// u[b][i] = m_i - sum_r Phi_ir x_r (fp64); with sq, also sq[b][i] = sum_r Phi_ir^2.
// One warp per row, eight loads in flight per lane; x is widened once per CTA.
constexpr int kIrTile = 2048;   // columns of x in shared memory at a time
__global__ void __launch_bounds__(256) ir_rows_kernel(const float* Phi, const float* m,
                                                      const float* x, double* __restrict__ u,
                                                      double* __restrict__ sq, int n, int t) {
  chain_wait();
  __shared__ double xd[kIrTile];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.y, row = blockIdx.x * 8 + warp;
  const long long gr = (long long)b * n + row;
  const float* p = Phi + gr * t;
  const float* xb = x + (long long)b * t;
  double a = 0.0, q = 0.0;
  for (int c0 = 0; c0 < t; c0 += kIrTile) {
    const int cn = min(kIrTile, t - c0);
    __syncthreads();
    for (int c = threadIdx.x; c < cn; c += 256) xd[c] = widen_bits(xb[c0 + c]);
    __syncthreads();
    if (row < n) {
      for (int r0 = lane; r0 < cn; r0 += 256) {
        float pv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) pv[e] = r0 + 32 * e < cn ? p[c0 + r0 + 32 * e] : 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (r0 + 32 * e < cn) {
            const double v = widen_bits(pv[e]);
            a = fma(v, xd[r0 + 32 * e], a);
            if (sq) q = fma(v, v, q);
          }
        }
      }
    }
  }
  if (row >= n) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    q += __shfl_xor_sync(0xffffffffu, q, o);
  }
  if (lane == 0) {
    u[gr] = (double)m[gr] - a;
    if (sq) sq[gr] = q;
  }
}

// lam[b] = ridge * sum_i sq[b][i] / t, summed in a fixed order (one CTA per head).
__global__ void __launch_bounds__(256) ir_lambda_kernel(const double* sq, double* __restrict__ lam, int n,
                                                        int t, double ridge) {
  chain_wait();
  __shared__ double red[8];
  const int b = blockIdx.x;
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) a += sq[(long long)b * n + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    lam[b] = ridge * s / t;
  }
}

// r[b][c] = sum_i Phi_ic u_i - lam x_c (fp64 sums, rounded to fp32 at the end).
// A CTA takes 32 columns (lane = column, coalesced rows); its 32 warps are 8
// row phases of four chains each: chain q of phase w takes the rows w + 8 q +
// 32 j, chain 0 also what is left below n.  The chains of a phase are added,
// then the phases in order.
__global__ void __launch_bounds__(1024) ir_cols_kernel(const float* Phi, const double* u,
                                                       const float* x, const double* lam,
                                                       float* __restrict__ r, int n, int t) {
  chain_wait();
  __shared__ double part[32][32];
  const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int w = warp & 7, q = warp >> 3;
  const float* p = Phi + (long long)b * n * t + c;
  const double* ub = u + (long long)b * n;
  double a = 0.0;
  if (c < t) {
    int i = w;
    for (; i + 24 + 96 < n; i += 128) {   // four rows of the chain in flight
      float pv[4];
      double uv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        pv[e] = p[(long long)(i + 8 * q + 32 * e) * t];
        uv[e] = ub[i + 8 * q + 32 * e];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) a = fma(widen_bits(pv[e]), uv[e], a);
    }
    for (; i + 24 < n; i += 32) a = fma(widen_bits(p[(long long)(i + 8 * q) * t]), ub[i + 8 * q], a);
    if (q == 0)
      for (; i < n; i += 8) a = fma(widen_bits(p[(long long)i * t]), ub[i], a);
  }
  part[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && c < t) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double ph = (part[k][lane] + part[k + 8][lane]) + (part[k + 16][lane] + part[k + 24][lane]);
      s = k == 0 ? ph : s + ph;
    }
    r[(long long)b * t + c] = (float)(s - lam[b] * (double)x[(long long)b * t + c]);
  }
}

// x += (L L^T)^-1 r, one cluster of eight CTAs per head, for the refinement
// steps of the primal beta solve: forward y_k = Linv_kk (r_k - sum_{j<k} L_kj y_j),
// then d_k = Linv_kk^T (y_k - sum_{j>k} L_jk^T d_j), x_k += d_k.  Serial over the
// blocks, so the time of a step is what counts: one exchange between the CTAs
// (remote stores counted on mbarriers, about half a cluster barrier), a short
// sum and a 64 x 64 mat-vec, everything that does not depend on the previous
// block loaded ahead.
//   forward, right-looking: rank k % 8 keeps the sums of block k's rows in
//     registers (row = thread / 8; chain (part, q) takes the columns part + 8 q
//     + 32 i), adds each y_j as it comes and broadcasts y_k;
//   backward: a sum runs upwards from the newest block, so it cannot be formed
//     ahead; its chains (part, q, column; rows part + 8 q + 32 i below block k,
//     chain 0 also what is left below t) are dealt by part over the ranks, whose
//     slices of L's column panel arrive by cp.async a step ahead, and every
//     rank forms d_k for itself from the eight parts.
// 43 us at t = 819 and 93 us at t = 1638 (8 heads); one CTA per head took 219
// and 740 us.
constexpr int kTriCL = 8, kTriMaxT = 2048, kTriSlots = kTriMaxT / (NB * kTriCL);
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
// Store to the same shared address of another CTA of the cluster, counted on
// that CTA's mbarrier.
__device__ __forceinline__ void st_remote(const float* p, const uint64_t* bar, int rank, float v) {
  asm volatile(
      "{\n\t.reg .b32 a, m;\n\t"
      "mapa.shared::cluster.u32 a, %0, %2;\n\t"
      "mapa.shared::cluster.u32 m, %1, %2;\n\t"
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [a], %3, [m];\n\t}\n" ::"r"(tc::smem_u32(p)),
      "r"(tc::smem_u32(bar)), "r"(rank), "r"(__float_as_uint(v))
      : "memory");
}
__global__ void __cluster_dims__(kTriCL, 1, 1) __launch_bounds__(512, 1)
    tri_solve_cluster32_kernel(const float* A, const float* Linv,
                               const float* r, float* __restrict__ x, int t, DevStatus* stt) {
  chain_wait();
  extern __shared__ __align__(16) float psm[];   // two panel slices [2 nblk][4][64]
  __shared__ float yv[kTriMaxT];                 // y, then d block by block
  __shared__ float v[NB];
  __shared__ float parts[2][8][NB];              // backward: the ranks' sums of alternate steps
  // one-shot mbarriers: y_k has arrived (forward), all parts of step k have (backward)
  __shared__ uint64_t ybar[kTriMaxT / NB], pbar[kTriMaxT / NB];
  __shared__ int abort_flag;
  const int head = blockIdx.x / kTriCL, rank = (int)cluster_rank(), tid = threadIdx.x;
  const int nblk = (t + NB - 1) / NB;
  if (tid < nblk) {
    tc::mbar_init(&ybar[tid], 1);
    tc::mbar_init(&pbar[tid], 1);
    tc::mbar_fence_init();
    tc::mbar_arrive_expect_tx(&ybar[tid], NB * 4);
    tc::mbar_arrive_expect_tx(&pbar[tid], kTriCL * NB * 4);
  }
  if (tid == 0) abort_flag = 0;
  __syncthreads();
  cluster_sync_all();   // every rank's barriers are armed
  const float* Ab = A + (long long)head * t * t;
  const float* Lb = Linv + (long long)head * nblk * NB * NB;
  const float* rb = r + (long long)head * t;
  float* xb = x + (long long)head * t;
  const int rr = tid >> 3, pt = tid & 7;
  // forward
  float ch[kTriSlots][4], lv[kTriSlots][8];
#pragma unroll
  for (int s = 0; s < kTriSlots; ++s)
#pragma unroll
    for (int q = 0; q < 4; ++q) ch[s][q] = 0.f;
  auto fetch = [&](int j) {   // L_kj of this rank's blocks k > j
#pragma unroll
    for (int s = 0; s < kTriSlots; ++s) {
      const int k = rank + kTriCL * s, row = k * NB + rr;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        lv[s][e] = (k > j && k < nblk && row < t) ? __ldcg(Ab + (long long)row * t + j * NB + pt + 8 * e) : 0.f;
    }
  };
  float li[8], rv = 0.f;   // Linv_k row rr (from part pt) and r of this rank's next block
  auto fetch_li = [&](int k) {
    if (rank != k % kTriCL || k >= nblk) return;
    const float* Li = Lb + (long long)k * NB * NB + rr * NB;
#pragma unroll
    for (int e = 0; e < 8; ++e) li[e] = pt + 8 * e <= rr ? __ldcg(Li + pt + 8 * e) : 0.f;
    rv = k * NB + rr < t ? rb[k * NB + rr] : 0.f;
  };
  fetch_li(0);
  for (int k = 0; k < nblk; ++k) {
    if (k > 0) {   // y_{k-1} has arrived: add it to the sums
      tc::mbar_wait(&ybar[k - 1], 0, &abort_flag, stt);
      const float* y = yv + (k - 1) * NB;
#pragma unroll
      for (int s = 0; s < kTriSlots; ++s)
        if (rank + kTriCL * s >= k) {
#pragma unroll
          for (int e = 0; e < 8; ++e) ch[s][e & 3] = fmaf(lv[s][e], y[pt + 8 * e], ch[s][e & 3]);
        }
    }
    if (rank == k % kTriCL) {
      const int k0 = k * NB, kb = min(NB, t - k0);
      float a = 0.f;
#pragma unroll
      for (int s = 0; s < kTriSlots; ++s)
        if (s == k / kTriCL) a = (ch[s][0] + ch[s][1]) + (ch[s][2] + ch[s][3]);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      if (pt == 0) v[rr] = rr < kb ? rv - a : 0.f;
      __syncthreads();
      float y = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (pt + 8 * e <= rr) y = fmaf(li[e], v[pt + 8 * e], y);
      y += __shfl_xor_sync(0xffffffffu, y, 1);
      y += __shfl_xor_sync(0xffffffffu, y, 2);
      y += __shfl_xor_sync(0xffffffffu, y, 4);
      st_remote(&yv[k0 + rr], &ybar[k], pt, rr < kb ? y : 0.f);   // lane pt of the row writes it to rank pt
    }
    fetch(k);
    fetch_li(k + 1);
  }
  tc::mbar_wait(&ybar[nblk - 1], 0, &abort_flag, stt);
  // backward; thread (c, q) of the first 256 owns chain (rank, q, c)
  const int c = tid & 63, q = tid >> 6;
  const int slice = 2 * nblk * 256;
  auto panel = [&](int k) {   // this rank's rows of L's column block k, below the block
    float* dst = psm + (k & 1) * slice;
    const int k0 = k * NB;
    if (k >= 0 && tid < 256)
      for (int i = 0, base = k0 + NB + rank; base < t; base += 32, ++i) {
        const int row = base + 8 * q;
        if (row < t) cp_async4(dst + i * 256 + q * 64 + c, Ab + (long long)row * t + k0 + c);
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  panel(nblk - 1);
  panel(nblk - 2);
  for (int k = nblk - 1; k >= 0; --k) {
    const int k0 = k * NB, kb = min(NB, t - k0);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // this step's slice, and the previous step's d
    const float* P = psm + (k & 1) * slice;
    if (tid < 256) {
      float a = 0.f;
      if (c < kb) {
        int i = 0, base = k0 + NB + rank;
#pragma unroll 4
        for (; base + 24 < t; base += 32, ++i) a = fmaf(P[i * 256 + q * 64 + c], yv[base + 8 * q], a);
        if (q == 0)   // rows base, base + 8, base + 16 below t
          for (int e = 0; base + 8 * e < t; ++e) a = fmaf(P[i * 256 + e * 64 + c], yv[base + 8 * e], a);
      }
      // the four chains of a column are in warps w, w + 2, w + 4, w + 6: through shared memory
      psm[2 * slice + q * 64 + c] = a;
    }
    __syncthreads();
    {
      const float* s4 = psm + 2 * slice;
      const int col = tid >> 3;   // lane pt of the column writes it to rank pt
      const float a = (s4[col] + s4[64 + col]) + (s4[128 + col] + s4[192 + col]);
      st_remote(&parts[k & 1][rank][col], &pbar[k], pt, a);
    }
    panel(k - 2);
    const float* Li = Lb + (long long)k * NB * NB;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int l = rr + pt + 8 * e;   // column rr of Linv, rows l >= rr
      li[e] = l < NB ? __ldcg(Li + l * NB + rr) : 0.f;
    }
    if (tid < NB) {
      tc::mbar_wait(&pbar[k], 0, &abort_flag, stt);
      float a = 0.f;
#pragma unroll
      for (int p = 0; p < 8; ++p) a += parts[k & 1][p][tid];
      v[tid] = tid < kb ? yv[k0 + tid] - a : 0.f;
    }
    __syncthreads();
    float d = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (rr + pt + 8 * e < NB) d = fmaf(li[e], v[rr + pt + 8 * e], d);
    d += __shfl_xor_sync(0xffffffffu, d, 1);
    d += __shfl_xor_sync(0xffffffffu, d, 2);
    d += __shfl_xor_sync(0xffffffffu, d, 4);
    if (pt == 0 && rr < kb) {
      yv[k0 + rr] = d;
      if (rank == k % kTriCL) xb[k0 + rr] += d;
    }
  }
  cluster_sync_all();   // nobody leaves before the last stores into its shared memory have been waited for
}

// x += (L L^T)^-1 r for one head per CTA (512 threads): forward substitution
// y_k = Linv_kk (r_k - sum_{j<k} L_kj y_j), then x_k += Linv_kk^T (y_k -
// sum_{j>k} L_jk^T d_j).  y and the correction d live in `yd` ([H][t]).
// Serves the refinement steps beyond kTriMaxT, where a rank's sums and panel
// slices no longer fit.
template <typename R>
__global__ void __launch_bounds__(512) tri_solve_kernel(const R* A, const R* Linv,
                                                        const R* r, R* __restrict__ yd,
                                                        R* __restrict__ x, int t) {
  chain_wait();
  constexpr int NBk = kCholNB;
  __shared__ R v[NBk];
  __shared__ R part[8][NBk];
  const int b = blockIdx.x, tid = threadIdx.x;
  const int nblk = (t + NBk - 1) / NBk;
  const R* Ab = A + (long long)b * t * t;
  const R* Lb = Linv + (long long)b * nblk * NBk * NBk;
  const R* rb = r + (long long)b * t;
  R* y = yd + (long long)b * t;
  R* xb = x + (long long)b * t;
  // forward: 8 threads per row of block k sum L_kj y_j over the columns before k0
  for (int k = 0; k < nblk; ++k) {
    const int k0 = k * NBk, kb = min(NBk, t - k0);
    {
      const int rr = tid >> 3, pt = tid & 7;
      R a = R(0), a2 = R(0), a3 = R(0), a4 = R(0);
      if (rr < kb) {
        const R* row = Ab + (long long)(k0 + rr) * t;
        int c = pt;
        for (; c + 24 < k0; c += 32) {   // four independent chains: eight loads in flight together
          const R l0 = __ldcg(row + c), l1 = __ldcg(row + c + 8), l2 = __ldcg(row + c + 16), l3 = __ldcg(row + c + 24);
          const R y0 = __ldcg(y + c), y1 = __ldcg(y + c + 8), y2 = __ldcg(y + c + 16), y3 = __ldcg(y + c + 24);
          a = fma_r(l0, y0, a);
          a2 = fma_r(l1, y1, a2);
          a3 = fma_r(l2, y2, a3);
          a4 = fma_r(l3, y3, a4);
        }
        for (; c < k0; c += 8) a = fma_r(__ldcg(row + c), __ldcg(y + c), a);
      }
      a = (a + a2) + (a3 + a4);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      if (pt == 0) v[rr] = rr < kb ? rb[k0 + rr] - a : R(0);
    }
    __syncthreads();
    {  // y_k[c] = sum_{l <= c} Linv_k[c][l] v[l]
      const int c = tid >> 3, pt = tid & 7;
      const R* Li = Lb + (long long)k * NBk * NBk + c * NBk;
      R a = R(0);
      for (int l = pt; l <= c; l += 8) a = fma_r(__ldcg(Li + l), v[l], a);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      if (pt == 0 && c < kb) y[k0 + c] = a;
    }
    __threadfence_block();
    __syncthreads();
  }
  // backward: column c of block k, eight row parts; the correction d
  // overwrites y block by block (rows after k0 + kb already hold d)
  for (int k = nblk - 1; k >= 0; --k) {
    const int k0 = k * NBk, kb = min(NBk, t - k0);
    {
      const int c = tid & (NBk - 1), pt = tid >> 6;
      R a = R(0), a2 = R(0), a3 = R(0), a4 = R(0);
      if (c < kb) {
        const R* col = Ab + k0 + c;
        int rr = k0 + kb + pt;
        for (; rr + 24 < t; rr += 32) {
          const R l0 = __ldcg(col + (long long)rr * t), l1 = __ldcg(col + (long long)(rr + 8) * t);
          const R l2 = __ldcg(col + (long long)(rr + 16) * t), l3 = __ldcg(col + (long long)(rr + 24) * t);
          const R y0 = __ldcg(y + rr), y1 = __ldcg(y + rr + 8), y2 = __ldcg(y + rr + 16), y3 = __ldcg(y + rr + 24);
          a = fma_r(l0, y0, a);
          a2 = fma_r(l1, y1, a2);
          a3 = fma_r(l2, y2, a3);
          a4 = fma_r(l3, y3, a4);
        }
        for (; rr < t; rr += 8) a = fma_r(__ldcg(col + (long long)rr * t), __ldcg(y + rr), a);
      }
      part[pt][c] = (a + a2) + (a3 + a4);
    }
    __syncthreads();
    if (tid < NBk) {
      R a = R(0);
#pragma unroll
      for (int q = 0; q < 8; ++q) a += part[q][tid];
      v[tid] = tid < kb ? y[k0 + tid] - a : R(0);
    }
    __syncthreads();
    {  // d_k[c] = sum_{l >= c} Linv_k[l][c] v[l]
      const int c = tid >> 3, pt = tid & 7;
      const R* Li = Lb + (long long)k * NBk * NBk;
      R a = R(0);
      for (int l = c + pt; l < NBk; l += 8) a = fma_r(__ldcg(Li + (long long)l * NBk + c), v[l], a);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      if (pt == 0 && c < kb) {
        y[k0 + c] = a;
        xb[k0 + c] += a;
      }
    }
    __threadfence_block();
    __syncthreads();
  }
}

constexpr int kBetaRefineSteps = 2;

static int refine_beta(const Dims& D, float ridge_w, const float* m, const FitBufs& B, DevStatus* stt, cudaStream_t st) {
  const dim3 rows(cdiv(D.n, 8), D.H);
  const int nblk = cdiv(D.t, NB), smem = (2 * 2 * nblk * 256 + 256) * (int)sizeof(float);
  const bool cluster = D.t <= kTriMaxT;
  if (cluster && set_dyn_smem((const void*)tri_solve_cluster32_kernel, smem) != cudaSuccess) return -1;
  launch_chained(ir_rows_kernel, rows, 256, 0, st, B.Phi, m, B.wsol, B.ir_u, B.ir_sq, D.n, D.t);
  launch_chained(ir_lambda_kernel, D.H, 256, 0, st, B.ir_sq, B.ir_lam, D.n, D.t, (double)ridge_w);
  int nl = 2;
  for (int it = 0; it < kBetaRefineSteps; ++it) {
    if (it > 0) {
      launch_chained(ir_rows_kernel, rows, 256, 0, st, B.Phi, m, B.wsol, B.ir_u, nullptr, D.n, D.t);
      ++nl;
    }
    launch_chained(ir_cols_kernel, dim3(cdiv(D.t, 32), D.H), 1024, 0, st, B.Phi, B.ir_u, B.wsol, B.ir_lam, B.rhs, D.n, D.t);
    if (cluster)
      launch_chained(tri_solve_cluster32_kernel, kTriCL * D.H, 512, smem, st, B.Gram, B.Linv, B.rhs, B.wsol, D.t, stt);
    else
      launch_chained(tri_solve_kernel<float>, D.H, 512, 0, st, B.Gram, B.Linv, B.rhs, B.Z, B.wsol, D.t);
    nl += 2;
  }
  return nl;
}

int launch_fits(const Dims& D, float scale, float ridge_w, float ridge_v, float eps_w, float b_min,
                float b_max, const bf16* Q, const float* C_k, const float* z, const float* m,
                const float* Y, const FitBufs& B, float* beta, float* C_v, DevStatus* stt, cudaStream_t st,
                cudaEvent_t const* ev) {
  auto mark = [&](int s) {
    if (ev) cudaEventRecord(ev[s], st);
  };
  int nl = 0;
  const long long nt = (long long)D.n * D.t;
  // logits of the compact keys LC = scale Q C_k^T [n][t]: C_k enters as a bf16
  // triple, LC^T = C_k Q^T runs on the tensor cores and is stored transposed
  {
    const long long htd = (long long)D.H * D.t * D.d;
    bf16 *ck_h = B.ck3, *ck_m = B.ck3 + htd, *ck_l = B.ck3 + 2 * htd;
    nl += launch_split3(C_k, ck_h, ck_m, ck_l, htd, st);
    CUtensorMap mA, mA2, mA3, mB;
    if (!encode_bf16_map_3d(&mA, ck_h, D.d, D.t, D.H, 128) || !encode_bf16_map_3d(&mA2, ck_m, D.d, D.t, D.H, 128) ||
        !encode_bf16_map_3d(&mA3, ck_l, D.d, D.t, D.H, 128) || !encode_bf16_map_3d(&mB, Q, D.d, D.n, D.H, 128))
      return -1;
    if (launch_tc_gemm<128, kSplit3A>(mA, mB, mA2, mA, TcEpiStoreT{B.LC, nt, D.t, scale}, D.H, D.t, D.n, D.d, D.d,
                                      stt, st, 0, &mA3) != cudaSuccess)
      return -1;
    ++nl;
  }
  const long long cnt = (long long)D.H * nt;
  launch_chained(phi_kernel, stride_grid(cnt, 256, 16), 256, 0, st, B.LC, z, B.Phi, D.n, D.t, cnt);
  ++nl;
  if (D.t > D.n) {
    const int nd = fits_dual(D, ridge_w, ridge_v, eps_w, b_min, b_max, m, Y, B, beta, C_v, stt, st, ev);
    return nd < 0 ? -1 : nl + nd;
  }
  // beta system: Gram = Phi_C^T Phi_C.  Its condition number reaches ~1e6 on
  // long caches, beyond what a split-bf16 pair (~1e-5 relative per entry)
  // resolves within tolerance: the operand enters as a bf16 triple and the
  // tensor-core Gram keeps every product term down to 2^-24 (kSplit3S).
  const int ldn = (D.n + 7) / 8 * 8;
  const dim3 tgrid(cdiv(D.t, 32), cdiv(ldn, 32), D.H);
  launch_chained(transpose_split3_kernel, tgrid, 256, 0, st, B.Phi, D.n, D.t, B.PT_hi, B.PT_mid, B.PT_lo, ldn);
  if (gram3_tc(D.H, D.t, ldn, B.PT_hi, B.PT_mid, B.PT_lo, B.Gram, stt, st) < 0) return -1;
  nl += 2;
  launch_chained(mass_rhs_kernel, dim3(cdiv(D.t, 32), D.H), 1024, 0, st, B.Phi, m, B.rhs, D.n, D.t);
  ++nl;
  mark(8);
  const int nb = launch_chol(D.H, D.t, B.Gram, B.Linv, B.rhs, B.Z, B.wsol, 1, D.t, ridge_w, B.ctrip, stt, st);
  if (nb < 0) return -1;
  nl += nb;
  const int nrf = refine_beta(D, ridge_w, m, B, stt, st);
  if (nrf < 0) return -1;
  nl += nrf;
  const long long ht = (long long)D.H * D.t;
  launch_chained(beta_kernel, cdiv(ht, 256), 256, 0, st, B.wsol, beta, ht, eps_w, b_min, b_max);
  ++nl;
  // value system: P^ over the compact keys with the fitted bias; its Gram and
  // P^T Y on the tensor cores from transposed split-bf16 operands
  mark(9);
  launch_chained(softmax_bias_kernel, dim3(cdiv(D.n, 8), D.H), 256, 0, st, B.LC, beta, B.Phi, D.n, D.t);
  ++nl;
  launch_chained(transpose_split_kernel, tgrid, 256, 0, st, B.Phi, D.n, D.t, B.PT_hi, B.PT_lo, ldn);
  launch_chained(transpose_split_kernel, dim3(cdiv(D.d, 32), cdiv(ldn, 32), D.H), 256, 0, st, Y, D.n, D.d, B.YT_hi, B.YT_lo,
                                                                                    ldn);
  nl += 2;
  if (gram_tc(D.H, D.t, D.t, ldn, B.PT_hi, B.PT_lo, B.PT_hi, B.PT_lo, B.Gram, D.t, stt, st) < 0) return -1;
  // R = P^T Y
  const long long td = (long long)D.t * D.d;
  if (gram_tc(D.H, D.t, D.d, ldn, B.PT_hi, B.PT_lo, B.YT_hi, B.YT_lo, B.R, D.d, stt, st) < 0) return -1;
  nl += 2;
  mark(10);
  const int nv = launch_chol(D.H, D.t, B.Gram, B.Linv, B.R, B.Z, C_v, D.d, td, ridge_v, B.ctrip, stt, st);
  return nv < 0 ? -1 : nl + nv;
}

// NaN or Inf in any of three arrays, one after another in the grid's stride
__global__ void check_finite_kernel(const float* x, long long nx, const float* y, long long ny, const float* z,
                                    long long nz, DevStatus* stt) {
  chain_wait();
  bool bad = false;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  for (long long k = i; k < nx; k += step) bad |= !isfinite(x[k]);
  for (long long k = i; k < ny; k += step) bad |= !isfinite(y[k]);
  for (long long k = i; k < nz; k += step) bad |= !isfinite(z[k]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) set_status(stt, ARCKV_ERR_NONFINITE);
}

int launch_check_finite(const float* x, long long nx, const float* y, long long ny, const float* z, long long nz,
                        DevStatus* stt, cudaStream_t st) {
  launch_chained(check_finite_kernel, stride_grid(std::max(nx, std::max(ny, nz)), 256, 8), 256, 0, st, x, nx, y, ny, z, nz,
                 stt);
  return 1;
}

}  // namespace arckv
