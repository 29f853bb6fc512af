// Cluster Cholesky solver of the fp32 normal systems (App. A.9, t <= n):
// (Gram + lam I) X = B for every head in one launch, lam = ridge trace / t.
//
// One cluster of kCL CTAs per head; the matrix, its factor and the right-hand
// sides live in global memory (L2-resident at these sizes) and are read with
// ld.global.cg, so that no CTA sees a stale L1 line of another CTA's writes.
// Right-looking over 64-wide block columns, forward substitution fused into
// the trailing updates.  Step k:
//   trsm    L_ik = A_ik Linv_kk^T (i > k) and Y_k = Linv_kk B_k, SIMT fp32; each
//           64 x 64 result also goes out as a bf16 triple in the swizzled layout
//           of an MMA operand (its `trip` slot), so that the split is done once;
//   update  A_ij -= L_ik L_jk^T (k < j <= i) and B_i -= L_ik Y_k in tcgen05 units
//           of two tiles of one block row,
//             D [128 x 64] = [X_1; X_2] L_ik^T,  X = L_jk or Y_k^T,
//           hh + hm + mh + hl + lh + mm per 16-wide K step (fp32-grade).
// The chain diagonal update -> factor (chol.cuh) -> Linv is what bounds a
// system of few blocks: the CTA that owns block k + 1 forms L_{k+1,k}, updates
// the diagonal block from its own registers and TMEM and factors it in shared
// memory while the others go on with the panel and the units; it waits for
// nobody in between.  A unit costs a CTA little more than its read-modify-
// write: operands arrive by bulk copies two units ahead, the MMAs of the next unit
// run under this one's, and the old values come in under its own.  (Reductions at
// L2 would flush subnormal values, and save 8 us of the two solves of 8 heads at t
// = 819.)  Units are dealt in a fixed order, the first kHeadStart rounds to the
// CTAs that do not factor.
//
// Then the back substitution X_k = Linv_kk^T (Y_k + Z_k), Z_i -= L_ki^T X_k:
// tcgen05 units for up to 128 right-hand sides; with one, mat-vecs whose
// blocks are dealt over the cluster, X_k broadcast through distributed shared
// memory.
//
// Eight heads on a GB300, one right-hand side / 128: 0.28 / 0.34 ms at t = 819,
// 0.77 / 0.98 ms at t = 1638; 0.67 / 0.81 and 1.88 / 2.09 ms before, with the
// split redone in every unit, 4 (8) CTAs a head and a 40 K cycle factor.  At t =
// 819 a step is its owner's chain, 36 K cycles: L_{k+1,k} 8.5, diagonal update
// 5, factor and inverse 21.
#include <cooperative_groups.h>
#include <map>
#include <mutex>

#include "chol.cuh"
#include "tc.cuh"

namespace arckv {

// defined in tc_host.cu
cudaError_t set_dyn_smem(const void* kern, int bytes);

// Byte offset of element (r, l) of a 64 x 64 bf16 operand block: row r (128
// bytes) with its 16-byte chunks permuted by r % 8 (128-byte swizzle, K-major).
__device__ __forceinline__ int op_off(int r, int l) { return r * 128 + (((l >> 3) ^ (r & 7)) << 4) + ((l & 7) << 1); }

// Operand slots: 3 parts (h, m, l) of 64 x 64 bf16.  A stage holds two tiles'
// triples part by part (A: rows 0-63 tile 1, 64-127 tile 2) and the triple of L_ik (B).
constexpr int kOpPart = 64 * 128, kOpSlot = 3 * kOpPart;
constexpr int kStageA = 2 * kOpPart, kStageBytes = 3 * kStageA + kOpSlot;
constexpr int kCholSmem = 3 * kTileF<float> * 4 + 2 * kStageBytes + 1024;
// rounds of units that go to the other CTAs only: the owner's chain (about 15
// us) is as long as ten units
constexpr int kHeadStart = 10;

size_t chol_trip_bytes(int H, int t) { return (size_t)H * ((t + NB - 1) / NB + 2) * kOpSlot; }

// Eight fp32 values of operand row r, K elements 8 ch .. 8 ch + 7, as bf16
// triples in the three part tiles.
__device__ __forceinline__ void put_split3_chunk(uint8_t* h, uint8_t* m, uint8_t* l, int r, int ch,
                                                 const float (&x)[8]) {
  __align__(16) bf16 hh[8], mm[8], ll[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) split3_bf16(x[e], hh[e], mm[e], ll[e]);
  const int off = op_off(r, 8 * ch);
  *(uint4*)(h + off) = *(const uint4*)hh;
  *(uint4*)(m + off) = *(const uint4*)mm;
  *(uint4*)(l + off) = *(const uint4*)ll;
}

// This thread's 4 x 2 results of a 64 x 64 product as an operand block's
// triple at `dst` (global or shared): element (r, l) = acc of row r, column l,
// or with kT of row l, column r.
template <bool kT>
__device__ __forceinline__ void put_acc_triple(uint8_t* dst, int ry, int cx, const float (&acc)[kTP][kTQ]) {
  if (!kT) {
#pragma unroll
    for (int p = 0; p < kTP; ++p) {
      __nv_bfloat162 h, m, l;
      split3_bf16x2(acc[p][0], acc[p][1], h, m, l);
      uint8_t* d = dst + op_off(ry + p, cx);
      *(__nv_bfloat162*)d = h;
      *(__nv_bfloat162*)(d + kOpPart) = m;
      *(__nv_bfloat162*)(d + 2 * kOpPart) = l;
    }
  } else {
#pragma unroll
    for (int q = 0; q < kTQ; ++q) {
      __nv_bfloat162 h[2], m[2], l[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) split3_bf16x2(acc[2 * e][q], acc[2 * e + 1][q], h[e], m[e], l[e]);
      uint8_t* d = dst + op_off(cx + q, ry);
      *(uint2*)d = *(const uint2*)h;
      *(uint2*)(d + kOpPart) = *(const uint2*)m;
      *(uint2*)(d + 2 * kOpPart) = *(const uint2*)l;
    }
  }
}

template <int kCL>
__global__ void __cluster_dims__(kCL, 1, 1) __launch_bounds__(kCT, 1)
    chol_tc_kernel(float* A, float* Linv, float* B, float* Z, float* X, uint8_t* trip, int t, int nrhs, int ldb,
                   long long bbs, float ridge, float tdiv, DevStatus* stt) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ float red[kCT / 32];
  __shared__ int bad, tc_abort;
  __shared__ uint64_t fullb[2], accb[2];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(16) float xs[3][NB];   // X_k of the single-right-hand-side back substitution
  const uint32_t s0 = tc::smem_u32(smraw);
  uint8_t* stage = smraw + (((s0 + 1023u) & ~1023u) - s0);   // two operand stages, 1024-byte aligned
  float* tiles = (float*)(stage + 2 * kStageBytes);
  Tile<float> S1 = (Tile<float>)tiles;
  Tile<float> S2 = (Tile<float>)(tiles + kTileF<float>);
  Tile<float> S3 = (Tile<float>)(tiles + 2 * kTileF<float>);
  const int head = blockIdx.x / kCL, rank = (int)cluster_rank(), tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int nblk = (t + NB - 1) / NB, nct = (nrhs + NB - 1) / NB;
  float* Ab = A + (long long)head * t * t;
  float* Lb = Linv + (long long)head * nblk * NB * NB;
  float* Bb = B + (long long)head * bbs;
  float* Zb = Z + (long long)head * bbs;
  float* Xb = X + (long long)head * bbs;
  uint8_t* tb = trip + (long long)head * (nblk + 2) * kOpSlot;
  const int ry = tile_ry(), cx = tile_cx();
  // this thread's slice of D: rows (TMEM lanes) dq * 32 + lane, columns 16 dg .. 16 dg + 15
  const int dq = warp & 3, dg = warp >> 2;
  volatile int* abp = &tc_abort;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&fullb[i], 1);
      tc::mbar_init(&accb[i], 1);
    }
    tc_abort = 0;
    bad = 0;
    tc::mbar_fence_init();
  }
  chain_wait();
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 128);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  // operand loads (full barriers) and MMA groups (accumulator barriers) of this
  // CTA are numbered; number q uses buffer q & 1 in its (q / 2)-th phase
  int ql = 0, qm = 0;      // next unit's load / MMA group (the same in all threads)
  int issued = 0;          // thread 0: loads issued
  auto release = [&]() {
    if (tid == 0) {   // copies still in flight (only after a wait gave up) land first
      volatile int never = 0;
      for (int q = issued > 2 ? issued - 2 : 0; q < issued; ++q) tc::mbar_wait(&fullb[q & 1], (q >> 1) & 1, &never, stt);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
      tc::fence_after_sync();
      tc::tmem_dealloc(tmem, 128);
    }
  };
  // D [128 x 64] = A B^T of the triples at a (parts pa apart) and b (parts pb
  // apart), issued by one thread into accumulator q & 1
  auto issue_mma = [&](const uint8_t* a, int pa, const uint8_t* b, int pb, int q) {
    constexpr uint32_t idesc = tc::idesc_bf16_f32(64);
    const uint32_t a0 = tc::smem_u32(a), b0 = tc::smem_u32(b), d = tmem + (uint32_t)((q & 1) * 64);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint32_t o = ks * 32;
      const uint64_t ah = tc::sdesc_k128(a0 + o), am = tc::sdesc_k128(a0 + pa + o), al = tc::sdesc_k128(a0 + 2 * pa + o);
      const uint64_t bh = tc::sdesc_k128(b0 + o), bm = tc::sdesc_k128(b0 + pb + o), bl = tc::sdesc_k128(b0 + 2 * pb + o);
      tc::mma_f16(d, ah, bh, idesc, ks > 0 ? 1u : 0u);
      tc::mma_f16(d, ah, bm, idesc, 1u);
      tc::mma_f16(d, am, bh, idesc, 1u);
      tc::mma_f16(d, ah, bl, idesc, 1u);
      tc::mma_f16(d, al, bh, idesc, 1u);
      tc::mma_f16(d, am, bm, idesc, 1u);
    }
    tc::mma_commit(&accb[q & 1]);
  };
  auto wait_acc = [&]() -> bool {   // all threads; the group becomes the last one read
    const bool ok = tc::mbar_wait(&accb[qm & 1], (qm >> 1) & 1, abp, stt);
    tc::fence_after_sync();
    return ok;
  };
  auto ld_slice = [&](float (&v)[16]) {
    __syncwarp();
    tc::tmem_ld16(tmem + ((uint32_t)(dq * 32) << 16) + (uint32_t)((qm & 1) * 64 + dg * 16), v);
  };

  // lam = ridge * trace / t (every CTA forms it; the trace precedes all writes)
  float tr = 0.f;
  for (int r = tid; r < t; r += kCT) tr += __ldcg(Ab + (long long)r * t + r);
  tr = warp_sum_r(tr);
  if (lane == 0) red[warp] = tr;
  __syncthreads();
  if (tid < 32) {
    float v = tid < kCT / 32 ? red[tid] : 0.f;
    v = warp_sum_r(v);
    if (tid == 0) red[0] = v;
  }
  __syncthreads();
  const float trace = red[0];
  const float lam = ridge * trace / tdiv;
  if (rank == 0 && tid == 0 && !isfinite(trace)) set_status(stt, ARCKV_ERR_NONFINITE);
  for (long long e = (long long)rank * kCT + tid; e < (long long)t * ldb; e += (long long)kCL * kCT) Zb[e] = 0.f;
  cluster_sync_all();   // everyone has read the unmodified diagonal for the trace
  if (rank == 0) {
    load_diag(S1, Ab, t, 0, min(NB, t), lam);
    factor_diag<float>(Ab, Lb, t, 0, S1, S2, S3, &bad);
  }
  cluster_sync_all();

  // Units of step k with m trailing blocks, row by row; row ii's tiles are its
  // syrk tiles j = k+1 .. k+1+ii (the diagonal tile of row 0 is its owner's)
  // and then the nct rhs tiles, two per unit.
  auto row_len = [&](int ii) { return (ii > 0 ? ii + 1 : 0) + nct; };
  // a cursor over the rows: units are visited in ascending order
  struct Cursor {
    int ii = 0, first = 0;   // row, its first unit
  };
  auto seek = [&](Cursor& c, int x) -> int {   // unit x's first tile in its row
    for (int u; x >= c.first + (u = (row_len(c.ii) + 1) / 2); ++c.ii) c.first += u;
    return 2 * (x - c.first);
  };
  Cursor lcur;   // thread 0: of the operand loads
  auto load_unit = [&](int k, int x, int q) {   // thread 0: the operands of unit x into stage q & 1
    const int e0 = seek(lcur, x), ii = lcur.ii, len = row_len(ii), ns = ii > 0 ? ii + 1 : 0;
    uint8_t* st = stage + (q & 1) * kStageBytes;
    uint64_t* bar = &fullb[q & 1];
    const int two = e0 + 1 < len ? 2 : 1;
    tc::mbar_arrive_expect_tx(bar, (uint32_t)((1 + two) * kOpSlot));
    tc::bulk_load(st + 3 * kStageA, tb + (long long)(k + 1 + ii) * kOpSlot, kOpSlot, bar);
    for (int h = 0; h < two; ++h) {
      const int e = e0 + h;
      const uint8_t* src = tb + (long long)(e < ns ? k + 1 + e : nblk + e - ns) * kOpSlot;
#pragma unroll
      for (int p = 0; p < 3; ++p) tc::bulk_load(st + p * kStageA + h * kOpPart, src + p * kOpPart, kOpPart, bar);
    }
    ++issued;
  };
  // a triple staged in shared memory to its slot (thread 0, after a barrier)
  auto store_slot = [&](int slot, const uint8_t* src) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                     (uint64_t)(tb + (long long)slot * kOpSlot)),
                 "r"(tc::smem_u32(src)), "r"(kOpSlot)
                 : "memory");
    tc::bulk_commit();
  };

  for (int k = 0; k < nblk; ++k) {
    const int m = nblk - k - 1, k0 = k * NB, kb = min(NB, t - k0);
    const float* Lk = Lb + (long long)k * NB * NB;
    const int own = (k + 1) % kCL;
    const bool owner = m > 0 && rank == own;
    // position among the CTAs that share the panel (all of them in the last step)
    const int pos = m > 0 ? (rank - own - 1 + kCL) % kCL : rank, npos = m > 0 ? kCL - 1 : kCL;
    float acc[kTP][kTQ];
    if (owner) {
      // L_{k+1,k}, then the diagonal block k + 1: its update, factor and inverse
      const int i0 = k0 + NB, rb = min(NB, t - i0);
      float old[16];   // A_{k+1,k+1}[n][r] of this thread's slice of D (rows 64.. of D are not used)
      const int r = (dq & 1) * 32 + lane;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int n = 16 * dg + c;
        old[c] = (dq < 2 && n < rb && r <= n) ? __ldcg(Ab + (long long)(i0 + n) * t + i0 + r) : 0.f;
      }
      ld_tiles(S1, Ab, t, i0, k0, rb, NB, true,                  // S1[l][r] = A_ik[r][l]
               S2, Lk, (long long)NB, 0, 0, NB, NB, true);       // S2[l][c] = Linv[c][l]
      __syncthreads();
      mm64(S1, S2, acc);
      uint8_t* st = stage;
      put_acc_triple<false>(st, ry, cx, acc);
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after_sync();
        issue_mma(st, kOpPart, st, kOpPart, qm);   // rows 64.. of A: whatever follows, unused
        store_slot(k + 1, st);
      }
      st_acc(Ab + (long long)(i0 + ry) * t + k0 + cx, t, rb - ry, NB, acc);   // L_{k+1,k}: read after the factorisation
      const bool ok = wait_acc();
      float v[16];
      ld_slice(v);
      if (dq < 2) {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int n = 16 * dg + c;
          float a = n == r ? 1.f : 0.f;
          if (n < rb && r <= n) a = (ok ? old[c] - v[c] : old[c]) + (n == r ? lam : 0.f);
          S1[n][r] = a;
        }
      }
      tc::fence_before_sync();
      ++qm;
      if (tid == 0) tc::bulk_wait_all();   // the slot is written
      cluster_arrive();
      factor_diag<float>(Ab, Lb, t, k + 1, S1, S2, S3, &bad);
      cluster_wait();
    } else {
      // panel tiles x = 1 .. m-1 (block rows k+1+x; x = 0 is the owner's) and the nct tiles of Y_k
      const int x0 = m > 0 ? 1 : 0, nx = m + nct;
      int x = x0 + pos;
      if (x < nx) {
        ld_tile(S2, Lk, (long long)NB, 0, 0, NB, NB, true);   // S2[l][c] = Linv[c][l]
        TileRegs<float> f;
        auto fetch = [&](int y) {
          if (y < m) {
            const int i0 = (k + 1 + y) * NB;
            tile_fetch(f, (const float*)Ab, (long long)t, i0, k0, min(NB, t - i0), NB, true);
          } else {
            const int c0 = (y - m) * NB;
            tile_fetch(f, (const float*)Bb, (long long)ldb, k0, c0, kb, min(NB, nrhs - c0), false);
          }
        };
        fetch(x);
        int buf = 0;
        for (; x < nx; x += npos) {
          tile_put(S1, f);
          __syncthreads();
          if (x + npos < nx) fetch(x + npos);   // in flight under this tile's product
          uint8_t* st = stage + (buf ^= 1) * kOpSlot;   // its triple goes through two staging buffers
          if (x < m) {
            const int i0 = (k + 1 + x) * NB;
            mm64(S1, S2, acc);
            put_acc_triple<false>(st, ry, cx, acc);
            st_acc(Ab + (long long)(i0 + ry) * t + k0 + cx, t, min(NB, t - i0) - ry, NB, acc);
          } else {
            const int c0 = (x - m) * NB;
            mm64(S2, S1, acc);   // Y[r][c] = sum_l Linv[r][l] B[l][c]
            put_acc_triple<true>(st, ry, cx, acc);
            st_acc(Bb + (long long)(k0 + ry) * ldb + c0 + cx, ldb, kb - ry, min(NB, nrhs - c0) - cx, acc);
          }
          tc::fence_proxy_async_smem();
          __syncthreads();
          if (tid == 0) {
            store_slot(x < m ? k + 1 + x : nblk + x - m, st);
            tc::bulk_wait_read<1>();   // the other buffer is free for the next tile (a barrier follows)
          }
        }
        if (tid == 0) tc::bulk_wait_all();
        __syncwarp();
      }
      cluster_sync_all();
    }
    if (m == 0) break;
    // trailing update: the units dealt to this CTA
    // (row 0: ceil(nct / 2); rows ii >= 1: floor((ii + 2 + nct) / 2), and sum_{j<=x} floor(j / 2) = floor(x^2 / 4))
    const int nu = (nct + 1) / 2 + (m + 1 + nct) * (m + 1 + nct) / 4 - (2 + nct) * (2 + nct) / 4;
    auto unit = [&](int j) {
      if (owner) return kHeadStart * (kCL - 1) + j * kCL + kCL - 1;
      return j < kHeadStart ? j * (kCL - 1) + pos : kHeadStart * (kCL - 1) + (j - kHeadStart) * kCL + pos;
    };
    auto start_mma = [&](int q, int qa) {   // thread 0: unit's operands -> accumulator
      if (!tc::mbar_wait(&fullb[q & 1], (q >> 1) & 1, abp, stt)) return;
      tc::fence_after_sync();
      const uint8_t* st = stage + (q & 1) * kStageBytes;
      issue_mma(st, kStageA, st + 3 * kStageA, kOpPart, qa);
    };
    int x = unit(0);
    if (tid == 0) {
      asm volatile("fence.proxy.async;" ::: "memory");
      lcur = Cursor();
      if (x < nu) load_unit(k, x, ql);
      if (unit(1) < nu) load_unit(k, unit(1), ql + 1);
      if (x < nu) start_mma(ql, qm);
    }
    Cursor cur;
    for (int j = 0; x < nu; ++j) {
      const int e0 = seek(cur, x), ii = cur.ii, len = row_len(ii), ns = ii > 0 ? ii + 1 : 0;
      const int i0 = (k + 1 + ii) * NB, e = e0 + (dq >> 1), r = (dq & 1) * 32 + lane;
      float* dst;   // A_ij[n][r] or B_i[n][c0 + r], n = 16 dg ..
      long long ld;
      bool col_ok;
      if (e < ns) {
        const int j0 = (k + 1 + e) * NB;
        dst = Ab + (long long)(i0 + 16 * dg) * t + j0 + r;
        ld = t;
        col_ok = j0 + r < t;
      } else {
        const int c0 = (e - ns) * NB;
        dst = Bb + (long long)(i0 + 16 * dg) * ldb + c0 + r;
        ld = ldb;
        col_ok = c0 + r < nrhs;
      }
      const int nok = (e < len && col_ok) ? min(16, t - i0 - 16 * dg) : 0;   // rows of this slice inside the matrix
      float old[16];   // in flight under the unit's MMAs
#pragma unroll
      for (int c = 0; c < 16; ++c) old[c] = c < nok ? __ldcg(dst + c * ld) : 0.f;
      const bool ok = wait_acc();
      const int xn = unit(j + 1);
      if (tid == 0) {
        // this unit's MMAs have read its stage; the next unit's accumulator was drained before the last barrier
        if (unit(j + 2) < nu) load_unit(k, unit(j + 2), ql + 2);
        if (xn < nu) start_mma(ql + 1, qm + 1);
      }
      float v[16];
      ld_slice(v);
      if (ok) {
#pragma unroll
        for (int c = 0; c < 16; ++c)
          if (c < nok) dst[c * ld] = old[c] - v[c];
      }
      tc::fence_before_sync();
      __syncthreads();
      ++ql;
      ++qm;
      x = xn;
    }
    cluster_sync_all();
  }

  if (nrhs == 1) {
    // Block j of Z is kept by rank j % kCL.  Rank k % kCL forms X_k and
    // broadcasts it; then the rank of block k - 1 updates that block from a tile
    // of L fetched ahead, forms X_{k-1} and arrives, and only then do the ranks
    // update their other blocks by X_k.  A rank may thus read X_k while X_{k-1}
    // and X_{k-2} are written: three buffers.
    float* vs = (float*)stage;        // Y_k + Z_k [64]
    float* zs = vs + NB;              // [ceil(nblk / kCL)][64]
    cg::cluster_group cl = cg::this_cluster();
    for (int e = tid; e < ((nblk + kCL - 1) / kCL) * NB; e += kCT) zs[e] = 0.f;
    __syncthreads();
    auto form_x = [&](int k) {   // X_k[c] = sum_l Linv_k[l][c] v[l]: eight threads per column, l = part, part + 8, ...
      const int k0 = k * NB, kb = min(NB, t - k0), c = tid >> 3, part = tid & 7;
      const float* Li = Lb + (long long)k * NB * NB;
      float li[8];
#pragma unroll
      for (int l = 0; l < 8; ++l) li[l] = __ldcg(Li + (part + 8 * l) * NB + c);
      if (tid < NB) vs[tid] = tid < kb ? __ldcg(Bb + (long long)(k0 + tid) * ldb) + zs[(k / kCL) * NB + tid] : 0.f;
      __syncthreads();
      float a = 0.f;
#pragma unroll
      for (int l = 0; l < 8; ++l) a = fmaf(li[l], vs[part + 8 * l], a);
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      if (part == 0) {
        if (c < kb) Xb[(long long)(k0 + c) * ldb] = a;
        else a = 0.f;
      }
      a = __shfl_sync(0xffffffffu, a, lane & 24);
      for (int rk = part; rk < kCL; rk += 8) cl.map_shared_rank(&xs[0][0], rk)[(k % 3) * NB + c] = a;
    };
    if (rank == (nblk - 1) % kCL) form_x(nblk - 1);
    cluster_arrive();
    for (int k = nblk - 1; k >= 1; --k) {
      const int k0 = k * NB, kb = min(NB, t - k0);
      const bool next = rank == (k - 1) % kCL;
      if (next) ld_tile(S1, (const float*)Ab, (long long)t, k0, k0 - NB, kb, NB, false);   // L_k,k-1
      cluster_wait();
      const float* xk = xs[k % 3];
      if (next) {
        __syncthreads();
        if (tid < NB) {   // Z_j -= L_kj^T X_k
          float a = 0.f;
#pragma unroll 16
          for (int l = 0; l < kb; ++l) a = fmaf(S1[l][tid], xk[l], a);
          zs[((k - 1) / kCL) * NB + tid] -= a;
        }
        __syncthreads();
        form_x(k - 1);
      }
      cluster_arrive();
      // this rank's other blocks j < k - 1, 64 threads each
      for (int j = rank + kCL * (tid >> 6); j < k - 1; j += kCL * (kCT / NB)) {
        const int c = tid & 63;
        const float* col = Ab + (long long)k0 * t + j * NB + c;
        float a = 0.f;
#pragma unroll 16
        for (int l = 0; l < kb; ++l) a = fmaf(__ldcg(col + (long long)l * t), xk[l], a);
        zs[(j / kCL) * NB + c] -= a;
      }
      __syncthreads();
    }
    cluster_wait();   // nobody leaves before the last write to its xs
    if (tid == 0 && bad) set_status(stt, ARCKV_ERR_NOT_SPD);
    release();
    return;
  }

  // Back substitution on the tensor cores (nrhs <= 128): rows m of D are the
  // right-hand-side columns, its columns n the rows of the block
  //   Z_i -= L_ki^T X_k:     D = X_k^T L_ki,          Z_i[n][m] -= D[m][n]
  //   X_k = Linv^T (Y + Z):  D = (Y_k + Z_k)^T Linv,  X_k[n][m] = D[m][n]
  // Serial over the blocks: the owner of block k - 1 stages the two operands that
  // do not depend on X_k while it waits for the others, takes X_k as the triple
  // its owner left in a slot (alternate slots), adds the update to Y + Z on the
  // way from TMEM to the second product's operand, and leaves X_{k-1} as a triple
  // in turn; the other CTAs apply X_k to their blocks of Z.
  uint8_t* const SA = stage;                               // X_k^T
  uint8_t* const SB = stage + 3 * kStageA;                 // L_ki
  uint8_t* const SA2 = stage + kStageBytes;                // (Y + Z)^T
  uint8_t* const SB2 = stage + kStageBytes + 3 * kStageA;  // Linv
  constexpr int kXSlot = 3 * kStageA;                      // triple of a 128 x 64 operand
  static_assert(2 * kXSlot <= 4 * kOpSlot, "two X slots in the operand slots of two blocks");
  const int mrow = dq * 32 + lane, ncol = dg * 16;
  // operand rows r < 64 of a triple from a column-major source: element (r, l) =
  // G[l * ld + r] for l < kvalid, zero elsewhere; consecutive threads take consecutive r
  auto stage_cols = [&](uint8_t* h, const float* G, long long ld, int kvalid) {
    const int r = tid & 63, ch = tid >> 6;
    float xv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) xv[q] = 8 * ch + q < kvalid ? __ldcg(G + (long long)(8 * ch + q) * ld + r) : 0.f;
    put_split3_chunk(h, h + kOpPart, h + 2 * kOpPart, r, ch, xv);
  };
  // this thread's 16 values of row mrow as operand elements l = ncol .. of a 128-row triple
  auto put_row = [&](uint8_t* h, const float (&x)[16]) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      float xv[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) xv[q] = x[8 * half + q];
      put_split3_chunk(h, h + kStageA, h + 2 * kStageA, mrow, ncol / 8 + half, xv);
    }
  };
  auto run_mma = [&](const uint8_t* A_, const uint8_t* B_, bool wait_x) -> bool {
    tc::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      if (!wait_x || tc::mbar_wait(&fullb[ql & 1], (ql >> 1) & 1, abp, stt)) {
        tc::fence_after_sync();
        issue_mma(A_, kStageA, B_, kOpPart, qm);
      }
    }
    return wait_acc();
  };
  auto mma_done = [&]() {   // the accumulator and its operands are free
    tc::fence_before_sync();
    __syncthreads();
    ++qm;
  };
  // X_k from y = Y_k + Z_k (this thread's 16 rows of column mrow) with Linv_k in SB2
  auto form_x = [&](int k, const float (&y)[16]) {
    const int k0 = k * NB, kb = min(NB, t - k0);
    put_row(SA2, y);
    const bool ok = run_mma(SA2, SB2, false);
    float v[16];
    ld_slice(v);
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = ok && ncol + c < kb ? v[c] : 0.f;
    put_row(tb + (k & 1) * kXSlot, v);
    if (ok && mrow < nrhs) {
      float* dst = Xb + (long long)(k0 + ncol) * ldb + mrow;
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (ncol + c < kb) dst[(long long)c * ldb] = v[c];
    }
    asm volatile("fence.proxy.async;" ::: "memory");   // the slot, for the other CTAs' bulk copies
    mma_done();
  };
  auto load_yz = [&](int k, float (&y)[16], float (&z)[16]) {
    const int k0 = k * NB, kb = min(NB, t - k0);
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const bool in = mrow < nrhs && ncol + c < kb;
      const long long o = (long long)(k0 + ncol + c) * ldb + mrow;
      y[c] = in ? __ldcg(Bb + o) : 0.f;
      z[c] = in ? __ldcg(Zb + o) : 0.f;
    }
  };
  if (rank == (nblk - 1) % kCL) {
    stage_cols(SB2, Lb + (long long)(nblk - 1) * NB * NB, NB, NB);
    float y[16], z[16];
    load_yz(nblk - 1, y, z);
#pragma unroll
    for (int c = 0; c < 16; ++c) y[c] += z[c];
    form_x(nblk - 1, y);
  }
  cluster_arrive();
  for (int k = nblk - 1; k >= 1; --k) {
    const int k0 = k * NB, kb = min(NB, t - k0), own = (k - 1) % kCL;
    const bool owner = rank == own;
    // this CTA's first block of Z: k - 1 for its owner, the others share i < k - 1
    int i = owner ? k - 1 : (rank - own - 1 + kCL) % kCL;
    const bool any = owner || i < k - 1;
    if (any) stage_cols(SB, Ab + (long long)k0 * t + i * NB, t, kb);
    if (owner) stage_cols(SB2, Lb + (long long)(k - 1) * NB * NB, NB, NB);
    cluster_wait();
    if (any && tid == 0) {
      asm volatile("fence.proxy.async;" ::: "memory");
      tc::mbar_arrive_expect_tx(&fullb[ql & 1], kXSlot);
      tc::bulk_load(SA, tb + (k & 1) * kXSlot, kXSlot, &fullb[ql & 1]);
      ++issued;
    }
    if (owner) {
      float y[16], z[16], v[16];
      load_yz(k - 1, y, z);
      const bool ok = run_mma(SA, SB, true);
      ld_slice(v);
#pragma unroll
      for (int c = 0; c < 16; ++c) y[c] += ok ? z[c] - v[c] : z[c];
      mma_done();
      form_x(k - 1, y);
    } else {
      bool first = true;
      for (; i < k - 1; i += kCL - 1) {
        if (!first) stage_cols(SB, Ab + (long long)k0 * t + i * NB, t, kb);
        float* dst = Zb + (long long)(i * NB + ncol) * ldb + mrow;   // block i < k is full
        float v[16], old[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) old[c] = mrow < nrhs ? __ldcg(dst + (long long)c * ldb) : 0.f;
        const bool ok = run_mma(SA, SB, first);
        ld_slice(v);
        if (ok && mrow < nrhs) {
#pragma unroll
          for (int c = 0; c < 16; ++c) dst[(long long)c * ldb] = old[c] - v[c];
        }
        mma_done();
        first = false;
      }
    }
    if (any) ++ql;
    cluster_arrive();
  }
  cluster_wait();
  if (tid == 0 && bad) set_status(stt, ARCKV_ERR_NOT_SPD);
  release();
}

// Launch with clusters of kCL CTAs per head; false when the device cannot hold
// H of them at a time (clusters above 8 need a non-portable launch).
template <int kCL>
static bool chol_launch(int H, int t, float* Gram, float* Linv, float* B, float* Z, float* X, int nrhs, long long bbs,
                        float ridge, uint8_t* trip, DevStatus* stt, cudaStream_t st) {
  const void* kern = (const void*)chol_tc_kernel<kCL>;
  if (set_dyn_smem(kern, kCholSmem) != cudaSuccess) return false;
  if (kCL > 8) {
    // resident clusters of this device, asked once (the answer depends on its GPCs alone)
    static std::mutex mu;
    static std::map<int, int> resident;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> g(mu);
    auto it = resident.find(dev);
    if (it == resident.end()) {
      int n = 0;
      cudaLaunchConfig_t cfg{};
      cudaLaunchAttribute at{};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = kCL;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cfg.gridDim = dim3(kCL);
      cfg.blockDim = dim3(kCT);
      cfg.dynamicSmemBytes = kCholSmem;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
          cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      it = resident.emplace(dev, n).first;
    }
    if (it->second < H) return false;
  }
  launch_chained(chol_tc_kernel<kCL>, kCL * H, kCT, kCholSmem, st, Gram, Linv, B, Z, X, trip, t, nrhs, nrhs, bbs, ridge, (float)t,
                                                       stt);
  return true;
}

// CTAs per head: as many as the trailing updates keep busy -- 4 up to 4 blocks,
// 8 up to 8, above that 16 or 12 where the GPCs hold a cluster of that size
// for every head at once (8 heads: 12 on a GB300), else 8.
int launch_chol(int H, int t, float* Gram, float* Linv, float* B, float* Z, float* X, int nrhs, long long bbs,
                float ridge, uint8_t* trip, DevStatus* stt, cudaStream_t st) {
  const int nblk = (t + NB - 1) / NB;
  bool ok = false;
  if (nblk > 8) {
    ok = chol_launch<16>(H, t, Gram, Linv, B, Z, X, nrhs, bbs, ridge, trip, stt, st) ||
         chol_launch<12>(H, t, Gram, Linv, B, Z, X, nrhs, bbs, ridge, trip, stt, st);
  }
  if (!ok && nblk > 4) ok = chol_launch<8>(H, t, Gram, Linv, B, Z, X, nrhs, bbs, ridge, trip, stt, st);
  if (!ok) ok = chol_launch<4>(H, t, Gram, Linv, B, Z, X, nrhs, bbs, ridge, trip, stt, st);
  return ok ? 1 : -1;
}

}  // namespace arckv
