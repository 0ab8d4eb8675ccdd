// Batched dielectric factorisation eps = L D L^T (no pivoting) and the screened
// contraction W^c = b^T (eps^-1 - 1) b = y^T D^-1 y - b^T b with y = L^-1 b.
//
// eps(i xi) is real symmetric positive definite (Pi(i xi) is negative semidefinite), so
// there this is a Cholesky-type factorisation; eps(x + i eta) is complex SYMMETRIC (not
// Hermitian), so no conjugation appears anywhere. Without pivoting a zero pivot is
// possible in exact arithmetic only; it is detected (|d| below a floor) and reported
// through the status word, and the pivot is replaced by 1 so the batch stays finite.
//
// Storage after the factorisation (matrix [n][ldm], row-major):
//   strictly lower part  W = L D   (W_ij = L_ij d_j, j < i)
//   diagonal             d
//   strictly upper part  L^T       (A[j][i] = L_ij; scratch used by the trailing updates)
//
// Right-looking and blocked, by one CTA per matrix or as launches over all matrices (below):
//   * 64-wide panels, each factored as two 32-wide halves: the two 32 x 32 diagonal blocks in
//     shared memory, then every row below in one pass by one thread (solve against block 1,
//     apply block 1 to its block-2 columns, solve against block 2), storing W (lower) and L
//     (upper).
//   * the trailing lower triangle is updated with the rank-64 product W_panel L_panel^T, in
//     64 x 64 tiles (4 x 4 per thread); both operands are staged through shared memory by
//     cp.async in 32-deep chunks, double-buffered across chunks and tiles.
#include <cooperative_groups.h>

#include <algorithm>

#include "gwc_internal.h"
#include "ldlt_simt.cuh"

namespace gwc {

namespace {

template <typename S>
__global__ void __launch_bounds__(256) ldlt_kernel(S* __restrict__ mats, int n, int nrow, long long ldm, long long stride,
                                                    const int* __restrict__ active, unsigned* __restrict__ status) {
  const int f = blockIdx.x;
  if (active && !active[f]) return;
  S* A = mats + f * stride;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the panel scratch and the update stages alias (the phases alternate)
  const PanelSmem<S, kSimtThreads> ps(smem_raw);
  S* stages = reinterpret_cast<S*>(smem_raw);
  __shared__ int sing;
  if (threadIdx.x == 0) sing = 0;

  for (int k0 = 0; k0 < n; k0 += PW) {
    const int kb = min(PW, n - k0);
    factor_panel<S, kSimtThreads>(A, n, nrow, ldm, k0, ps, sing);
    // rank-kb trailing update of the lower triangle beyond the panel (and of appended rows)
    if (k0 + kb < n) update_region(A, nrow, ldm, k0 + kb, k0 + kb, n, k0, kb, stages);
  }
  __syncthreads();
  if (threadIdx.x == 0 && sing) atomicOr(status, kStatSingular);
}

// ---- the same factorisation over all SMs ------------------------------------------------------------
// The kernel above keeps a matrix on one SM, so a few large matrices leave the chip idle (8 of N_aux 1100 in FP64: 279 ms on 8 SMs).
// Per panel: the diagonal blocks (one CTA per matrix), the rows below (64 per CTA, the factored diagonal read back from the
// matrix), and the rank-64 update with one 64 x 64 trailing tile per CTA; the arithmetic of every element is the same.
// Measured in complex FP64: 8 matrices of N_aux 1100, 279 -> 24 ms (update 13.3 ms, of which 12.2 are FP64 multiply-adds at
// the card's rate; diagonal blocks 5.6 ms, rows 5.1 ms); a batch of 608 matrices of N_aux 200, 18.5 -> 11 ms. Which
// of the two: one_cta_factor.
template <typename S>
struct DiagOnlySmem {  // the part of PanelSmem the diagonal needs
  S (*lkk1)[NB + 1];
  S (*lkk2)[NB + 1];
  S (*w1s)[NB + 1];
  S (*l1s)[NB + 1];
  S* dinv1;
  S* dinv2;
  static constexpr size_t bytes() { return sizeof(S) * (4 * NB * (NB + 1) + 2 * NB); }
  __device__ explicit DiagOnlySmem(void* base) {
    S* p = reinterpret_cast<S*>(base);
    lkk1 = reinterpret_cast<S(*)[NB + 1]>(p);
    lkk2 = reinterpret_cast<S(*)[NB + 1]>(p + NB * (NB + 1));
    w1s = reinterpret_cast<S(*)[NB + 1]>(p + 2 * NB * (NB + 1));
    l1s = reinterpret_cast<S(*)[NB + 1]>(p + 3 * NB * (NB + 1));
    dinv1 = p + 4 * NB * (NB + 1);
    dinv2 = dinv1 + NB;
  }
};
constexpr int kRowThreads = 64, kDiagThreads = 128;

template <typename S>
__global__ void __launch_bounds__(kDiagThreads) ldlt_split_diag_kernel(S* __restrict__ mats, int n, long long ldm, long long stride, int k0,
                                                               const int* __restrict__ active, unsigned* __restrict__ status) {
  const int f = blockIdx.x;
  if (active && !active[f]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const DiagOnlySmem<S> ps(smem_raw);
  __shared__ int sing;
  if (threadIdx.x == 0) sing = 0;
  factor_panel_diag<S, kDiagThreads>(mats + f * stride, n, ldm, k0, ps, sing);
  __syncthreads();
  if (threadIdx.x == 0 && sing) atomicOr(status, kStatSingular);
}

template <typename S>
__global__ void __launch_bounds__(kRowThreads) ldlt_split_rows_kernel(S* __restrict__ mats, int n, int nrow, long long ldm,
                                                                       long long stride, int k0, const int* __restrict__ active) {
  const int f = blockIdx.y;
  if (active && !active[f]) return;
  S* A = mats + f * stride;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const PanelSmem<S, kRowThreads> ps(smem_raw);
  const int kb = min(PW, n - k0), kb1 = min(NB, kb), kb2 = kb - kb1, c2 = k0 + NB;
  for (int e = threadIdx.x; e < NB * NB; e += kRowThreads) {
    const int j = e / NB, i = e % NB;  // L_ij from the row j above the diagonal
    ps.lkk1[i][j] = (j < i && i < kb1) ? A[(long long)(k0 + j) * ldm + k0 + i] : szero<S>();
    ps.l1s[i][j] = (i < kb2) ? A[(long long)(k0 + j) * ldm + c2 + i] : szero<S>();
    ps.lkk2[i][j] = (j < i && i < kb2) ? A[(long long)(c2 + j) * ldm + c2 + i] : szero<S>();
  }
  for (int j = threadIdx.x; j < kb; j += kRowThreads) (j < NB ? ps.dinv1 : ps.dinv2 - NB)[j] = sinv(A[(long long)(k0 + j) * ldm + k0 + j]);
  __syncthreads();
  const int i = k0 + kb + kRowThreads * blockIdx.x + threadIdx.x;
  factor_panel_rows<S, kRowThreads>(A, n, nrow, ldm, k0, ps, i, nrow);  // one row per thread
}

// tile t of the trailing lower part [R0, nrow) x [R0, n): row tile tI holds column tiles 0 .. min(tI, last)
template <typename S>
__global__ void __launch_bounds__(256) ldlt_split_update_kernel(S* __restrict__ mats, int n, int nrow, long long ldm,
                                                                 long long stride, int k0, int n_tj,
                                                                 const int* __restrict__ active) {
  const int f = blockIdx.y;
  if (active && !active[f]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int t = blockIdx.x, tI = 0;
  while (t >= min(tI + 1, n_tj)) {
    t -= min(tI + 1, n_tj);
    ++tI;
  }
  const int R0 = k0 + PW, i0 = R0 + TT * tI, j0 = R0 + TT * t;
  update_region(mats + f * stride, min(nrow, i0 + TT), ldm, i0, j0, min(n, j0 + TT), k0, PW, reinterpret_cast<S*>(smem_raw));
}

template <typename S>
int run_ldlt_split(S* mats, int n, int nrow, long long ldm, long long stride, int F, const int* active, unsigned* status,
                   cudaStream_t s) {
  static bool attr = false;
  constexpr int dsm = (int)DiagOnlySmem<S>::bytes(), rsm = (int)PanelSmem<S, kRowThreads>::bytes(), usm = (int)FactorSmem<S>::bytes();
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_split_diag_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, dsm) != cudaSuccess ||
        cudaFuncSetAttribute(ldlt_split_rows_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, rsm) != cudaSuccess ||
        cudaFuncSetAttribute(ldlt_split_update_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, usm) != cudaSuccess)
      return -1;
    attr = true;
  }
  int launches = 0;
  for (int k0 = 0; k0 < n; k0 += PW) {
    const int R0 = k0 + std::min(PW, n - k0);
    ldlt_split_diag_kernel<S><<<F, kDiagThreads, dsm, s>>>(mats, n, ldm, stride, k0, active, status);
    ++launches;
    if (R0 < nrow) {
      ldlt_split_rows_kernel<S><<<dim3((nrow - R0 + kRowThreads - 1) / kRowThreads, F), kRowThreads, rsm, s>>>(mats, n, nrow, ldm,
                                                                                                               stride, k0, active);
      ++launches;
    }
    if (R0 < n) {
      const int n_ti = (nrow - R0 + TT - 1) / TT, n_tj = (n - R0 + TT - 1) / TT;
      int tiles = 0;
      for (int tI = 0; tI < n_ti; ++tI) tiles += std::min(tI + 1, n_tj);
      ldlt_split_update_kernel<S><<<dim3(tiles, F), 256, usm, s>>>(mats, n, nrow, ldm, stride, k0, n_tj, active);
      ++launches;
    }
    if (cudaPeekAtLastError() != cudaSuccess) return -1;
  }
  return launches;
}

// Forward substitution with the W storage, for a block of SR right-hand sides (in place):
//   y_i = b_i - sum_{l<i} W_il u_l,  u_l = y_l / d_l   (since L_il = W_il / d_l)
//   w_q = sum_i y_i^2 / d_i - |b_q|^2 = sum_i u_i^2 d_i - |b_q|^2.
// The right-hand-side buffer ends up holding u. Grid: (matrix f, RHS block). Per 64-row panel:
//   * update: acc = -W[panel rows][0 .. k0) U[0 .. k0)[block], a product in 32-deep chunks staged through
//     shared memory, 4 x 4 outputs per thread (rows strided by 16 so that a warp reads distinct rows);
//   * panel: the 64 x 64 diagonal block by four threads per right-hand side (strided partial sums of the
//     row, two shuffles), u_i = (b_i + acc_i - sum_{l<i} W_il u_l) / d_i, u_i^2 d_i summed in FP64.
constexpr int SB = 64;  // panel rows
constexpr int SR = 64;  // right-hand sides per CTA
constexpr int SK = 32;  // depth of the staged update chunks

template <typename S>
struct SolveSmem {
  // update phase: ls[SB][SK + 1], us[SK][SR + 1]; panel phase: acc (then u) [SB][SR + 1], wd [SB][SB + 1], dv [SB]
  static constexpr size_t upd = (size_t)SB * (SK + 1) + (size_t)SK * (SR + 1);
  static constexpr size_t pan = (size_t)SB * (SR + 1) + (size_t)SB * (SB + 1) + SB;
  static constexpr size_t elems = upd > pan ? upd : pan;
  static size_t bytes() { return elems * sizeof(S); }
};

template <typename S>
__global__ void __launch_bounds__(256) ldlt_solve_kernel(const S* __restrict__ mats, int n, long long ldm, long long stride,
                                                          S* __restrict__ rhs, int r, long long ldr, long long rhs_stride,
                                                          const double* __restrict__ bnorm2, double* __restrict__ w,
                                                          long long w_stride, const int* __restrict__ active) {
  const int f = blockIdx.x;
  if (active && !active[f]) return;
  const int q0 = blockIdx.y * SR;
  const int nq = min(SR, r - q0);
  const S* L = mats + f * stride;
  S* Y = rhs + f * rhs_stride + (long long)q0 * ldr;
  const int tid = threadIdx.x;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  S(*ls)[SK + 1] = reinterpret_cast<S(*)[SK + 1]>(smem_raw);
  S(*us)[SR + 1] = reinterpret_cast<S(*)[SR + 1]>(smem_raw + sizeof(S) * SB * (SK + 1));
  S(*acc_s)[SR + 1] = reinterpret_cast<S(*)[SR + 1]>(smem_raw);
  S(*wd)[SB + 1] = reinterpret_cast<S(*)[SB + 1]>(smem_raw + sizeof(S) * SB * (SR + 1));
  S* dv = reinterpret_cast<S*>(smem_raw + sizeof(S) * (SB * (SR + 1) + SB * (SB + 1)));

  const int tr = tid & 15, tc = tid >> 4;         // update: rows tr + 16 a, columns 4 tc + b
  const int cq = tid >> 2, cp = tid & 3;           // panel: right-hand side cq, quarter cp of each row sum
  double wr = 0.0, wi = 0.0;                       // sum u_i^2 d_i of right-hand side cq (kept by cp == 0)
  for (int k0 = 0; k0 < n; k0 += SB) {
    const int kb = min(SB, n - k0);
    S acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = szero<S>();
    for (int l0 = 0; l0 < k0; l0 += SK) {
      for (int e = tid; e < SB * SK; e += 256) {
        const int i = e / SK, l = e % SK;
        ls[i][l] = i < kb ? L[(long long)(k0 + i) * ldm + l0 + l] : szero<S>();
      }
      for (int e = tid; e < SR * SK; e += 256) {
        const int q = e / SK, l = e % SK;
        us[l][q] = q < nq ? Y[(long long)q * ldr + l0 + l] : szero<S>();
      }
      __syncthreads();
#pragma unroll 4
      for (int l = 0; l < SK; ++l) {
        S av[4], bv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) av[a] = ls[tr + 16 * a][l];
#pragma unroll
        for (int b = 0; b < 4; ++b) bv[b] = us[l][4 * tc + b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = sfnms(av[a], bv[b], acc[a][b]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc_s[tr + 16 * a][4 * tc + b] = acc[a][b];
    for (int e = tid; e < SB * SB; e += 256) {
      const int i = e / SB, l = e % SB;
      wd[i][l] = (i < kb && l < i) ? L[(long long)(k0 + i) * ldm + k0 + l] : szero<S>();
    }
    if (tid < SB) dv[tid] = tid < kb ? L[(long long)(k0 + tid) * ldm + k0 + tid] : sfrom<S>(1.0, 0.0);
    __syncthreads();
    // the panel's rows in order; the four threads of a right-hand side are consecutive lanes of one warp
    for (int i = 0; i < kb; ++i) {
      S part = szero<S>();
      for (int l = cp; l < i; l += 4) part = sadd(part, smul(wd[i][l], acc_s[l][cq]));
      part = sadd(part, shfl_xor_s(part, 1));
      part = sadd(part, shfl_xor_s(part, 2));
      if (cp == 0 && cq < nq) {
        const S v = ssub(sadd(Y[(long long)cq * ldr + k0 + i], acc_s[i][cq]), part);
        const S u = smul(v, sinv(dv[i]));
        acc_s[i][cq] = u;
        Y[(long long)cq * ldr + k0 + i] = u;
        const S t = smul(smul(u, u), dv[i]);
        wr += sre(t);
        wi += sim(t);
      }
      __syncwarp();
    }
    __syncthreads();
  }
  if (cp == 0 && cq < nq) {
    double* o = w + f * w_stride + (long long)(q0 + cq) * 2;
    o[0] = wr - bnorm2[(long long)f * r + q0 + cq];
    o[1] = wi;
  }
}

// The same substitution for few right-hand sides (r <= kFewRhs, the residue and screening calls): u and w exactly as above, with
// the sums over l in the same order. The kernel above keeps one CTA per matrix on n/64 serial panels and multiplies 64
// columns whatever r is, so at r = 6 .. 12 it waits on latency: 9.6 ms for 8 matrices of N_aux 2450. Here a cluster of C CTAs
// holds a matrix's rows (64-row blocks round robin, their running sums in shared memory) and goes right-looking:
//   solve   the owner of panel k takes its 64 x 64 diagonal block, a warp per right-hand side and two rows per lane (one
//           exchange per row, no barrier), and puts u into the shared memory of all C CTAs;
//   update  every CTA subtracts W[rows][panel] u from the rows it owns, W read once through L1.
// Measured: 8 complex FP32 matrices of N_aux 2450, r = 12, 9.65 -> 0.78 ms; 64 of 1100, r = 6, 2.43 -> 0.29 ms; 8 complex
// FP64 ones of 1100, 45 -> 2.3 ms. The chain of the n/64 panels bounds it (about 20 us each: 64 exchanges, the cluster
// barrier and the rows' loads). Beyond kFewRhs right-hand sides (the W table, CD-WAC) the kernel above fills the chip.
// (Which cluster, and where the kernel above stays: few_ctas.)
constexpr int kFewRhs = 32;
constexpr int kFewSmem = 200 * 1024;
constexpr int FQ = 4;  // right-hand sides per thread of the update

__device__ __forceinline__ float shfl_s(float v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ double shfl_s(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ float2 shfl_s(float2 v, int l) { return make_float2(shfl_s(v.x, l), shfl_s(v.y, l)); }
__device__ __forceinline__ double2 shfl_s(double2 v, int l) { return make_double2(shfl_s(v.x, l), shfl_s(v.y, l)); }

// products and reciprocals with the roundings of the kernel above written out for complex FP32 (the contractions there are the
// compiler's; here they decide whether the two agree bit by bit)
template <typename S> __device__ __forceinline__ S fmul(S a, S b) { return smul(a, b); }
template <> __device__ __forceinline__ float2 fmul<float2>(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}
template <typename S> __device__ __forceinline__ S finv(S a) { return sinv(a); }
template <> __device__ __forceinline__ float2 finv<float2>(float2 a) {
  const float d = __fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y));
  return make_float2(__fdiv_rn(a.x, d), __fdiv_rn(-a.y, d));
}

// elements of S: diagonal block, d, two u buffers, the sums of `blocks` row blocks; then C * r partial results (2 doubles each)
inline size_t few_elems(int blocks, int rp) { return (size_t)SB * (SB + 1) + SB + 2 * (size_t)SB * rp + (size_t)blocks * SB * rp; }

template <typename S, int QW>  // QW right-hand sides per warp: r <= 8 QW
__global__ void __launch_bounds__(256) ldlt_solve_few_kernel(const S* __restrict__ mats, int n, long long ldm, long long stride,
                                                              const S* __restrict__ rhs, int r, long long ldr,
                                                              long long rhs_stride, const double* __restrict__ bnorm2,
                                                              double* __restrict__ w, long long w_stride,
                                                              const int* __restrict__ active) {
  constexpr int PER = 16 / (int)sizeof(S);
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), f = blockIdx.x / C;
  if (active && !active[f]) return;  // the whole cluster
  const S* L = mats + f * stride;
  const S* Y = rhs + f * rhs_stride;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int np = (n + SB - 1) / SB, cnt = rank < np ? (np - rank + C - 1) / C : 0;  // panels; row blocks owned
  const int groups = (r + FQ - 1) / FQ, rp = groups * FQ;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  S* us = reinterpret_cast<S*>(smem_raw);            // [2][SB][rp]
  S* acc = us + 2 * SB * rp;                         // [cnt * SB][rp]
  S* wd = acc + (size_t)((np + C - 1) / C) * SB * rp;  // [SB][SB + 1]
  S* dv = wd + SB * (SB + 1);                        // [SB]
  double* part = reinterpret_cast<double*>(dv + SB);  // [C][r][2] (on rank 0)

  for (int e = tid; e < cnt * SB * rp; e += 256) acc[e] = szero<S>();
  auto load_diag = [&](int k) {
    const int k0 = k * SB, kb = min(SB, n - k0);
    for (int e = tid; e < SB * SB; e += 256) {
      const int i = e / SB, l = e % SB;
      if (i < kb && l < i) cp_async_elem<(int)sizeof(S)>(wd + i * (SB + 1) + l, L + (long long)(k0 + i) * ldm + k0 + l);
    }
    if (tid < kb) cp_async_elem<(int)sizeof(S)>(dv + tid, L + (long long)(k0 + tid) * ldm + k0 + tid);
    cp_commit();
  };
  double wr[QW], wi[QW];  // sum u_i^2 d_i over this CTA's panels (every lane its rows)
#pragma unroll
  for (int t = 0; t < QW; ++t) wr[t] = wi[t] = 0.0;
  if (rank == 0) load_diag(0);
  cl.sync();  // every CTA of the cluster runs before u goes into its shared memory
  for (int k = 0; k < np; ++k) {
    const int k0 = k * SB, kb = min(SB, n - k0);
    S* u_k = us + (k & 1) * SB * rp;
    if (k % C == rank) {
      cp_wait<0>();
      __syncthreads();
      // a warp's right-hand sides warp + 8 t; lane: rows lane and lane + 32
      const S* ak = acc + (size_t)(k / C) * SB * rp;
      S v[QW][2], p[QW][2][4], inv[2], d[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        d[h] = i < kb ? dv[i] : sfrom<S>(1.0, 0.0);
        inv[h] = finv(d[h]);
#pragma unroll
        for (int t = 0; t < QW; ++t) {
          const int q = warp + 8 * t;
          v[t][h] = (i < kb && q < r) ? sadd(Y[(long long)q * ldr + k0 + i], ak[i * rp + q]) : szero<S>();
#pragma unroll
          for (int m = 0; m < 4; ++m) p[t][h][m] = szero<S>();
        }
      }
      if (warp < r) {
#pragma unroll
        for (int hl = 0; hl < 2; ++hl) {  // rows l of the first, then of the second half
#pragma unroll 1
          for (int l4 = 0; l4 < 32; l4 += 4) {
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const int l = 32 * hl + l4 + m;
              const S w0 = wd[lane * (SB + 1) + l], w1 = wd[(lane + 32) * (SB + 1) + l];
#pragma unroll
              for (int t = 0; t < QW; ++t) {
                const S* ph = p[t][hl];
                const S own = fmul(inv[hl], ssub(v[t][hl], sadd(sadd(ph[0], ph[1]), sadd(ph[2], ph[3]))));
                const S u = shfl_s(own, l4 + m);
                if (lane == l4 + m) v[t][hl] = own;  // (u_l; the row takes no further updates)
                if (hl == 0) p[t][0][m] = sadd(p[t][0][m], fmul(w0, u));
                p[t][1][m] = sadd(p[t][1][m], fmul(w1, u));
              }
            }
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
#pragma unroll
        for (int t = 0; t < QW; ++t) {
          const int q = warp + 8 * t;
          if (i >= kb || q >= r) continue;
          const S u = v[t][h], x = fmul(d[h], fmul(u, u));
          wr[t] += sre(x);
          wi[t] += sim(x);
          u_k[i * rp + q] = u;
        }
      }
      __syncthreads();
      for (int o = 1; o < C; ++o) {
        S* there = cl.map_shared_rank(u_k, (rank + o) % C);
        for (int e = tid; e < SB * rp; e += 256) there[e] = u_k[e];
      }
    }
    cl.sync();
    if (k + 1 == np) break;
    if ((k + 1) % C == rank) load_diag(k + 1);  // (its previous block here was solved before the barrier)
    const int m0 = k < rank ? 0 : (k - rank) / C + 1;  // first owned block below panel k
    if (tid < groups * (256 / groups)) {
      const int q0 = FQ * (tid % groups);
      for (int row = m0 * SB + tid / groups; row < cnt * SB; row += 256 / groups) {
        const int gi = (rank + (row / SB) * C) * SB + row % SB;
        if (gi >= n) break;
        const S* wrow = L + (long long)gi * ldm + k0;
        S* ar = acc + (size_t)row * rp + q0;
        S a[FQ];
#pragma unroll
        for (int j = 0; j < FQ; ++j) a[j] = ar[j];
        // the row's next 64 bytes are on their way while the current ones are used
        constexpr int ST4 = 4 * PER;
        float4 x[4], y[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) x[c] = __ldg(reinterpret_cast<const float4*>(wrow + c * PER));
#pragma unroll 1
        for (int l0 = 0; l0 < SB; l0 += ST4) {
          const int ln = l0 + ST4 < SB ? l0 + ST4 : l0;
#pragma unroll
          for (int c = 0; c < 4; ++c) y[c] = __ldg(reinterpret_cast<const float4*>(wrow + ln + c * PER));
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const S* xs = reinterpret_cast<const S*>(&x[c]);
#pragma unroll
            for (int e = 0; e < PER; ++e) {
              const S* ul = u_k + (l0 + c * PER + e) * rp + q0;
#pragma unroll
              for (int j = 0; j < FQ; ++j) a[j] = sfnms(xs[e], ul[j], a[j]);
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) x[c] = y[c];
        }
#pragma unroll
        for (int j = 0; j < FQ; ++j) ar[j] = a[j];
      }
    }
  }
  double* there = cl.map_shared_rank(part, 0);
#pragma unroll
  for (int t = 0; t < QW; ++t) {
    const int q = warp + 8 * t;
    for (int o = 16; o > 0; o >>= 1) {
      wr[t] += __shfl_xor_sync(0xffffffffu, wr[t], o);
      wi[t] += __shfl_xor_sync(0xffffffffu, wi[t], o);
    }
    if (lane == 0 && q < r) {
      there[(rank * r + q) * 2] = wr[t];
      there[(rank * r + q) * 2 + 1] = wi[t];
    }
  }
  cl.sync();
  if (rank == 0 && tid < r) {
    double a = 0.0, b = 0.0;
    for (int c = 0; c < C; ++c) {
      a += part[(c * r + tid) * 2];
      b += part[(c * r + tid) * 2 + 1];
    }
    double* o = w + f * w_stride + (long long)tid * 2;
    o[0] = a - bnorm2[(long long)f * r + tid];
    o[1] = b;
  }
}

template <typename S>
size_t few_bytes(int n, int r, int C) {
  const int np = (n + SB - 1) / SB, rp = (r + FQ - 1) / FQ * FQ;
  return few_elems((np + C - 1) / C, rp) * sizeof(S) + (size_t)C * r * 16;
}

int sm_count() {
  int dev = 0, n = 1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
  return n;
}

// CTAs per cluster for F matrices, 0 for the one-CTA kernel. Both were measured for real and complex, FP32 and FP64, n 65 .. 1100, r 6
// .. 32 and 1 to 608 matrices with every cluster size:
//   the cluster grows until every SM has a CTA; where the arithmetic of a CTA fills an SM (FP64 beyond 8 right-hand sides, complex
//   FP32 beyond 16), while all of them still run at once (33 complex FP32 matrices of n 416, r = 32: 479 us with 8 CTAs each, 168
//   with 4, 446 with the kernel above; 64 real FP64 ones of 192, r = 24: 753 us with 4, 401 with 2, 428), and more where
//   the sums need the room. Up to two panels a second CTA has next to nothing to do.
//   Beyond 16 right-hand sides a panel's block is work for the one SM that solves it. FP64: one round of such CTAs takes (1.2 +
//   n / 208) (complex) or (2.45 + n / 300) (real) of what one round of the other kernel takes per panel (1 complex matrix, r = 24: n
//   65 776 against 616 us, n 192 1320 against 1835, n 416 3340 against 7630). FP32: three rounds of clusters of four and more
//   lose (152 complex ones of 1100, r = 32: 3270 against 2490 us).
// At none of the 600 points this is more than 5 % slower than the one-CTA kernel.
template <typename S>
int few_ctas(int n, int r, int F) {
  constexpr bool fp64 = sizeof(typename ST<S>::R) == 8, cplx = ST<S>::kComplex;
  const int np = (n + SB - 1) / SB, sms = sm_count();
  const bool full = sizeof(S) >= 8 && r > (fp64 ? 8 : 16);
  int C = 1;
  while (C < 8 && C < np - 1 && (full ? 2LL * F * C <= sms : (long long)F * C < sms)) C <<= 1;
  while (C <= 8 && few_bytes<S>(n, r, C) > (size_t)kFewSmem) C <<= 1;
  if (C > 8) return 0;
  if (r > 16) {
    const double rounds = (double)(((long long)F * C + sms - 1) / sms), other = (double)((F + sms - 1) / sms);
    if (fp64 && rounds * (cplx ? 1.2 + n / 208.0 : 2.45 + n / 300.0) > other * n / SB) return 0;
    if (!fp64 && C > 2 && (long long)F * C > 3LL * sms) return 0;
  }
  return C;
}

template <typename S, int QW>
int run_solve_few(const S* mats, int n, long long ldm, long long stride, const S* rhs, int r, long long ldr,
                  long long rhs_stride, const double* bnorm2, int F, double* w, long long w_stride, const int* active, int C,
                  size_t sm, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_solve_few_kernel<S, QW>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFewSmem) != cudaSuccess)
      return -1;
    attr = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(F * C);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ldlt_solve_few_kernel<S, QW>, mats, n, ldm, stride, rhs, r, ldr, rhs_stride, bnorm2, w, w_stride,
                            active) == cudaSuccess
             ? 1
             : -1;
}

template <typename S>
size_t solve_smem() {
  return SolveSmem<S>::bytes();
}

// Whether F matrices go by one CTA each. They do with a single panel, which has no update, and where they all run at once (two per
// SM, one in complex FP64) and either the chain of a small matrix's panels is shorter inside one CTA than as launches, up to n0, or
// there are so many that they fill the chip: the launches' time grows with F n^3, the other does not grow. The line is F =
// slots (1 - (n0 / n)^2). Measured (real and complex, FP32 and FP64, n 65 .. 1100, 1 to 608 matrices; launches against one CTA, us):
// complex FP32 n 96 F 64 146 and 125, n 320 F 152 691 and 651, F 33 558 and 612; real FP64 n 128 F 64 400 and 348, n 256 F 152
// 1447 and 1261, F 33 1053 and 1253; real FP32 n 200 F 152 316 and 247. Nowhere more than 4 % slower
// than one CTA per matrix, 12 % than the launches.
template <typename S>
bool one_cta_factor(int n, int F) {
  if (n <= PW) return true;
  constexpr bool fp64 = sizeof(typename ST<S>::R) == 8, cplx = ST<S>::kComplex;
  const int n0 = fp64 ? (cplx ? 128 : 160) : (cplx ? 192 : 256), sms = sm_count();
  const int slots = F <= sms || (fp64 && cplx) ? sms : 2 * sms;
  return F <= slots && (n <= n0 || (double)F * n * n >= (double)slots * ((double)n * n - (double)n0 * n0));
}

template <typename S>
int run_ldlt(S* mats, int n, int nrow, long long ldm, long long stride, int F, const int* active, unsigned* status,
             cudaStream_t s) {
  // a batch beyond the grid's y extent stays with the kernel above
  if (!one_cta_factor<S>(n, F) && F <= 65535) return run_ldlt_split(mats, n, nrow, ldm, stride, F, active, status, s);
  static bool attr = false;
  const size_t sm = std::max(FactorSmem<S>::bytes(), PanelSmem<S, kSimtThreads>::bytes());
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) return -1;
    attr = true;
  }
  ldlt_kernel<S><<<F, 256, sm, s>>>(mats, n, nrow, ldm, stride, active, status);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

template <typename S>
int run_solve(const S* mats, int n, long long ldm, long long stride, S* rhs, int r, long long ldr, long long rhs_stride,
              const double* bnorm2, int F, double* w, long long w_stride, const int* active, cudaStream_t s) {
  if (r <= kFewRhs && ldm % 4 == 0 && stride % 4 == 0 && (reinterpret_cast<uintptr_t>(mats) & 15) == 0) {  // 16-byte loads
    const int C = few_ctas<S>(n, r, F);
    const size_t few = C ? few_bytes<S>(n, r, C) : 0;
    if (C && r <= 8) return run_solve_few<S, 1>(mats, n, ldm, stride, rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, C, few, s);
    if (C && r <= 16) return run_solve_few<S, 2>(mats, n, ldm, stride, rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, C, few, s);
    if (C) return run_solve_few<S, 4>(mats, n, ldm, stride, rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, C, few, s);
  }
  static bool attr = false;
  const size_t sm = solve_smem<S>();
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_solve_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
      return -1;
    attr = true;
  }
  dim3 g(F, (r + SR - 1) / SR);
  ldlt_solve_kernel<S><<<g, 256, sm, s>>>(mats, n, ldm, stride, rhs, r, ldr, rhs_stride, bnorm2, w, w_stride, active);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace

int launch_ldlt(MatKind kind, void* mats, int n, int nrow, long long ldm, long long stride, int F, const int* active,
                unsigned* status, cudaStream_t s) {
  // 16-byte staging needs even leading dimensions and 16-byte aligned matrices
  if ((ldm % 4) || (stride % 4) || (reinterpret_cast<uintptr_t>(mats) & 15) || nrow < n) return -1;
  switch (kind) {
    case MatKind::RealF32: return run_ldlt((float*)mats, n, nrow, ldm, stride, F, active, status, s);
    case MatKind::CplxF32: return run_ldlt((float2*)mats, n, nrow, ldm, stride, F, active, status, s);
    case MatKind::RealF64: return run_ldlt((double*)mats, n, nrow, ldm, stride, F, active, status, s);
    default: return run_ldlt((double2*)mats, n, nrow, ldm, stride, F, active, status, s);
  }
}

// ---- appended right-hand-side rows ("bordered" matrix) -------------------------------------------
// With the r vectors b_q appended as rows n..n+r-1 of the lower triangle, the factorisation's row
// solves give W[n+q][k] = (L^-1 b_q)_k = y_k, so W^c_q = sum_k y_k^2 / d_k - |b_q|^2 follows from
// the factored rows without a separate forward substitution.
template <typename S>
__global__ void border_rows_kernel(S* __restrict__ mats, int n, long long ldm, long long stride,
                                   const double* __restrict__ src, long long src_row_stride, const int* __restrict__ row_of,
                                   int r, double* __restrict__ bnorm2) {
  const int f = blockIdx.y, q = blockIdx.x;
  const double* b = src + (size_t)row_of[f * r + q] * src_row_stride;
  S* row = mats + f * stride + (long long)(n + q) * ldm;
  double acc = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const double v = b[k];
    row[k] = sfrom<S>(v, 0.0);
    acc += v * v;
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    bnorm2[f * r + q] = t;
  }
}

template <typename S>
__global__ void border_w_kernel(const S* __restrict__ mats, int n, long long ldm, long long stride, int r,
                                const double* __restrict__ bnorm2, double* __restrict__ w, long long w_stride,
                                const int* __restrict__ active) {
  const int f = blockIdx.y, q = blockIdx.x;
  if (active && !active[f]) return;
  const S* A = mats + f * stride;
  const S* y = A + (long long)(n + q) * ldm;
  double sr = 0.0, si = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const S yk = y[k];
    const S t = smul(smul(yk, yk), sinv(A[(long long)k * ldm + k]));
    sr += sre(t);
    si += sim(t);
  }
  __shared__ double red[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, o);
    si += __shfl_down_sync(0xffffffffu, si, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sr;
    red[1][threadIdx.x >> 5] = si;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int v = 0; v < (int)(blockDim.x >> 5); ++v) {
      a += red[0][v];
      b += red[1][v];
    }
    double* o = w + f * w_stride + (long long)q * 2;
    o[0] = a - bnorm2[(long long)f * r + q];
    o[1] = b;
  }
}

int launch_border_rows(MatKind kind, void* mats, int n, long long ldm, long long stride, const double* src,
                       long long src_row_stride, const int* row_of, int F, int r, double* bnorm2, cudaStream_t s) {
  dim3 g(r, F);
  switch (kind) {
    case MatKind::CplxF32:
      border_rows_kernel<float2><<<g, 256, 0, s>>>((float2*)mats, n, ldm, stride, src, src_row_stride, row_of, r, bnorm2);
      break;
    case MatKind::CplxF64:
      border_rows_kernel<double2><<<g, 256, 0, s>>>((double2*)mats, n, ldm, stride, src, src_row_stride, row_of, r, bnorm2);
      break;
    case MatKind::RealF32:
      border_rows_kernel<float><<<g, 256, 0, s>>>((float*)mats, n, ldm, stride, src, src_row_stride, row_of, r, bnorm2);
      break;
    default:
      border_rows_kernel<double><<<g, 256, 0, s>>>((double*)mats, n, ldm, stride, src, src_row_stride, row_of, r, bnorm2);
      break;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_border_w(MatKind kind, const void* mats, int n, long long ldm, long long stride, int F, int r,
                    const double* bnorm2, double* w, long long w_stride, const int* active, cudaStream_t s) {
  dim3 g(r, F);
  switch (kind) {
    case MatKind::CplxF32:
      border_w_kernel<float2><<<g, 256, 0, s>>>((const float2*)mats, n, ldm, stride, r, bnorm2, w, w_stride, active);
      break;
    case MatKind::CplxF64:
      border_w_kernel<double2><<<g, 256, 0, s>>>((const double2*)mats, n, ldm, stride, r, bnorm2, w, w_stride, active);
      break;
    case MatKind::RealF32:
      border_w_kernel<float><<<g, 256, 0, s>>>((const float*)mats, n, ldm, stride, r, bnorm2, w, w_stride, active);
      break;
    default:
      border_w_kernel<double><<<g, 256, 0, s>>>((const double*)mats, n, ldm, stride, r, bnorm2, w, w_stride, active);
      break;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_ldlt_solve_w(MatKind kind, const void* mats, int n, long long ldm, long long stride, void* rhs, int r,
                        long long ldr, long long rhs_stride, const double* bnorm2, int F, double* w, long long w_stride,
                        const int* active, cudaStream_t s) {
  switch (kind) {
    case MatKind::RealF32:
      return run_solve((const float*)mats, n, ldm, stride, (float*)rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, s);
    case MatKind::CplxF32:
      return run_solve((const float2*)mats, n, ldm, stride, (float2*)rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, s);
    case MatKind::RealF64:
      return run_solve((const double*)mats, n, ldm, stride, (double*)rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active, s);
    default:
      return run_solve((const double2*)mats, n, ldm, stride, (double2*)rhs, r, ldr, rhs_stride, bnorm2, F, w, w_stride, active,
                       s);
  }
}

}  // namespace gwc
