// Tensor-core LDL^T of complex-symmetric FP32 dielectric matrices (sm_103a: tcgen05 + TMEM).
//
// Same factorisation, storage and panel order as the SIMT kernel (eps = L D L^T without pivoting;
// W = L D below the diagonal, d on it, L^T above it; appended rows n..nrow-1 become L^-1 b), with
// the rank-64 trailing update of every panel moved to the tensor cores:
//
//   C[i][j] -= sum_l W[i][l] L[j][l],   l in the panel, i >= j beyond the panel.
//
// Complex products as real GEMMs over split planes. With A = W rows (Ar, Ai) and B = L rows
// (Lr, Li) stored as the 128-row window [Lr ; Li], two accumulators of N = 128 columns take
//     P = Ar [Lr ; Li]^T = [Ar Lr^T | Ar Li^T],   Q = Ai [Lr ; Li]^T = [Ai Lr^T | Ai Li^T],
// and the epilogue forms Re = Ar Lr^T - Ai Li^T and Im = Ar Li^T + Ai Lr^T from them (N = 128 MMAs
// run at full rate; N = 64 ones at about 60 %).
//
// FP32 accuracy from TF32 operands (kind::tf32): every value v is split into hi = tf32(v) and
// lo = tf32(v - hi) (3xTF32; Henry, Tang & Heinecke 2019 for the BF16 analogue): each accumulator
// takes hi*hi + hi*lo + lo*hi, and the epilogue forms C - (P and Q terms) in round-to-nearest FP32.
//
// Roles (416 threads, one CTA per matrix):
//   warps 0-11  panel factorisation (factor_panel_tc below, named barrier 1)
//   warps 4-7   operand transform: global memory (L2) -> hi/lo planes in the 128-byte-swizzled
//               K-major layout. The A operand (W rows of a 128-row tile, all 64 panel columns)
//               stays resident while the tile row's column tiles pass; the B operand (L rows of a
//               64-column tile) streams through two stages of 32 panel columns, the global loads
//               of a stage issued before the wait for its buffer.
//   warp 12     TMEM allocation (512 columns: two tiles in flight x {D1, D2}) and the MMA issuer
//   warps 0-3,  epilogue: one thread per tile row and half of the tile's columns, the target values
//   8-11        read and written with 16-byte accesses, the next chunk's values loaded ahead
// The panel scratch aliases the operand buffers (the phases alternate).
// Every mbarrier wait is bounded (one second); on expiry the CTA records kStatTimeout, stops,
// drains the MMAs it issued and frees TMEM.
#include <algorithm>
#include <cstring>

#include "gwc_internal.h"
#include "ldlt_simt.cuh"
#include "tc_common.cuh"

namespace gwc {

namespace {

constexpr int TM = 128;                                  // rows per trailing tile (MMA M)
constexpr int TN = 64;                                   // complex columns per tile (MMA N per part)
constexpr int KH = 32;                                   // panel columns per stage (128-byte plane rows)
constexpr int A_PLANE = TM * 128;                        // 16 KB: [half][Ar, Ai, Ar_lo, Ai_lo]
constexpr int A_BYTES = 8 * A_PLANE;                     // 128 KB: the resident A operand
constexpr int B_PLANE = TN * 128;                        // 8 KB: Lr, Li, Lr_lo, Li_lo
constexpr int B_STAGE = 4 * B_PLANE;                     // 32 KB
constexpr int NSTAGE = 2;
constexpr int NT_TC = 416;                               // 13 warps
constexpr int MMA_WARP = 12;
constexpr int N_EPI = 256;                               // epilogue threads (warps 0-3, 8-11)
constexpr int META_BYTES = 128;
constexpr int OPS_BYTES = A_BYTES + NSTAGE * B_STAGE;    // 192 KB
constexpr int SMEM_TC = 1024 + OPS_BYTES + META_BYTES;
static_assert(PW == 2 * KH, "one panel is two stages");
constexpr int NT_PANEL = 384;                            // warps 0-11 factor the panels

// kind::tf32 instruction descriptor: D = F32, A = B = TF32, both K-major, N = 2 TN, M = TM.
constexpr uint32_t kIdescTf32 =
    (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(2 * TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "n"(kIdescTf32), "r"(accum));
}

// round to the nearest TF32 value (10 explicit mantissa bits), kept in an FP32 container
__device__ __forceinline__ float tf32_rn(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ void split4(const float (&v)[4], float4& hi, float4& lo) {
  float h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = tf32_rn(v[e]);
    l[e] = tf32_rn(v[e] - h[e]);
  }
  hi = make_float4(h[0], h[1], h[2], h[3]);
  lo = make_float4(l[0], l[1], l[2], l[3]);
}

// ---- diagonal blocks ---------------------------------------------------------------------------------
// The kb x kb diagonal block (kb <= 64) and X = L^-1 of its unit lower factor, by NT threads. Every element (i, c) of the
// lower triangle takes the right-looking updates in the order of the columns j,
//     a_ic -= W_ij (d_j^-1 W_cj), j < c,     X_ic -= W_ij (d_j^-1 X_jc), c <= j < i (X_jj = 1).
// What bounds the block is the chain of its 64 pivots (a reciprocal, two products and an exchange each), not its
// arithmetic, so the columns go in four blocks of 16:
//   pivots  one warp factors the 16 x 16 block in registers, two lanes per row;
//   panel   four lanes per row below and per column of X finish the block's columns (one exchange per pivot);
//   update  the next 16 x 16 block by all threads, then the rows below, for a and for X, in 2 x 4 tiles by the other warps
//           while the first warp takes the next block's pivots.
// The loops over j keep the current columns in front and shift: unrolled fully they were bound by instruction fetches. With one
// CTA barrier per pivot and every d_j^-1 W_cj formed again by each thread that uses it a block took 38 us; this takes
// 23 us, about 3.2 us for the 16 pivots of a block and 1.3 us for its panel step.
constexpr int DB = 16;        // columns per block
constexpr int LDB = 2 * DB;   // row of the in-block factors (the second half pads the shifted reads)
constexpr int LDP = PW + 1;   // padded row (conflict-free column access)
constexpr int LDM = PW + 2;   // row of the update's second operand (16-byte pairs)

// Scratch of a diagonal block at byte offset `o` of the dynamic shared memory (addressed through the shared array itself:
// pointers kept in a struct became generic loads)
struct DiagSmem {
  static constexpr int MJ = 0;                       // [16][66] d_j^-1 X_jc (columns c up to the block), d_j^-1 W_cj (beyond)
  static constexpr int LB = MJ + DB * LDM;           // [16][32] d_j^-1 W_ij inside the block, (j, i)
  static constexpr int WB = LB + DB * LDB;           // [16][32] W_ij inside the block, (j, i)
  static constexpr int DINV = WB + DB * LDB;         // [64] 1 / d
  static constexpr int DPIV = DINV + PW;             // [64] d (a zero pivot replaced by 1)
  static constexpr int DM = DPIV + PW;               // [64][65] a, then W below the diagonal
  static constexpr int XR = DM + PW * LDP;           // [64][65] X by rows
  static constexpr int ELEMS = XR + PW * LDP;
  uint32_t o;
  __device__ __forceinline__ float2& at(int e) const {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    return *reinterpret_cast<float2*>(smem_raw + o + e * 8);
  }
  __device__ __forceinline__ float4 pair(int e) const {  // two neighbours, e even
    extern __shared__ __align__(16) uint8_t smem_raw[];
    return *reinterpret_cast<const float4*>(smem_raw + o + e * 8);
  }
  __device__ __forceinline__ float2& dm(int i, int c) const { return at(DM + i * LDP + c); }
  __device__ __forceinline__ float2& xr(int i, int c) const { return at(XR + i * LDP + c); }
  __device__ __forceinline__ float2& mj(int j, int c) const { return at(MJ + j * LDM + c); }
  __device__ __forceinline__ float2& lb(int j, int i) const { return at(LB + j * LDB + i); }
  __device__ __forceinline__ float2& wb(int j, int i) const { return at(WB + j * LDB + i); }
  __device__ __forceinline__ float2& dinv(int j) const { return at(DINV + j); }
  __device__ __forceinline__ float2& dpiv(int j) const { return at(DPIV + j); }
};

// products with their roundings written out, so that a factor has the same bits whichever thread forms it
__device__ __forceinline__ float2 cmul_rn(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}
__device__ __forceinline__ float cabs2_rn(float2 a) { return __fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y)); }

__device__ __forceinline__ float2 shfl2(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// Pivots of the 16 x 16 block at j0 (its values in ds.dm) by one warp. Lanes i and 16 + i share row i: both carry the current pair
// of columns (v0, v1), and each the further columns of its parity (f[k] = column 2 + 2k + h of the row, relative to the pair). Of the
// reciprocal each half forms one part (one division instead of two in the chain), and the next pivot is formed by its own lane.
__device__ __forceinline__ void diag_pivots(int j0, int w16, const DiagSmem& ds, int* sing) {
  const int lane = threadIdx.x & 31, i = lane & 15, h = lane >> 4;
  float2 v0 = ds.dm(j0 + i, j0), v1 = ds.dm(j0 + i, j0 + 1), f[DB / 2 - 1];
#pragma unroll
  for (int k = 0; k + 1 < DB / 2; ++k) f[k] = ds.dm(j0 + i, j0 + 2 + 2 * k + h);
  bool zero;
  float2 d = shfl2(v0, 0), inv;
  auto pivot = [&] {
    zero = fabsf(d.x) + fabsf(d.y) < 1e-30f;
    if (zero) d = make_float2(1.f, 0.f);
    const float den = cabs2_rn(d);
    const float q = __fdiv_rn(h ? -d.y : d.x, den), o = __shfl_xor_sync(0xffffffffu, q, 16);
    inv = h ? make_float2(o, q) : make_float2(q, o);
  };
  pivot();
  // one column: l = d^-1 w published, the next column `next` updated, its pivot and reciprocal started
  auto column = [&](int j, float2 w, float2& next) {
    const float2 l = cmul_rn(inv, w), inv_j = inv, d_j = d;
    const bool zero_j = zero;
    const float2 e = sfnms(w, l, next);  // the diagonal entry in lane j + 1
    d = shfl2(e, j + 1);                 // (after the last column, a value that is not used)
    next = sfnms(w, shfl2(l, j + 1), next);
    if (i > j && lane < w16) {
      ds.dm(j0 + i, j0 + j) = w;
      ds.wb(j, i) = w;
      ds.lb(j, i) = l;
    }
    pivot();
    if (lane == j) {
      ds.dinv(j0 + j) = inv_j;
      ds.dpiv(j0 + j) = d_j;
      if (zero_j) *sing = 1;
    }
    __syncwarp();
  };
#pragma unroll 1
  for (int j = 0; j < w16; j += 2) {
    const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, f[0].x, 16), __shfl_xor_sync(0xffffffffu, f[0].y, 16));
    float2 v2 = h ? o : f[0], v3 = h ? f[0] : o;
    column(j, v0, v1);
    {
      const float4 x = ds.pair(DiagSmem::LB + j * LDB + j + 2);
      v2 = sfnms(v0, make_float2(x.x, x.y), v2);
      v3 = sfnms(v0, make_float2(x.z, x.w), v3);
#pragma unroll
      for (int k = 1; k + 1 < DB / 2; ++k) f[k] = sfnms(v0, ds.lb(j, j + 2 + 2 * k + h), f[k]);
    }
    if (j + 1 >= w16) break;  // uniform
    column(j + 1, v1, v2);
    {
      v3 = sfnms(v1, ds.lb(j + 1, j + 3), v3);
#pragma unroll
      for (int k = 1; k + 1 < DB / 2; ++k) f[k] = sfnms(v1, ds.lb(j + 1, j + 2 + 2 * k + h), f[k]);
    }
    v0 = v2;
    v1 = v3;
#pragma unroll
    for (int k = 0; k + 2 < DB / 2; ++k) f[k] = f[k + 1];
  }
}

// The panel step of the block at j0, four lanes per line: the lines t >= j1 are the rows below (their 16 columns of W), the lines t
// < j1 the columns of X (their 16 rows; zero above the diagonal). Lane s of a line holds its elements s, s + 4, s + 8, s + 12 as v;
// element j goes from its lane to the others, and each takes it off the elements beyond j. The results are W (ds.dm) or X
// (ds.xr), and d_j^-1 times them as the update's second operand.
template <bool COL>
__device__ __forceinline__ void diag_panel_lines(int j0, int w16, int kb, const DiagSmem& ds) {
  const int t = threadIdx.x >> 2, s = threadIdx.x & 3, grp = (threadIdx.x & 31) & ~3, line = min(t, kb - 1);
  float2 v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = COL ? ds.xr(j0 + s + 4 * q, line) : ds.dm(line, j0 + s + 4 * q);
#pragma unroll 1
  for (int j4 = 0; j4 < w16; j4 += 4) {
    float2 own = v[0];  // this lane's element of the four
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = j4 + e, m = (COL ? DiagSmem::WB : DiagSmem::LB) + j * LDB + j4 + s;
      const float2 x = shfl2(own, grp + e);
      float2 xs = cmul_rn(ds.dinv(j0 + j), x);
      if (COL) {  // X_ic -= W_ij (d_j^-1 X_jc), X_jc = 0 above the diagonal
        const bool on = j0 + j >= t;
        if (!on) xs = make_float2(0.f, 0.f);
        const float2 u = sfnms(ds.at(m), xs, own);
        if (on && s > e) own = u;
#pragma unroll
        for (int q = 1; q < 4; ++q) {
          const float2 y = sfnms(ds.at(m + 4 * q), xs, v[q]);
          if (on) v[q] = y;
        }
      } else {  // a_ic -= W_ij (d_j^-1 W_cj)
        const float2 u = sfnms(x, ds.at(m), own);
        if (s > e) own = u;
#pragma unroll
        for (int q = 1; q < 4; ++q) v[q] = sfnms(x, ds.at(m + 4 * q), v[q]);
      }
      if (s == e && t < kb && j < w16) {
        if (COL)
          ds.xr(j0 + j, t) = x;
        else
          ds.dm(t, j0 + j) = x;
        ds.mj(j, t) = xs;
      }
    }
    v[0] = v[1];
    v[1] = v[2];
    v[2] = v[3];
  }
}

// (8 lines per warp; below the block j1 is a multiple of 16, and with the last block there are no rows: a warp takes one side)
__device__ __forceinline__ void diag_panel(int j0, int kb, int j1, const DiagSmem& ds) {
  if ((int)(threadIdx.x >> 2) < j1 || j1 == kb)
    diag_panel_lines<true>(j0, j1 - j0, kb, ds);
  else
    diag_panel_lines<false>(j0, j1 - j0, kb, ds);
}

// diagonal block [k0, k0 + kb): W and d stored to A (and L^T above the diagonal if `lt`); dinv and xr left in shared memory
template <int NT>
__device__ void factor_diag_block(float2* __restrict__ A, long long ldm, int k0, int kb, const DiagSmem& ds, int* sing, bool lt) {
  static_assert(NT % 32 == 0 && NT >= DB * DB, "a thread per entry of a 16 x 16 block");
  const int tid = threadIdx.x;
  grp_sync_n<NT>();  // the previous phase's use of the scratch is over
  constexpr int PT = (PW * PW + NT - 1) / NT;
  for (int h = 0; h < PT; h += 8) {
    float2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + (h + q) * NT, i = e >> 6, c = e & 63;
      v[q] = (i < kb && c <= i) ? A[(long long)(k0 + i) * ldm + (k0 + c)] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + (h + q) * NT, i = e >> 6, c = e & 63;
      if (e < PW * PW) {
        ds.dm(i, c) = v[q];
        ds.xr(i, c) = make_float2(i == c ? 1.f : 0.f, 0.f);
      }
    }
  }
  grp_sync_n<NT>();
  if (tid < 32) diag_pivots(0, min(DB, kb), ds, sing);
  grp_sync_n<NT>();
  for (int j0 = 0; j0 < kb; j0 += DB) {
    const int j1 = min(j0 + DB, kb);
    if (tid < 4 * PW) diag_panel(j0, kb, j1, ds);
    grp_sync_n<NT>();
    const int nr = kb - j1;
    if (nr <= 0) break;  // (below, j1 < kb: the block is full)
    if (tid < DB * DB) {  // the next 16 x 16 block takes the 16 updates, an entry per thread
      const int r = tid >> 4, c = tid & 15, i = j1 + r;
      if (c <= r && i < kb) {
        float2 v = ds.dm(i, j1 + c);
#pragma unroll 8
        for (int j = 0; j < DB; ++j) v = sfnms(ds.dm(i, j0 + j), ds.mj(j, j1 + c), v);
        ds.dm(i, j1 + c) = v;
      }
    }
    grp_sync_n<NT>();
    if (tid < 32) {
      diag_pivots(j1, min(DB, nr), ds, sing);
    } else if ((tid >> 5) & 3) {  // (no warp on the first one's scheduler: its chain is the longer of the two)
      // rows below the block: a_ic (c beyond the block) and X_ic (c up to it); a thread's rows are r and r + tr
      const int tr = (nr + 1) >> 1;
      for (int e = tid - 32 - 32 * (tid >> 7); e < tr * (PW / 4); e += NT / 4 * 3) {
        const int r = e % tr, c0 = 4 * (e / tr), i0 = j1 + r, i1 = min(i0 + tr, kb - 1);
        if (c0 > i1 || (c0 >= j1 && i1 < j1 + DB)) continue;  // above the diagonal, or the next 16 x 16 block
        const bool x_side = c0 < j1;  // a tile lies on one side: j1 is a multiple of 4
        const int t = (x_side ? DiagSmem::XR : DiagSmem::DM) + c0, t0 = t + i0 * LDP, t1 = t + i1 * LDP;
        float2 v[2][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          v[0][c] = ds.at(t0 + c);
          v[1][c] = ds.at(t1 + c);
        }
#pragma unroll 2
        for (int j = 0; j < DB; ++j) {
          const float2 w0 = ds.dm(i0, j0 + j), w1 = ds.dm(i1, j0 + j);
          const float4 m0 = ds.pair(DiagSmem::MJ + j * LDM + c0);
          const float4 m1 = ds.pair(DiagSmem::MJ + j * LDM + c0 + 2);
          const float2 m[4] = {make_float2(m0.x, m0.y), make_float2(m0.z, m0.w), make_float2(m1.x, m1.y),
                               make_float2(m1.z, m1.w)};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            v[0][c] = sfnms(w0, m[c], v[0][c]);
            v[1][c] = sfnms(w1, m[c], v[1][c]);
          }
        }
        // (entries above the diagonal of a tile on it are not used; the next 16 x 16 block is the first warp's)
        const bool s0 = x_side || i0 >= j1 + DB, s1 = i0 + tr < kb;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (s0) ds.at(t0 + c) = v[0][c];
          if (s1) ds.at(t1 + c) = v[1][c];
        }
      }
    }
    grp_sync_n<NT>();
  }
  for (int e = tid; e < PW * PW; e += NT) {
    const int i = e >> 6, c = e & 63;
    if (i >= kb || c > i) continue;
    const float2 w = c < i ? ds.dm(i, c) : ds.dpiv(i);
    A[(long long)(k0 + i) * ldm + (k0 + c)] = w;
    if (lt && c < i) A[(long long)(k0 + c) * ldm + (k0 + i)] = smul(w, ds.dinv(c));
  }
}

// ---- panel factorisation of the one-CTA kernel (warps 0-11) --------------------------------------------
// The diagonal block above, then the rows below without any dependent chain: W_rows = A_rows X^T (a product over the panel
// columns, X^T upper triangular) and L^T_rows = (W_rows D^-1)^T.
struct PanelInv {
  static constexpr int CH = 16 * (NT_PANEL / 32);     // 192 staged rows: 6 blocks of 32 x 2 group pairs
  float2 (*xg)[PW];    // [64][64] xg[l][c] = X_cl (zero for c < l), 16-byte rows for broadcast loads
  DiagSmem ds;         // scratch of the diagonal block (1 / d stays) ...
  float2* dinv;
  float2 (*ach)[LDP];  // [CH][65] ... the staged rows below the panel after it (aliases dm and xr)
  static constexpr size_t bytes() { return sizeof(float2) * (PW * PW + DiagSmem::DM + (size_t)CH * LDP); }
  __device__ explicit PanelInv(uint8_t* base) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    float2* p = reinterpret_cast<float2*>(base);
    xg = reinterpret_cast<float2(*)[PW]>(p);
    p += PW * PW;
    ds.o = smem_u32(p) - smem_u32(smem_raw);
    dinv = p + DiagSmem::DINV;
    ach = reinterpret_cast<float2(*)[LDP]>(p + DiagSmem::DM);
  }
};
static_assert(PanelInv::bytes() <= (size_t)OPS_BYTES, "panel scratch fits in the operand buffers");
static_assert(2 * PW <= PanelInv::CH, "the diagonal block fits in the staging rows");

__device__ __forceinline__ void panel_sync() { grp_sync_n<NT_PANEL>(); }

// One warp's share of a staged chunk: rows r0 .. r0 + 31 (one per lane), the 16 columns of group g,
// w_c = sum_{l <= c} a_l X_cl in packed FP32 pairs (re and im of X per product), then W (row-major,
// lower part) and L^T (transposed, coalesced over the lanes) stored.
__device__ __forceinline__ void panel_rows_group(float2* __restrict__ A, int n, long long ldm, int k0, int kb,
                                                 const PanelInv& ps, int r, int i, bool row_ok, int g) {
  const int cb = 16 * g, ncol = min(16, kb - cb);
  const float2* arow = ps.ach[r];
  float2* rowp = A + (long long)i * ldm + k0 + cb;
  // two passes of 8 columns (c0 = 0, 8): 16 float2 accumulators per pass keep the loop in registers
#pragma unroll 1
  for (int c0 = 0; c0 < 16; c0 += 8) {
    if (c0 >= ncol) break;
    const int lmax = min(cb + c0 + 8, kb);  // X_cl = 0 for l > c
    float2 pr[8], pi[8];  // pr[c] = sum a.re (X re, X im), pi[c] = sum a.im (X re, X im)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      pr[c] = make_float2(0.f, 0.f);
      pi[c] = make_float2(0.f, 0.f);
    }
#pragma unroll 4
    for (int l = 0; l < lmax; ++l) {
      const float2 a = arow[l];
      const float2 ar = make_float2(a.x, a.x), ai = make_float2(a.y, a.y);
      const float4* xp = reinterpret_cast<const float4*>(&ps.xg[l][cb + c0]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 x = xp[q];
        const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
        pr[2 * q] = __ffma2_rn(ar, x0, pr[2 * q]);
        pi[2 * q] = __ffma2_rn(ai, x0, pi[2 * q]);
        pr[2 * q + 1] = __ffma2_rn(ar, x1, pr[2 * q + 1]);
        pi[2 * q + 1] = __ffma2_rn(ai, x1, pi[2 * q + 1]);
      }
    }
    if (!row_ok) continue;
    float2 w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = make_float2(pr[c].x - pi[c].y, pr[c].y + pi[c].x);
    const int nc8 = min(8, ncol - c0);
    if (nc8 == 8) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(rowp + c0 + 2 * q) = make_float4(w[2 * q].x, w[2 * q].y, w[2 * q + 1].x, w[2 * q + 1].y);
    } else {
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (c < nc8) rowp[c0 + c] = w[c];
    }
    if (i < n) {
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (c < nc8) A[(long long)(k0 + cb + c0 + c) * ldm + i] = smul(w[c], ps.dinv[cb + c0 + c]);
    }
  }
}

// Panel [k0, k0 + kb): the diagonal block, then every row below (appended right-hand-side rows
// n..nrow-1 included, W only) in chunks of CH staged rows; warp w takes the 32-row block w / 2 of a
// chunk and the column groups {0, 3} or {1, 2} (equal work: the triangle of X).
__device__ void factor_panel_tc(float2* __restrict__ A, int n, int nrow, long long ldm, int k0, const PanelInv& ps,
                                int* sing) {
  const int kb = min(PW, n - k0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    const DiagSmem ds = ps.ds;
    factor_diag_block<NT_PANEL>(A, ldm, k0, kb, ds, sing, true);
    for (int e = tid; e < PW * PW; e += NT_PANEL) {
      const int l = e >> 6, c = e & 63;
      ps.xg[l][c] = (c >= l && c < kb) ? ds.xr(c, l) : make_float2(0.f, 0.f);
    }
    panel_sync();  // xg, dinv complete; dm and xr may be overwritten by the staged rows
  }
  const int r = 32 * (warp >> 1) + lane;
  const int g0 = (warp & 1) ? 1 : 0, g1 = (warp & 1) ? 2 : 3;
  for (int base = k0 + kb; base < nrow; base += PanelInv::CH) {
    for (int e = tid; e < PanelInv::CH * PW; e += NT_PANEL) {
      const int rr = e >> 6, l = e & 63, i = base + rr;
      if (i < nrow && l < kb) cp_async_elem<8>(&ps.ach[rr][l], A + (long long)i * ldm + k0 + l);
    }
    cp_commit();
    cp_wait<0>();
    panel_sync();
    const int i = base + r;
    const bool row_ok = i < nrow;
    if (base + 32 * (warp >> 1) < nrow) {  // warp-uniform: the block has rows
      if (16 * g0 < kb) panel_rows_group(A, n, ldm, k0, kb, ps, r, i, row_ok, g0);
      if (16 * g1 < kb) panel_rows_group(A, n, ldm, k0, kb, ps, r, i, row_ok, g1);
    }
    panel_sync();  // the staging rows are free
  }
}

// column tiles of row tile tI: j0 = R0 + TN tJ < min(n, i0 + TM)
__device__ __forceinline__ int tile_cols(int R0, int n, int tI) {
  const int jmax = min(n, R0 + TM * tI + TM);
  return (jmax - R0 + TN - 1) / TN;
}

struct TcSmem {
  uint8_t* base;  // A operand, then the B stages
  uint64_t *a_full, *a_empty, *b_full, *b_empty, *tfull, *tempty, *mma_done;
  uint32_t* tmem_slot;
  volatile int* abort_flag;
  int* sing;
  unsigned long long wait_ns;  // bound of every mbarrier wait
};

// Iterates the (row tile, column tile, half) stages of one panel in issue order.
struct StageIt {
  int R0, n, n_ti;
  int tI, tJ, h, nc;
  __device__ void init(int R0_, int n_, int n_ti_) {
    R0 = R0_;
    n = n_;
    n_ti = n_ti_;
    tI = 0;
    tJ = 0;
    h = 0;
    nc = tile_cols(R0, n, 0);
  }
  __device__ bool valid() const { return tI < n_ti; }
  __device__ void next() {
    if (++h == 2) {
      h = 0;
      if (++tJ == nc) {
        tJ = 0;
        ++tI;
        nc = tI < n_ti ? tile_cols(R0, n, tI) : 0;
      }
    }
  }
};

// B operand values of one stage for this thread: L^T[k0 + KH h + 16 lh + e][j0 + jj], e < 16
__device__ __forceinline__ void load_b(float2 (&bv)[16], const float2* A, int n, long long ldm, int k0,
                                       const StageIt& it, int tt) {
  const int jj = tt & 63, lh = tt >> 6, j = it.R0 + TN * it.tJ + jj;
  const bool jv = j < n;
  const float2* colp = A + (long long)(k0 + KH * it.h + 16 * lh) * ldm + (jv ? j : 0);
#pragma unroll
  for (int e = 0; e < 16; ++e) bv[e] = jv ? colp[(long long)e * ldm] : make_float2(0.f, 0.f);
}

// ---- operand transform (warps 4-7) --------------------------------------------------------------
// (A is written by this kernel: plain coherent loads, no read-only path)
__device__ void transform_role(const TcSmem& sm, const float2* A, int n, int nrow, long long ldm, int k0, int R0,
                               int n_ti, int seq, int rt) {
  const int tt = threadIdx.x - 128;  // 0..127
  StageIt it;
  it.init(R0, n, n_ti);
  float2 bv[16];
  load_b(bv, A, n, ldm, k0, it, tt);
  bool ok = true;
  for (int tI = 0; tI < n_ti && ok; ++tI, ++rt) {
    // A operand of row tile tI: W[i0 + row][k0 .. k0 + 64), four threads per row (64 bytes each)
    if (!mbar_wait(smem_u32(sm.a_empty), (rt & 1) ^ 1, sm.abort_flag, sm.wait_ns)) break;
    {
      const int rq = tt & 3, rr = tt >> 2;
      const int i0 = R0 + TM * tI;
#pragma unroll 1
      for (int hp = 0; hp < 4; ++hp) {  // (half, pair of row passes)
        const int h = hp >> 1;
        float4 av[8];
#pragma unroll
        for (int pp = 0; pp < 2; ++pp) {
          const int i = i0 + rr + 32 * (2 * (hp & 1) + pp);
          const float4* src =
              reinterpret_cast<const float4*>(A + (long long)(i < nrow ? i : 0) * ldm + k0 + KH * h + 8 * rq);
#pragma unroll
          for (int c = 0; c < 4; ++c) av[4 * pp + c] = i < nrow ? src[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int pp = 0; pp < 2; ++pp) {
          const int r = rr + 32 * (2 * (hp & 1) + pp), sw = r & 7;
          uint8_t* rowp = sm.base + h * 4 * A_PLANE + r * 128;
#pragma unroll
          for (int e = 0; e < 2; ++e) {  // chunk 2 rq + e: complex l = 8 rq + 4 e .. + 3
            const float4 v0 = av[4 * pp + 2 * e], v1 = av[4 * pp + 2 * e + 1];
            const float re[4] = {v0.x, v0.z, v1.x, v1.z};
            const float im[4] = {v0.y, v0.w, v1.y, v1.w};
            float4 rh, rl, ih, il;
            split4(re, rh, rl);
            split4(im, ih, il);
            const int off = ((2 * rq + e) ^ sw) << 4;
            *reinterpret_cast<float4*>(rowp + off) = rh;
            *reinterpret_cast<float4*>(rowp + A_PLANE + off) = ih;
            *reinterpret_cast<float4*>(rowp + 2 * A_PLANE + off) = rl;
            *reinterpret_cast<float4*>(rowp + 3 * A_PLANE + off) = il;
          }
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(smem_u32(sm.a_full));
    // B operand stages of this row tile
    const int nc = tile_cols(R0, n, tI);
    for (int q = 0; q < 2 * nc; ++q, ++seq) {
      const int s = seq & 1, us = seq >> 1;
      if (!mbar_wait(smem_u32(&sm.b_empty[s]), (us & 1) ^ 1, sm.abort_flag, sm.wait_ns)) {
        ok = false;
        break;
      }
      const int jj = tt & 63, lh = tt >> 6, sw = jj & 7;
      uint8_t* rowp = sm.base + A_BYTES + s * B_STAGE + jj * 128;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float lr[4], li[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          lr[e] = bv[4 * c + e].x;
          li[e] = bv[4 * c + e].y;
        }
        float4 rh, rl, ih, il;
        split4(lr, rh, rl);
        split4(li, ih, il);
        const int off = ((4 * lh + c) ^ sw) << 4;
        *reinterpret_cast<float4*>(rowp + off) = rh;
        *reinterpret_cast<float4*>(rowp + B_PLANE + off) = ih;
        *reinterpret_cast<float4*>(rowp + 2 * B_PLANE + off) = rl;
        *reinterpret_cast<float4*>(rowp + 3 * B_PLANE + off) = il;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(smem_u32(&sm.b_full[s]));
      // the next stage's loads travel while this thread waits for that stage's buffer
      it.next();
      if (it.valid()) load_b(bv, A, n, ldm, k0, it, tt);
    }
  }
}

// ---- MMA issuer (one thread of warp 8) ----------------------------------------------------------
__device__ void mma_role(const TcSmem& sm, uint32_t tmem_base, int n, int R0, int n_ti, int seq, int tcount, int rt) {
  bool ok = true;
  const uint32_t abase = smem_u32(sm.base);
  for (int tI = 0; tI < n_ti && ok; ++tI, ++rt) {
    if (!mbar_wait(smem_u32(sm.a_full), rt & 1, sm.abort_flag, sm.wait_ns)) break;
    tc_fence_after();
    const int nc = tile_cols(R0, n, tI);
    for (int tJ = 0; tJ < nc && ok; ++tJ, ++tcount) {
      const int b = tcount & 1, ub = tcount >> 1;
      if (!mbar_wait(smem_u32(&sm.tempty[b]), (ub & 1) ^ 1, sm.abort_flag, sm.wait_ns)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t dp = tmem_base + (uint32_t)(b * 256), dq = dp + 128;  // P and Q accumulators
      for (int h = 0; h < 2; ++h, ++seq) {
        const int s = seq & 1, us = seq >> 1;
        if (!mbar_wait(smem_u32(&sm.b_full[s]), us & 1, sm.abort_flag, sm.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t ah = abase + h * 4 * A_PLANE;
        const uint32_t ar = ah, ai = ah + A_PLANE, arl = ah + 2 * A_PLANE, ail = ah + 3 * A_PLANE;
        const uint32_t bb = abase + A_BYTES + s * B_STAGE;
        const uint32_t br = bb, bi = bb + B_PLANE, brl = bb + 2 * B_PLANE, bil = bb + 3 * B_PLANE;
        // descriptors once per stage; a k step moves the start address by 32 bytes = 2 units of the
        // 16-byte address field (few instructions per MMA for the issuing thread)
        const uint64_t dar = sdesc(ar), dai = sdesc(ai), darl = sdesc(arl), dail = sdesc(ail);
        const uint64_t dbr = sdesc(br), dbi = sdesc(bi), dbrl = sdesc(brl), dbil = sdesc(bil);
#pragma unroll
        for (int k = 0; k < KH / 8; ++k) {
          const uint64_t o = 2u * k;  // 8 TF32 values = 32 bytes along K inside the 128-B row
          const uint32_t acc = (h == 0 && k == 0) ? 0u : 1u;
          const uint64_t a_r = dar + o, a_i = dai + o, a_rl = darl + o, a_il = dail + o;
          const uint64_t bh = dbr + o, bl = dbrl + o;  // [Lr ; Li] hi and lo windows (N = 128)
          mma_tf32(dp, a_r, bh, acc);
          mma_tf32(dp, a_r, bl, 1u);
          mma_tf32(dp, a_rl, bh, 1u);
          mma_tf32(dq, a_i, bh, acc);
          mma_tf32(dq, a_i, bl, 1u);
          mma_tf32(dq, a_il, bh, 1u);
        }
        mma_commit(smem_u32(&sm.b_empty[s]));
      }
      if (!ok) break;
      mma_commit(smem_u32(&sm.tfull[b]));
    }
    if (!ok) break;
    mma_commit(smem_u32(sm.a_empty));  // the row tile's A operand is free once its MMAs complete
  }
}

// ---- epilogue (warps 0-3 and 8-11): C -= D1 + D2 -----------------------------------------------
// Warp w serves TMEM lanes 32 (w % 4) .. +31 (rows of the tile) and, with its partner w ^ 8, half
// of the tile's 64 columns: two 16-column chunks. Each thread owns one row; the target values of
// its next chunk are loaded (16-byte loads) while the current one is formed.
// TMEM loads without the implicit wait, so the accumulator slices of a chunk share one wait
__device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// this thread's chunks in issue order: (row tile, column tile, chunk cc0 or cc0 + 1)
struct ChunkIt {
  int R0, n, nrow, n_ti, r, cc0;
  int tI, tJ, cc, nc, i, jlim;
  __device__ void set_row() {
    i = R0 + TM * tI + r;
    jlim = i < nrow ? (i < n ? min(n, i + 1) : n) : 0;  // j <= i inside the factored block
  }
  __device__ void init(int R0_, int n_, int nrow_, int n_ti_, int r_, int cc0_) {
    R0 = R0_;
    n = n_;
    nrow = nrow_;
    n_ti = n_ti_;
    r = r_;
    cc0 = cc0_;
    tI = 0;
    tJ = 0;
    cc = cc0;
    nc = tile_cols(R0, n, 0);
    set_row();
  }
  __device__ bool valid() const { return tI < n_ti; }
  __device__ int jb() const { return R0 + TN * tJ + 16 * cc; }
  __device__ bool full() const { return valid() && jb() + 16 <= jlim; }
  __device__ void next() {
    if (++cc == cc0 + 2) {
      cc = cc0;
      if (++tJ == nc) {
        tJ = 0;
        ++tI;
        nc = tI < n_ti ? tile_cols(R0, n, tI) : 0;
        set_row();
      }
    }
  }
};

__device__ void epilogue_role(const TcSmem& sm, uint32_t tmem_base, float2* __restrict__ A, int n, int nrow,
                              long long ldm, int R0, int n_ti, int tcount) {
  const int warp = threadIdx.x >> 5, q = warp & 3, cc0 = 2 * (warp >> 3);
  const int r = 32 * q + (threadIdx.x & 31);
  const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16);
  ChunkIt it;
  it.init(R0, n, nrow, n_ti, r, cc0);
  float4 nxt[8];
  if (it.full()) {
    const float2* p = A + (long long)it.i * ldm + it.jb();
#pragma unroll
    for (int e = 0; e < 8; ++e) nxt[e] = *reinterpret_cast<const float4*>(p + 2 * e);
  }
  bool ok = true;
  for (int tI = 0; tI < n_ti && ok; ++tI) {
    const int nc = tile_cols(R0, n, tI);
    for (int tJ = 0; tJ < nc; ++tJ, ++tcount) {
      const int b = tcount & 1, ub = tcount >> 1;
      ok = mbar_wait(smem_u32(&sm.tfull[b]), ub & 1, sm.abort_flag, sm.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int cc = cc0; cc < cc0 + 2; ++cc) {
        const bool full = it.full();
        const int jb = it.jb(), jlim = it.jlim, i = it.i;
        float4 cur[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) cur[e] = nxt[e];
        it.next();
        if (it.full()) {  // the next chunk's target values, in flight while this one is formed
          const float2* pn = A + (long long)it.i * ldm + it.jb();
#pragma unroll
          for (int e = 0; e < 8; ++e) nxt[e] = *reinterpret_cast<const float4*>(pn + 2 * e);
        }
        float2* p = A + (long long)i * ldm + jb;
        const bool part = !full && jb < jlim;
        if (part) {  // ragged chunk: the valid columns only
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float2 u = jb + 2 * e < jlim ? p[2 * e] : make_float2(0.f, 0.f);
            const float2 v = jb + 2 * e + 1 < jlim ? p[2 * e + 1] : make_float2(0.f, 0.f);
            cur[e] = make_float4(u.x, u.y, v.x, v.y);
          }
        }
        // Re = Ar Lr^T - Ai Li^T: P columns 16 cc.., Q columns 64 + 16 cc..
        const uint32_t col = lane_base + (uint32_t)(b * 256 + 16 * cc);
        uint32_t t1[16], t2[16];
        tmem_ld16_nw(col, t1);
        tmem_ld16_nw(col + 128 + 64, t2);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          cur[e].x = cur[e].x - __uint_as_float(t1[2 * e]) + __uint_as_float(t2[2 * e]);
          cur[e].z = cur[e].z - __uint_as_float(t1[2 * e + 1]) + __uint_as_float(t2[2 * e + 1]);
        }
        // Im = Ar Li^T + Ai Lr^T: P columns 64 + 16 cc.., Q columns 16 cc..
        tmem_ld16_nw(col + 64, t1);
        tmem_ld16_nw(col + 128, t2);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          cur[e].y = cur[e].y - __uint_as_float(t1[2 * e]) - __uint_as_float(t2[2 * e]);
          cur[e].w = cur[e].w - __uint_as_float(t1[2 * e + 1]) - __uint_as_float(t2[2 * e + 1]);
        }
        if (full) {
#pragma unroll
          for (int e = 0; e < 8; ++e) *reinterpret_cast<float4*>(p + 2 * e) = cur[e];
        } else if (part) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            if (jb + 2 * e < jlim) p[2 * e] = make_float2(cur[e].x, cur[e].y);
            if (jb + 2 * e + 1 < jlim) p[2 * e + 1] = make_float2(cur[e].z, cur[e].w);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(smem_u32(&sm.tempty[b]));
    }
  }
}

// The factorisation of one matrix A (n columns, nrow rows) by one CTA.
__device__ __forceinline__ void ldlt_tc_matrix(float2* __restrict__ A, int n, int nrow, long long ldm,
                                               unsigned* __restrict__ status, unsigned long long wait_ns) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  TcSmem sm;
  sm.base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm.base + OPS_BYTES);
  sm.a_full = bars;
  sm.a_empty = bars + 1;
  sm.b_full = bars + 2;
  sm.b_empty = bars + 4;
  sm.tfull = bars + 6;
  sm.tempty = bars + 8;
  sm.mma_done = bars + 10;
  sm.tmem_slot = reinterpret_cast<uint32_t*>(bars + 11);
  sm.abort_flag = reinterpret_cast<volatile int*>(sm.tmem_slot + 1);
  sm.sing = reinterpret_cast<int*>(sm.tmem_slot + 2);
  sm.wait_ns = wait_ns;
  const PanelInv ps(sm.base);  // aliases the operand buffers (the phases alternate)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(sm.a_full), 128);
    mbar_init(smem_u32(sm.a_empty), 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&sm.b_full[i]), 128);
      mbar_init(smem_u32(&sm.b_empty[i]), 1);
      mbar_init(smem_u32(&sm.tfull[i]), 1);
      mbar_init(smem_u32(&sm.tempty[i]), N_EPI);
    }
    mbar_init(smem_u32(sm.mma_done), 1);
    *sm.abort_flag = 0;
    *sm.sing = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(sm.tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem_slot;

  // B stages, tiles and row tiles issued so far; every role advances them alike
  int seq = 0, tcount = 0, rt = 0;
  for (int k0 = 0; k0 < n; k0 += PW) {
    const int kb = min(PW, n - k0);
    if (warp < NT_PANEL / 32) factor_panel_tc(A, n, nrow, ldm, k0, ps, sm.sing);
    __syncthreads();  // panel W / L^T in global memory; the panel scratch is free
    const int R0 = k0 + kb;
    if (R0 < n) {
      const int n_ti = (nrow - R0 + TM - 1) / TM;
      if (warp == MMA_WARP) {
        if (lane == 0) mma_role(sm, tmem_base, n, R0, n_ti, seq, tcount, rt);
        __syncwarp();
      } else if (warp >= 4 && warp < 8) {
        transform_role(sm, A, n, nrow, ldm, k0, R0, n_ti, seq, rt);
      } else {
        epilogue_role(sm, tmem_base, A, n, nrow, ldm, R0, n_ti, tcount);
      }
      int nt = 0;
      for (int tI = 0; tI < n_ti; ++tI) nt += tile_cols(R0, n, tI);
      seq += 2 * nt;
      tcount += nt;
      rt += n_ti;
    }
    tc_fence_before();
    __syncthreads();  // every tile of the panel is written back; the operand buffers are free
    tc_fence_after();
    if (*sm.abort_flag) break;
  }
  // every MMA issued has completed before TMEM is freed (immediate unless a wait gave up)
  if (warp == MMA_WARP) {
    if (lane == 0) {
      mma_commit(smem_u32(sm.mma_done));
      mbar_drain(smem_u32(sm.mma_done), 0);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (*sm.abort_flag) atomicOr(status, kStatTimeout);
    if (*sm.sing) atomicOr(status, kStatSingular);
  }
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
  }
}

__global__ void __launch_bounds__(NT_TC, 1)
    ldlt_tc_kernel(float2* __restrict__ mats, int n, int nrow, long long ldm, long long stride,
                   const int* __restrict__ active, unsigned* __restrict__ status, unsigned long long wait_ns) {
  const int f = blockIdx.x;
  if (active && !active[f]) return;  // uniform across the CTA, before any barrier or TMEM use
  ldlt_tc_matrix(mats + f * stride, n, nrow, ldm, status, wait_ns);
}

// Grouped: CTA b factors matrix b - cta0 of the group whose CTA range holds b (groups ascending in cta0).
__global__ void __launch_bounds__(NT_TC, 1)
    ldlt_tc_grouped_kernel(const LdltGroup* __restrict__ gs, int n_groups, unsigned* __restrict__ status,
                           unsigned long long wait_ns) {
  int lo = 0, hi = n_groups - 1;
  while (lo < hi) {  // last group with cta0 <= blockIdx.x
    const int mid = (lo + hi + 1) / 2;
    if (gs[mid].cta0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const LdltGroup& G = gs[lo];
  const int f = blockIdx.x - G.cta0;
  if (f >= G.F) return;
  if (G.active && !G.active[f]) return;  // uniform across the CTA, before any barrier or TMEM use
  ldlt_tc_matrix(G.mats + f * G.stride, G.n, G.nrow, G.ldm, status, wait_ns);
}

// ---- split factorisation: per panel, launches over all matrices of the batch -------------------------
// The kernel above gives each matrix one CTA for its whole factorisation, and its tensor phase waits on
// the per-thread global loads of one SM (a 4500-wide matrix takes ~190 ms). Here every panel is three
// launches over all matrices of the batch:
//   ldlt_diag_kernel    the 64 x 64 diagonal block and the inverse of its unit lower factor (one CTA per matrix);
//   ldlt_rows_kernel    the rows below it (64 per CTA), with the panel's W columns and L rows as TF32 hi / lo
//                       planes, K-major (L^T is not kept above the diagonal: only the planes feed the update);
//   ldlt_update_kernel  C[i][j] -= sum_l W[i][l] L[j][l] over the trailing 128 x 64 tiles of every matrix,
//                       one tile per CTA, two CTAs per SM: TMA-fed planes, the P and Q accumulators of the
//                       one-CTA kernel, and the target tile staged through shared memory by TMA (128-byte
//                       swizzle, clipped at column n and row nrow; the part of a diagonal tile above the
//                       diagonal holds nothing).
// Panels go in pairs with a one-panel lookahead: panel p's update is first applied to panel p + 1's 64
// columns only, panel p + 1 is factored, and then one rank-128 update (K = 128: both panels' planes side by
// side) covers the trailing matrix, which is thus read and written once per two panels.

constexpr int UP_A = TM * 128;                   // one A plane chunk: 128 rows x 32 FP32 = 16 KB
constexpr int UP_B = TN * 128;                   // one B plane chunk: 64 rows x 32 FP32 = 8 KB
constexpr int UP_STAGE = 4 * UP_A + 4 * UP_B;    // Ar, Ai, Ar_lo, Ai_lo | Lr, Li, Lr_lo, Li_lo: 96 KB
constexpr int UP_SMEM = 1024 + UP_STAGE + 128;
constexpr int UP_THREADS = 256;                  // warp 0 TMA, 1 MMA, 2 TMEM, 4-7 epilogue
constexpr int XD = PW * PW + PW;                 // X and 1 / d of a panel, per matrix
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_SMEM = DiagSmem::ELEMS * (int)sizeof(float2);
constexpr int ROWS_THREADS = 128;                // 64 rows x 64 columns per CTA
constexpr int ROWS_SMEM = (XD + 64 * LDP) * (int)sizeof(float2);
static_assert(TM * TN * 8 <= UP_STAGE, "the target tile fits in the stage");

constexpr int KW = 2 * PW;  // K width of the planes: two panels

struct UpParams {
  CUtensorMap a[4];  // Ar_hi, Ai_hi, Ar_lo, Ai_lo  [F * nrow][KW]
  CUtensorMap b[4];  // Lr_hi, Li_hi, Lr_lo, Li_lo  [F * n][KW]
  CUtensorMap c;     // targets: (2n FP32 along a row, nrow rows, F matrices)
  int n, nrow, R0, F, tiles;
  int nkc;           // 32-wide K chunks of this update (2: one panel, 4: two)
  int one_col;       // lookahead: only the column tile [R0, R0 + 64)
  const int* active;
  unsigned* status;
  unsigned long long wait_ns;
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* tm, int x, int y, int z, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(tm)),
               "r"(x), "r"(y), "r"(z), "r"(src)
               : "memory");
}

// the diagonal block of panel k0 of every matrix (one CTA each); X = L^-1 as xg[l][c] = X_cl and 1 / d to `xd` for the rows below
__global__ void __launch_bounds__(DIAG_THREADS)
    ldlt_diag_kernel(float2* __restrict__ mats, int n, long long ldm, long long stride, int k0, const int* __restrict__ active,
                     float2* __restrict__ xd, unsigned* __restrict__ status) {
  const int f = blockIdx.x;
  if (active && !active[f]) return;
  const DiagSmem ds{0};
  __shared__ int sing;
  if (threadIdx.x == 0) sing = 0;
  const int kb = min(PW, n - k0);
  factor_diag_block<DIAG_THREADS>(mats + f * stride, ldm, k0, kb, ds, &sing, false);
  float2* o = xd + (size_t)f * XD;
  for (int e = threadIdx.x; e < PW * PW; e += DIAG_THREADS) {
    const int l = e >> 6, c = e & 63;
    o[e] = (c >= l && c < kb) ? ds.xr(c, l) : make_float2(0.f, 0.f);
  }
  if (threadIdx.x < PW) o[PW * PW + threadIdx.x] = threadIdx.x < kb ? ds.dinv(threadIdx.x) : make_float2(0.f, 0.f);
  if (threadIdx.x == 0 && sing) atomicOr(status, kStatSingular);
}

// four columns of a row as TF32 hi and lo planes (re hi, im hi, re lo, im lo)
__device__ __forceinline__ void store_planes(float* __restrict__ o, size_t plane, const float2 (&v)[4]) {
  const float re[4] = {v[0].x, v[1].x, v[2].x, v[3].x}, im[4] = {v[0].y, v[1].y, v[2].y, v[3].y};
  float4 rh, rl, ih, il;
  split4(re, rh, rl);
  split4(im, ih, il);
  *reinterpret_cast<float4*>(o) = rh;
  *reinterpret_cast<float4*>(o + plane) = ih;
  *reinterpret_cast<float4*>(o + 2 * plane) = rl;
  *reinterpret_cast<float4*>(o + 3 * plane) = il;
}

// Rows below panel k0, 64 per CTA (blockIdx.x) of matrix blockIdx.y: W = A X^T, stored to A, and the TF32 hi / lo planes of W
// (rows i) and of L = W D^-1 (the rows that are columns of the trailing matrix, j < n) that the update reads, K-major at K
// column koff. Warp w takes the 32-row block w / 2 and the column groups {0, 3} or {1, 2} (equal work: the triangle of X).
// The rows were the panel CTA's second half, 192 at a time on one SM per matrix (21 us each), and the planes a kernel
// of their own: 8 matrices of N_aux 2450, panels and planes of a factorisation 7.1 ms, diagonal blocks and rows now 1.4 ms;
// 64 matrices of N_aux 1100 2.2 and 0.95 ms. With many matrices the planes' traffic (8 floats per complex value) bounds it: W goes
// through shared memory so that every plane is written in whole 256-byte row segments (0.94 -> 0.54 ms for the 64).
__global__ void __launch_bounds__(ROWS_THREADS)
    ldlt_rows_kernel(float2* __restrict__ mats, int n, int nrow, long long ldm, long long stride, int k0, int koff,
                     const int* __restrict__ active, const float2* __restrict__ xd, float* __restrict__ ap,
                     float* __restrict__ bp) {
  const int f = blockIdx.y;
  if (active && !active[f]) return;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  float2* xg = reinterpret_cast<float2*>(smem_raw);                        // [64][64], then dinv [64]
  float2(*ach)[LDP] = reinterpret_cast<float2(*)[LDP]>(xg + XD);           // [64][65]
  float2* A = mats + f * stride;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kb = min(PW, n - k0), base = k0 + kb + 64 * blockIdx.x;  // (with columns beyond it, the panel is 64 wide)
  const float2* src = xd + (size_t)f * XD;
  for (int e = tid; e < XD / 2; e += ROWS_THREADS) cp_async16(xg + 2 * e, src + 2 * e, true);
  for (int e = tid; e < 64 * PW; e += ROWS_THREADS) {
    const int rr = e >> 6, l = e & 63, i = base + rr;
    if (i < nrow && l < kb) cp_async_elem<8>(&ach[rr][l], A + (long long)i * ldm + k0 + l);
  }
  cp_commit();
  cp_wait<0>();
  __syncthreads();
  const float2* dinv = xg + PW * PW;
  const int r = 32 * (warp >> 1) + lane;
  const float2* arow = ach[r];
  float2 w[4][8];
#pragma unroll
  for (int pass = 0; pass < 4; ++pass) {  // 8 columns each: 16 float2 accumulators
    const int g = (warp & 1) ? 1 + (pass >> 1) : 3 * (pass >> 1);
    const int c0 = 16 * g + 8 * (pass & 1), lmax = c0 < kb ? min(c0 + 8, kb) : 0;  // X_cl = 0 for l > c
    float2 pr[8], pi[8];  // pr[c] = sum a.re (X re, X im), pi[c] = sum a.im (X re, X im)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      pr[c] = make_float2(0.f, 0.f);
      pi[c] = make_float2(0.f, 0.f);
    }
#pragma unroll 4
    for (int l = 0; l < lmax; ++l) {
      const float2 a = arow[l];
      const float2 ar = make_float2(a.x, a.x), ai = make_float2(a.y, a.y);
      const float4* xp = reinterpret_cast<const float4*>(xg + l * PW + c0);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 x = xp[q];
        const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
        pr[2 * q] = __ffma2_rn(ar, x0, pr[2 * q]);
        pi[2 * q] = __ffma2_rn(ai, x0, pi[2 * q]);
        pr[2 * q + 1] = __ffma2_rn(ar, x1, pr[2 * q + 1]);
        pi[2 * q + 1] = __ffma2_rn(ai, x1, pi[2 * q + 1]);
      }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) w[pass][c] = make_float2(pr[c].x - pi[c].y, pr[c].y + pi[c].x);
  }
  __syncthreads();  // the rows of A have been read: W takes their place, then goes out in whole row segments
#pragma unroll
  for (int pass = 0; pass < 4; ++pass) {
    const int c0 = 16 * ((warp & 1) ? 1 + (pass >> 1) : 3 * (pass >> 1)) + 8 * (pass & 1);
#pragma unroll
    for (int c = 0; c < 8; ++c) ach[r][c0 + c] = w[pass][c];
  }
  __syncthreads();
  const size_t a_plane = (size_t)gridDim.y * nrow * KW, b_plane = (size_t)gridDim.y * n * KW;
  for (int e = tid; e < 64 * 16; e += ROWS_THREADS) {
    const int rr = e >> 4, c = 4 * (e & 15), i = base + rr;
    if (i >= nrow || c >= kb) continue;
    float2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = ach[rr][c + q];
    float2* o = A + (long long)i * ldm + k0 + c;
    if (c + 4 <= kb) {
      *reinterpret_cast<float4*>(o) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
      *reinterpret_cast<float4*>(o + 2) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (c + q < kb) o[q] = v[q];
    }
    if (!ap) continue;  // the last panel: no trailing matrix
    store_planes(ap + ((size_t)f * nrow + i) * KW + koff + c, a_plane, v);
    if (i < n) {
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = cmul_rn(v[q], dinv[c + q]);
      store_planes(bp + ((size_t)f * n + i) * KW + koff + c, b_plane, v);
    }
  }
}

__global__ void __launch_bounds__(UP_THREADS, 2) ldlt_update_kernel(const __grid_constant__ UpParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + UP_STAGE);
  uint64_t* empty = full + 1;
  uint64_t* done = full + 2;
  uint64_t* c_full = full + 3;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(full + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int f = blockIdx.x / p.tiles;
  int t = blockIdx.x - f * p.tiles;
  if (f >= p.F || (p.active && !p.active[f])) return;  // uniform, before any barrier or TMEM use
  int tI = 0;
  if (p.one_col) {  // lookahead: row tile t, the column tile [R0, R0 + 64)
    tI = t;
    t = 0;
  } else {
    for (;;) {  // (row tile, column tile) of tile t of the trailing lower part
      const int nc = tile_cols(p.R0, p.n, tI);
      if (t < nc) break;
      t -= nc;
      ++tI;
    }
  }
  const int i0 = p.R0 + TM * tI, j0 = p.R0 + TN * t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(smem_u32(full), 1);
    mbar_init(smem_u32(empty), 1);
    mbar_init(smem_u32(done), 1);
    mbar_init(smem_u32(c_full), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int kc = 0; kc < p.nkc; ++kc) {  // one stage, reused by every chunk
        if (kc > 0 && !mbar_wait(smem_u32(empty), (uint32_t)(kc - 1) & 1, abort_flag, p.wait_ns)) break;
        mbar_expect_tx(smem_u32(full), UP_STAGE);
        const int ay = f * p.nrow + i0, by = f * p.n + j0;
        for (int q = 0; q < 4; ++q) tma_load_2d(smem_u32(base + q * UP_A), &p.a[q], KH * kc, ay, smem_u32(full));
        for (int q = 0; q < 4; ++q) tma_load_2d(smem_u32(base + 4 * UP_A + q * UP_B), &p.b[q], KH * kc, by, smem_u32(full));
        issued = kc + 1;
      }
      if (issued > 0) mbar_drain(smem_u32(full), (uint32_t)(issued - 1) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t st = smem_u32(base);
      const uint64_t dar = sdesc(st), dai = sdesc(st + UP_A), darl = sdesc(st + 2 * UP_A), dail = sdesc(st + 3 * UP_A);
      const uint64_t dbh = sdesc(st + 4 * UP_A), dbl = sdesc(st + 4 * UP_A + 2 * UP_B);  // [Lr; Li] hi, lo
      const uint32_t dp = tmem, dq = tmem + 128;
      bool committed = false;  // `done` takes exactly one commit (a second would flip its phase back)
      for (int kc = 0; kc < p.nkc; ++kc) {
        if (!mbar_wait(smem_u32(full), (uint32_t)kc & 1, abort_flag, p.wait_ns)) break;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < KH / 8; ++k) {
          const uint64_t o = 2u * k;
          const uint32_t acc = (kc == 0 && k == 0) ? 0u : 1u;
          mma_tf32(dp, dar + o, dbh + o, acc);
          mma_tf32(dp, dar + o, dbl + o, 1u);
          mma_tf32(dp, darl + o, dbh + o, 1u);
          mma_tf32(dq, dai + o, dbh + o, acc);
          mma_tf32(dq, dai + o, dbl + o, 1u);
          mma_tf32(dq, dail + o, dbh + o, 1u);
        }
        if (kc + 1 < p.nkc) {
          mma_commit(smem_u32(empty));
        } else {
          mma_commit(smem_u32(done));
          committed = true;
        }
      }
      if (!committed) mma_commit(smem_u32(done));  // after an early stop: fires once the issued MMAs complete
    }
  } else if (warp >= 4) {
    // ---- epilogue: C -= (P_re - Q_im, P_im + Q_re) through shared memory -------------------------
    const int q = warp & 3, r = 32 * q + lane;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(done), 0, abort_flag, p.wait_ns));
    tc_fence_after();
    bool landed = false;
    if (ok && !*abort_flag) {
      if (threadIdx.x == 128) {
        mbar_expect_tx(smem_u32(c_full), TM * TN * 8);
        for (int b = 0; b < 4; ++b) tma_load_3d(smem_u32(base + b * UP_A), &p.c, 2 * j0 + 32 * b, i0, f, smem_u32(c_full));
      }
      landed = __all_sync(0xffffffffu, mbar_wait(smem_u32(c_full), 0, abort_flag, p.wait_ns));
      if (landed) {
        const uint32_t lb = tmem + ((uint32_t)(32 * q) << 16);
        for (int c4 = 0; c4 < 4; ++c4) {  // complex columns 16 c4 .. + 15: box c4 of the staged tile
          uint32_t pr[16], pi[16], qr[16], qi[16];
          tmem_ld16_nw(lb + 16 * c4, pr);        // Ar Lr^T
          tmem_ld16_nw(lb + 64 + 16 * c4, pi);   // Ar Li^T
          tmem_ld16_nw(lb + 128 + 16 * c4, qr);  // Ai Lr^T
          tmem_ld16_nw(lb + 192 + 16 * c4, qi);  // Ai Li^T
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          uint8_t* rowp = base + c4 * UP_A + r * 128;
#pragma unroll
          for (int ch = 0; ch < 8; ++ch) {  // 16-byte chunk ch: complex columns 2 ch, 2 ch + 1
            float4* cp = reinterpret_cast<float4*>(rowp + ((ch ^ (r & 7)) << 4));
            float4 v = *cp;
            const int e0 = 2 * ch, e1 = 2 * ch + 1;
            v.x -= __uint_as_float(pr[e0]) - __uint_as_float(qi[e0]);
            v.y -= __uint_as_float(pi[e0]) + __uint_as_float(qr[e0]);
            v.z -= __uint_as_float(pr[e1]) - __uint_as_float(qi[e1]);
            v.w -= __uint_as_float(pi[e1]) + __uint_as_float(qr[e1]);
            *cp = v;
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");  // every epilogue warp, whatever its waits gave
    if (threadIdx.x == 128) {
      if (landed && !*abort_flag) {
        for (int b = 0; b < 4; ++b) tma_store_3d(&p.c, 2 * j0 + 32 * b, i0, f, smem_u32(base + b * UP_A));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      } else if (ok) {
        mbar_drain(smem_u32(c_full), 0);
      }
    }
  }
  if (warp == 2) {
    if (lane == 0) mbar_drain(smem_u32(done), 0);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, kStatTimeout);
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
  }
}

int host_tile_cols(int R0, int n, int tI) {
  const int jmax = std::min(n, R0 + TM * tI + TM);
  return (jmax - R0 + TN - 1) / TN;
}

}  // namespace

int launch_ldlt_tc_grouped(const LdltGroup* d_groups, int n_groups, int n_ctas, unsigned* status,
                           unsigned long long wait_ns, cudaStream_t s) {
  if (!tc_supported()) return -2;
  if (n_groups < 1 || n_ctas < 1) return -1;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_tc_grouped_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_TC) != cudaSuccess)
      return -1;
    attr = true;
  }
  ldlt_tc_grouped_kernel<<<n_ctas, NT_TC, SMEM_TC, s>>>(d_groups, n_groups, status, wait_ns);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

// Returns 1 (launches), -1 on a launch error or bad layout, -2 if the device has no tcgen05.
int launch_ldlt_tc(void* mats, int n, int nrow, long long ldm, long long stride, int F, const int* active,
                   unsigned* status, unsigned long long wait_ns, cudaStream_t s) {
  if (!tc_supported()) return -2;
  // 16-byte loads and stores: ldm and the matrix stride multiples of 4 complex values (32 B)
  if ((ldm % 4) || (stride % 4) || (reinterpret_cast<uintptr_t>(mats) & 15) || nrow < n || n < 1) return -1;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_TC) != cudaSuccess)
      return -1;
    attr = true;
  }
  ldlt_tc_kernel<<<F, NT_TC, SMEM_TC, s>>>(reinterpret_cast<float2*>(mats), n, nrow, ldm, stride, active, status,
                                                wait_ns);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

size_t ldlt_split_bytes(int n, int nrow, int F) {
  return (size_t)16 * F * KW * ((size_t)nrow + n) + (size_t)F * XD * sizeof(float2) + 1024;
}

// Returns the launches, -1 on a launch error or bad layout, -2 if unsupported.
int launch_ldlt_split(void* mats, int n, int nrow, long long ldm, long long stride, int F, const int* active,
                      unsigned* status, unsigned long long wait_ns, void* work, size_t work_bytes, cudaStream_t s) {
  if (!tc_supported()) return -2;
  if ((ldm % 4) || (stride % 4) || (reinterpret_cast<uintptr_t>(mats) & 15) || nrow < n || n < 1 || F < 1) return -1;
  if (ldlt_split_bytes(n, nrow, F) > work_bytes || (reinterpret_cast<uintptr_t>(work) & 15)) return -2;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(ldlt_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DIAG_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(ldlt_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ROWS_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(ldlt_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, UP_SMEM) != cudaSuccess)
      return -1;
    attr = true;
  }
  float* ap = static_cast<float*>(work);
  float* bp = ap + (size_t)4 * F * nrow * KW;
  float2* xd = reinterpret_cast<float2*>(bp + (size_t)4 * F * n * KW);
  UpParams p;
  std::memset(static_cast<void*>(&p), 0, sizeof(p));
  for (int q = 0; q < 4; ++q) {
    if (!make_map(&p.a[q], ap + (size_t)q * F * nrow * KW, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, F * nrow, KW, KH, TM) ||
        !make_map(&p.b[q], bp + (size_t)q * F * n * KW, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, F * n, KW, KH, TN))
      return -2;
  }
  {
    EncodeTiledFn enc = encoder();
    if (!enc) return -2;
    cuuint64_t dims[3] = {(cuuint64_t)2 * n, (cuuint64_t)nrow, (cuuint64_t)F};
    cuuint64_t strides[2] = {(cuuint64_t)ldm * 8, (cuuint64_t)stride * 8};
    cuuint32_t box[3] = {32, (cuuint32_t)TM, 1};
    cuuint32_t es[3] = {1, 1, 1};
    if (enc(&p.c, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, mats, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return -2;
  }
  p.n = n;
  p.nrow = nrow;
  p.F = F;
  p.active = active;
  p.status = status;
  p.wait_ns = wait_ns;
  float2* A = reinterpret_cast<float2*>(mats);
  int launches = 0;
  // panel k0; its planes (unless it is the last one) at K column koff
  auto panel = [&](int k0, int koff) {
    const int R0 = k0 + std::min(PW, n - k0);
    ldlt_diag_kernel<<<F, DIAG_THREADS, DIAG_SMEM, s>>>(A, n, ldm, stride, k0, active, xd, status);
    ++launches;
    if (R0 >= nrow) return;
    ldlt_rows_kernel<<<dim3((nrow - R0 + 63) / 64, F), ROWS_THREADS, ROWS_SMEM, s>>>(
        A, n, nrow, ldm, stride, k0, koff, active, xd, R0 < n ? ap : nullptr, R0 < n ? bp : nullptr);
    ++launches;
  };
  auto update = [&](int R0, int nkc, bool one_col) {
    const int n_ti = (nrow - R0 + TM - 1) / TM;
    int tiles = 0;
    if (one_col) {
      tiles = n_ti;
    } else {
      for (int tI = 0; tI < n_ti; ++tI) tiles += host_tile_cols(R0, n, tI);
    }
    p.R0 = R0;
    p.tiles = tiles;
    p.nkc = nkc;
    p.one_col = one_col ? 1 : 0;
    ldlt_update_kernel<<<F * tiles, UP_THREADS, UP_SMEM, s>>>(p);
    ++launches;
  };
  for (int k0 = 0; k0 < n;) {
    // panel p at k0, with the planes of its W columns and L rows in K columns 0..63
    const int R0 = k0 + std::min(PW, n - k0);
    panel(k0, 0);
    if (R0 >= n) break;
    // lookahead: panel p's update of panel p + 1's columns only, then panel p + 1
    update(R0, PW / KH, true);
    panel(R0, PW);
    const int R1 = R0 + std::min(PW, n - R0);
    if (R1 < n) {
      update(R1, KW / KH, false);  // both panels: K = 128
    }
    if (cudaPeekAtLastError() != cudaSuccess) return -1;
    k0 = R1;
  }
  if (cudaPeekAtLastError() != cudaSuccess) return -1;
  return launches;
}

}  // namespace gwc
