// FP64 polarizability on the tensor cores, by exact products of 8-bit digits (sm_103a: tcgen05 + TMEM + TMA).
//
//   Pi_PQ(z_f) = sum_k O_Pk (D_f(k) O_Qk)      (RI polarizability, Sec. "Self-energy evaluation")
//
// FP64 arithmetic runs at 1.2 TFLOP/s on this part and bounded the SIMT form (chi0_simt.cu). Here every row of O and of the
// scaled operand D O (one FP64 product per element, as in the SIMT form) is written as 79-bit fixed-point numbers under the
// row's own exponent, X = sum_{k<10} a_k 256^k with digits a_k in [-128, 127], which BF16 holds exactly (splitting into exact
// products: Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012). The digit pairs of one order u = k + l are products
// of small integers whose sums over up to 1024 terms stay below 2^24, so the FP32 accumulator of the tensor core is
// exact; the orders 9 .. 18 are kept (55 pairs).
//
// Accuracy. In units of the rows' maxima M_P, M_Q (their powers of two) the orders dropped and the rounding to fixed point come to
// sqrt(N_ov) 2^-76 per element for digits that look random, and to at most N_ov 10.1 2^-76 for any. That is relative to M_P M_Q
// and not to what the element sums, S_PQ = sum_k |O_Pk D_k O_Qk|, which is far smaller where one row's maximum meets a zero
// of the other (D near a pole that P does not see, rows that hardly overlap). So S is formed as well, as one more pair of
// planes that hold the magnitudes as BF16 rounded down, and an element with S < 16 sqrt(N_ov) 2^-22 M_P M_Q is summed in FP64
// instead, by a warp. What remains is 1/16 of 2^-54 S as a rule and 0.64 sqrt(N_ov) 2^-54 S at most, with the rounding of the
// FP64 product and those of the four group sums below, under 10.3 2^-53 S; the sequential FP64 sum may err by N_ov 2^-53 S.
// (With eight digits, 36 pairs and no such check, elements of Im Pi near a pole erred by up to 175 2^-53 S at N_ov 1639,
// eta 1e-3, and more at smaller eta, where the sequential sum's worst was 24 2^-53 S.)
//
//   digits_kernel   row exponents, then the ten BF16 digit planes and the magnitudes [plane][row][k] of O (once per loaded
//                   system) or of D O (per frequency part, in chunks of the workspace): integer arithmetic but for the product;
//   fixed_gemm_kernel  one 128 x 128 tile of the lower triangle per CTA, order by order: TMA-fed digit tiles, four MMAs
//                   per digit pair and 64-wide chunk into one of two fresh accumulators; segments of at most 1024 terms
//                   are added, as integers, to a 64-bit sum in TMEM by the fold warps while the next segment runs; after
//                   the orders (9, 10, 11), (12, 13, 14), (15, 16, 17) and 18 that sum becomes FP64 and is added to the
//                   result. The magnitudes come last, as one segment.
//
// Rows with an infinity or NaN (a frequency on a pole) take the FP64 sum, element by element.
// Every mbarrier wait is bounded (the context's bound); on expiry the CTA records kStatTimeout, drains its copies and MMAs
// and frees TMEM.
// Measured, digits and products: 8 frequencies of N_aux 1100, N_ov 5859, 12.9 ms (SIMT form 137); 3133 frequencies of N_aux 200, N_ov
// 416, 44.8 ms (SIMT form 223). The digit tiles' way into shared memory bounds it (32 KB per pair and chunk; the MMAs alone
// would take 0.4 of the time). Eight digits and 36 pairs took 7.6 and 29.9 ms. W from it, against quad precision over 54
// frequencies of nine systems: geometric mean 6.4e-16 (1.03e-15 with the SIMT form), largest 3.1e-14 (4.3e-14).
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "gwc_internal.h"
#include "tc_common.cuh"

namespace gwc {

namespace {

constexpr int ND = 10;                   // digits
constexpr int NPL = ND + 1;              // planes: the digits, then the magnitudes
constexpr int U0 = ND - 1, U1 = 2 * ND - 2;  // orders kept
constexpr int FT = 128;                  // tile rows and columns
constexpr int FK = 64;                   // k per chunk (128-byte rows of BF16)
constexpr int FTILE = FT * FK * 2;       // 16 KB
constexpr int FST = 6;                   // ring stages, one digit pair each (A tile, B tile)
constexpr int FTHREADS = 256;            // warp 0 TMA, 1 MMA, 2 TMEM, 4-7 fold
constexpr int FSMEM = 1024 + FST * 2 * FTILE + 256;
constexpr int kTerms = 1024;             // 128 * 128 * 1024 = 2^24
constexpr int kMaxOv = 200000;           // the 64-bit sums stay below 2^51: k 2^14 (10 + 9 2^8 + 8 2^16)
constexpr int kNotFinite = 0x7ff, kZeroRow = -1;

constexpr uint32_t kIdescF = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FT >> 3) << 17) | ((uint32_t)(FT >> 4) << 24);

__device__ __forceinline__ void mma_digits(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(kIdescF), "r"(acc));
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_st16_u(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
      "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

// Fixed point of x under the row's exponent field e (the largest of the row): X = x 2^(78 + 1022 - e) rounded to nearest,
// |X| <= 2^78, with 128 added to every byte: byte k is a_k + 128 (the lower eight in lo, the upper two in the lower half of hi).
// The upper half of hi is |x| 2^(1023 - e) as BF16, rounded down (zero below 2^-126).
struct Fixed {
  unsigned long long lo;
  uint32_t hi;
};
__device__ __forceinline__ Fixed fixed_of(double x, int e) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)(bits >> 52) & 0x7ff;
  const unsigned long long m = (bits & 0xfffffffffffffull) | (ef ? 0x10000000000000ull : 0ull);
  const int s = max(ef, 1) - e + 25;
  unsigned long long lo, hi = 0;
  if (s > 0) {  // at most 25 (26 in a row of denormals)
    lo = m << s;
    hi = m >> (64 - s);
  } else {
    lo = s == 0 ? m : s < -54 ? 0ull : (m + (1ull << (-s - 1))) >> (-s);
  }
  if ((long long)bits < 0) {
    lo = 0ull - lo;
    hi = ~hi + (lo == 0);
  }
  Fixed r;
  r.lo = lo + 0x8080808080808080ull;
  const int me = ef - e + 127;
  const uint32_t mag = ef && me > 0 ? ((uint32_t)me << 7) | (uint32_t)(bits >> 45 & 0x7f) : 0u;
  r.hi = (((uint32_t)hi + 0x8080u + (r.lo < lo)) & 0xffffu) | mag << 16;
  return r;
}

// Row blockIdx.x of part blockIdx.y: part zp = zp0 + y of frequency zp / parts scales O by D (dtab null: O itself). ex[y][row] =
// exponent field of the row's largest element (kNotFinite: some element is not finite; kZeroRow: all are zero);
// dig[y][plane][row][k].
__global__ void __launch_bounds__(256) digits_kernel(const double* __restrict__ o, int n_aux, int n_ov, int n_ov_pad, int row0,
                                                      int rows, const double* __restrict__ dtab, int ld_dtab, int parts, int zp0,
                                                      const int* __restrict__ active, __nv_bfloat16* __restrict__ dig,
                                                      int* __restrict__ ex) {
  const int r = blockIdx.x, P = row0 + r, f = (zp0 + (int)blockIdx.y) / parts, part = (zp0 + (int)blockIdx.y) % parts;
  if (active && !active[f]) return;
  const int tid = threadIdx.x;
  const double* d = dtab ? dtab + ((size_t)f * 2 + part) * ld_dtab : nullptr;
  const double* row = o + (size_t)P * n_ov;
  auto value = [&](int k) { return d ? row[k] * d[k] : row[k]; };
  int e = kZeroRow;
  if (P < n_aux)
    for (int k = tid; k < n_ov; k += 256) {
      const long long b = __double_as_longlong(value(k)) & 0x7fffffffffffffffll;
      if (b) e = max(e, (int)(b >> 52));
    }
  __shared__ int red[8];
  e = __reduce_max_sync(0xffffffffu, e);
  if ((tid & 31) == 0) red[tid >> 5] = e;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) e = max(e, red[w]);
  if (tid == 0) ex[(size_t)blockIdx.y * rows + r] = e;
  e = max(e, 0);
  uint8_t* out = reinterpret_cast<uint8_t*>(dig) + (((size_t)blockIdx.y * NPL) * rows + r) * (size_t)n_ov_pad * 2;
  const size_t plane = (size_t)rows * n_ov_pad * 2;
  for (int k0 = 8 * tid; k0 < n_ov_pad; k0 += 8 * 256) {
    Fixed x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      x[q].lo = 0x8080808080808080ull;
      x[q].hi = 0x8080u;
      if (P < n_aux && k0 + q < n_ov) x[q] = fixed_of(value(k0 + q), e);
    }
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t u[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // digit as FP32: 2^23 + byte, minus 2^23 + 128; its upper half is the BF16
          const Fixed& y = x[2 * q + h];
          const uint32_t word = k < 4 ? (uint32_t)y.lo : k < 8 ? (uint32_t)(y.lo >> 32) : y.hi;
          u[h] = __float_as_uint(__uint_as_float(0x4b000000u | ((word >> (8 * (k & 3))) & 0xffu)) - 8388736.0f);
        }
        w[q] = __byte_perm(u[0], u[1], 0x7632);
      }
      *reinterpret_cast<uint4*>(out + k * plane + (size_t)k0 * 2) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = __byte_perm(x[2 * q].hi, x[2 * q + 1].hi, 0x7632);
    *reinterpret_cast<uint4*>(out + ND * plane + (size_t)k0 * 2) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

struct FixedParams {
  CUtensorMap a, b;      // planes of O [NPL * n_aux_pad][n_ov_pad], of D O [zps * NPL * b_rows][n_ov_pad]; boxes 64 x 128
  const int* ea;         // [n_aux_pad]
  const int* eb;         // [zps][b_rows]
  const double* o;       // FP64 rows and factors, for the elements summed in FP64
  const double* dtab;
  int n_ov, ld_dtab;
  int n_aux, n_aux_pad;
  int b_row0, b_rows;    // the rows of Q in the B digits
  int n_kc;
  int n_pb;              // 128-row blocks of P
  int zp0, parts;
  float s_min;           // least sum of magnitudes that the digits are good for
  double alpha, beta;
  double* out;           // element (P, Q) of matrix f at out[(f mat_stride + P ldm + Q) parts + part]
  long long ldm, mat_stride;
  const int* active;
  unsigned* status;
  unsigned long long wait_ns;
};

// 2^(e - 1028): the unit of a row with exponent field e (the sums carry 2^144)
__device__ __forceinline__ double row_unit(int e) {
  return e > 5 && e < kNotFinite ? __hiloint2double((e - 5) << 20, 0) : scalbn(1.0, e - 1028);
}

// Orders in the sequence of the sums: U0 .. U1, order u of 2 ND - 1 - u plane pairs (k from u - U0 on, the other u - k), in segments of
// seg_chunks(u) chunks, then "order" U1 + 1, the magnitudes in one segment.
__device__ __forceinline__ int pairs_of(int u) { return u > U1 ? 1 : 2 * ND - 1 - u; }
__device__ __forceinline__ int plane_a(int u, int i) { return u > U1 ? ND : u - U0 + i; }
__device__ __forceinline__ int plane_b(int u, int i) { return u > U1 ? ND : U0 - i; }
__device__ __forceinline__ int seg_chunks(int u) { return u > U1 ? kMaxOv : kTerms / FK / pairs_of(u); }
static_assert(kTerms / FK / ND >= 1, "a chunk of the lowest order fits in a segment");

// sum_k O_Pk D_k O_Qk in FP64 by a warp, eight partial sums per lane
__device__ __forceinline__ double warp_sum(const double* __restrict__ op, const double* __restrict__ oq,
                                           const double* __restrict__ d, int n) {
  double a[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int k = threadIdx.x & 31;
  for (; k + 224 < n; k += 256)
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = fma(op[k + 32 * q], oq[k + 32 * q] * d[k + 32 * q], a[q]);
  for (; k < n; k += 32) a[0] = fma(op[k], oq[k] * d[k], a[0]);
  double r = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

__global__ void __launch_bounds__(FTHREADS, 1) fixed_gemm_kernel(const __grid_constant__ FixedParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + FST * 2 * FTILE);
  uint64_t* empty = full + FST;
  uint64_t* seg_full = empty + FST;   // [2] fresh accumulator complete
  uint64_t* seg_free = seg_full + 2;  // [2] folded
  uint64_t* done = seg_free + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int zp = p.zp0 + blockIdx.y, f = zp / p.parts, part = zp % p.parts;
  if (p.active && !p.active[f]) return;  // uniform, before any barrier or TMEM use
  int t = blockIdx.x, iq = p.b_row0 / FT;  // tile t: Q blocks of this launch in order, P blocks iq .. n_pb - 1 of each
  while (t >= p.n_pb - iq) {
    t -= p.n_pb - iq;
    ++iq;
  }
  const int P0 = (iq + t) * FT, Q0 = iq * FT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < FST; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&seg_full[i]), 1);
      mbar_init(smem_u32(&seg_free[i]), 4);
    }
    mbar_init(smem_u32(done), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;  // columns: fresh 0, fresh 1, low and high words of the 64-bit sums

  if (warp == 0) {
    if (lane == 0) {
      int n = 0;
      bool ok = true;
      const int by = (int)blockIdx.y * NPL * p.b_rows + (Q0 - p.b_row0);
      for (int u = U0; u <= U1 + 1 && ok; ++u)
        for (int c0 = 0; c0 < p.n_kc && ok; c0 += seg_chunks(u))
          for (int kc = c0; kc < min(p.n_kc, c0 + seg_chunks(u)) && ok; ++kc)
            for (int i = 0; i < pairs_of(u); ++i, ++n) {
              const int s = n % FST;
              ok = mbar_wait(smem_u32(&empty[s]), ((uint32_t)(n / FST) & 1) ^ 1, abort_flag, p.wait_ns);
              if (!ok) break;
              mbar_expect_tx(smem_u32(&full[s]), 2 * FTILE);
              uint8_t* st = base + s * 2 * FTILE;
              tma_load_2d(smem_u32(st), &p.a, kc * FK, plane_a(u, i) * p.n_aux_pad + P0, smem_u32(&full[s]));
              tma_load_2d(smem_u32(st + FTILE), &p.b, kc * FK, by + plane_b(u, i) * p.b_rows, smem_u32(&full[s]));
            }
      for (int c = n > FST ? n - FST : 0; c < n; ++c) mbar_drain(smem_u32(&full[c % FST]), (uint32_t)(c / FST) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int n = 0, seg = 0;
      bool ok = true;
      for (int u = U0; u <= U1 + 1 && ok; ++u)
        for (int c0 = 0; c0 < p.n_kc && ok; c0 += seg_chunks(u), ++seg) {
          const uint32_t d = tmem + (uint32_t)((seg & 1) * FT);
          if (seg >= 2) ok = mbar_wait(smem_u32(&seg_free[seg & 1]), (uint32_t)((seg >> 1) - 1) & 1, abort_flag, p.wait_ns);
          tc_fence_after();
          uint32_t acc = 0;
          for (int kc = c0; kc < min(p.n_kc, c0 + seg_chunks(u)) && ok; ++kc)
            for (int i = 0; i < pairs_of(u); ++i, ++n) {
              const int s = n % FST;
              ok = mbar_wait(smem_u32(&full[s]), (uint32_t)(n / FST) & 1, abort_flag, p.wait_ns);
              if (!ok) break;
              tc_fence_after();
              const uint32_t st = smem_u32(base + s * 2 * FTILE);
              const uint64_t da = sdesc(st), db = sdesc(st + FTILE);
#pragma unroll
              for (int q = 0; q < FK / 16; ++q) {
                mma_digits(d, da + 2u * q, db + 2u * q, acc);
                acc = 1;
              }
              mma_commit(smem_u32(&empty[s]));
            }
          if (ok) mma_commit(smem_u32(&seg_full[seg & 1]));
        }
      mma_commit(smem_u32(done));
    }
  } else if (warp >= 4) {
    // ---- fold and epilogue: a TMEM lane (row of P) per thread ---------------------------------------
    const int q = warp & 3, P = P0 + 32 * q + lane;
    const uint32_t lb = tmem + ((uint32_t)(32 * q) << 16);
    const int* eb = p.eb + (size_t)blockIdx.y * p.b_rows + (Q0 - p.b_row0);
    const int ea = p.ea[P];
    const double sa = row_unit(ea);
    double* o = p.out + ((long long)f * p.mat_stride + (long long)P * p.ldm + Q0) * p.parts + part;
    const int jlim = P < p.n_aux ? min(FT, min(p.n_aux, P + 1) - Q0) : 0;  // columns written: the lower triangle
    int seg = 0;
    bool ok = true;
    for (int u = U0; u <= U1 && ok; ++u) {
      const int g = (u - U0) / 3, sh = 8 * ((u - U0) % 3);
      const bool first = sh == 0, last = sh == 16 || u == U1;  // order of its group
      for (int c0 = 0; c0 < p.n_kc && ok; c0 += seg_chunks(u), ++seg) {
        const bool start = first && c0 == 0, end = last && c0 + seg_chunks(u) >= p.n_kc;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&seg_full[seg & 1]), (uint32_t)(seg >> 1) & 1, abort_flag, p.wait_ns));
        if (!ok) break;
        tc_fence_after();
        const uint32_t fr = lb + (uint32_t)((seg & 1) * FT);
#pragma unroll 1
        for (int c = 0; c < FT; c += 16) {
          uint32_t x[16], lo[16], hi[16];
          tmem_ld16_nowait(fr + c, x);
          if (!start) {
            tmem_ld16_nowait(lb + 2 * FT + c, lo);
            tmem_ld16_nowait(lb + 3 * FT + c, hi);
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          long long v[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const long long old = start ? 0 : (long long)(((unsigned long long)hi[j] << 32) | lo[j]);
            v[j] = old + ((long long)__float2int_rn(__uint_as_float(x[j])) << sh);
          }
          if (!end) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              lo[j] = (uint32_t)v[j];
              hi[j] = (uint32_t)((unsigned long long)v[j] >> 32);
            }
            tmem_st16_u(lb + 2 * FT + c, lo);
            tmem_st16_u(lb + 3 * FT + c, hi);
          } else {
            // the group's sum as FP64 (|v| < 2^51: 1.5 2^52 + v is exact), 256^(3 g - 9) of the last group's unit
            const double w = g == 0 ? 0x1p-72 : g == 1 ? 0x1p-48 : g == 2 ? 0x1p-24 : 1.0;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              if (c + j >= jlim) continue;
              const double y = __longlong_as_double(0x4338000000000000ll + v[j]) - 0x1.8p52;
              double* e = o + (long long)(c + j) * p.parts;
              double r = g == 0 ? y * w : fma(y, w, *e);
              if (u == U1) {
                r = (r * sa) * row_unit(eb[c + j]);
                r = p.alpha * r + (part == 0 && P == Q0 + c + j ? p.beta : 0.0);
              }
              *e = r;
            }
          }
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&seg_free[seg & 1]));
      }
    }
    // the sums of magnitudes: elements that they do not cover (or rows that are not finite) are summed in FP64
    if (ok)
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&seg_full[seg & 1]), (uint32_t)(seg >> 1) & 1, abort_flag, p.wait_ns));
    if (ok) {
      tc_fence_after();
      const double* d = p.dtab + ((size_t)f * 2 + part) * p.ld_dtab;
#pragma unroll 1
      for (int c = 0; c < FT; c += 16) {
        uint32_t x[16];
        tmem_ld16_nowait(lb + (uint32_t)((seg & 1) * FT) + c, x);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        uint32_t redo = 0;  // bit j: column c + j of this lane's row
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (c + j >= jlim) continue;
          const int eq = eb[c + j];
          if (ea == kZeroRow || eq == kZeroRow) continue;
          if (ea == kNotFinite || eq == kNotFinite || !(__uint_as_float(x[j]) >= p.s_min)) redo |= 1u << j;
        }
        if (!__any_sync(0xffffffffu, redo)) continue;
#pragma unroll 1
        for (int j = 0; j < 16; ++j) {
          unsigned m = __ballot_sync(0xffffffffu, redo >> j & 1);
          const int Q = Q0 + c + j;
          while (m) {
            const int l = __ffs(m) - 1;
            m &= m - 1;
            const double r = warp_sum(p.o + (size_t)(P0 + 32 * q + l) * p.n_ov, p.o + (size_t)Q * p.n_ov, d, p.n_ov);
            if (lane == l) o[(long long)(c + j) * p.parts] = p.alpha * r + (part == 0 && P == Q ? p.beta : 0.0);
          }
        }
      }
    }
  }
  // every MMA issued has completed before TMEM is freed
  if (warp == 2) {
    if (lane == 0) mbar_drain(smem_u32(done), 0);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, kStatTimeout);
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

}  // namespace

size_t chi0_fixed_digits_bytes(int n_aux_pad, int n_ov_pad) { return (size_t)n_aux_pad * n_ov_pad * 2 * NPL; }

size_t chi0_fixed_work_bytes(int n_ov_pad, long long rows) {
  return (size_t)rows * ((size_t)n_ov_pad * 2 * NPL + sizeof(int)) + 1024;
}

bool chi0_fixed_shape(int n_aux, long long n_ov) { return n_aux >= kFixedMinAux && n_ov >= kFixedMinOv && n_ov <= kMaxOv; }
bool chi0_fixed_fits(int n_aux, long long n_ov) { return chi0_fixed_shape(n_aux, n_ov) && tc_supported(); }

int launch_chi0_digits(const double* o, int n_aux, int n_ov, int n_aux_pad, int n_ov_pad, void* digits, int* ex,
                       cudaStream_t s) {
  digits_kernel<<<dim3(n_aux_pad, 1), 256, 0, s>>>(o, n_aux, n_ov, n_ov_pad, 0, n_aux_pad, nullptr, 0, 1, 0, nullptr,
                                                   static_cast<__nv_bfloat16*>(digits), ex);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_chi0_fixed(bool complex_out, const double* o, const void* digits, const int* ex, int n_aux, int n_aux_pad, int n_ov,
                      int n_ov_pad, const double* dtab, int ld_dtab, int F, double alpha, double beta, void* out, long long ldm,
                      long long mat_stride, const int* active, void* work, size_t work_bytes, unsigned* status,
                      unsigned long long wait_ns, cudaStream_t s) {
  if (!tc_supported()) return -2;
  const int parts = complex_out ? 2 : 1, n_zp = F * parts, n_pb = n_aux_pad / FT;
  // per row of the B digits: the planes and an exponent
  const size_t row = (size_t)n_ov_pad * 2 * NPL + sizeof(int);
  const long long rows_fit = (long long)((work_bytes - 1024) / row);
  if (work_bytes < 1024 || rows_fit < FT || (reinterpret_cast<uintptr_t>(work) & 127) || n_aux_pad % FT || n_ov_pad % FK) return -2;
  const int b_rows = (int)std::min<long long>(n_aux_pad, rows_fit / FT * FT);  // Q rows per launch
  // parts per launch: as many launches as the workspace needs, of about equal size (every launch ends in a partial wave)
  const int zps_max = (int)std::min<long long>(std::min<long long>(n_zp, 65535), std::max<long long>(1, rows_fit / b_rows));
  const int n_run = (n_zp + zps_max - 1) / zps_max, zps = (n_zp + n_run - 1) / n_run;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(fixed_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FSMEM) != cudaSuccess) return -1;
    attr = true;
  }
  FixedParams p;
  std::memset(static_cast<void*>(&p), 0, sizeof(p));
  p.ea = ex;
  p.o = o;
  p.dtab = dtab;
  p.n_ov = n_ov;
  p.ld_dtab = ld_dtab;
  p.n_aux = n_aux;
  p.n_aux_pad = n_aux_pad;
  p.n_kc = n_ov_pad / FK;
  p.n_pb = n_pb;
  p.parts = parts;
  // (1.05: the FP32 sum of the magnitudes, a lower bound but for its rounding)
  p.s_min = (float)(1.05 * 16.0 * std::sqrt((double)n_ov) * 0x1p-22);
  p.alpha = alpha;
  p.beta = beta;
  p.out = static_cast<double*>(out);
  p.ldm = ldm;
  p.mat_stride = mat_stride;
  p.active = active;
  p.status = status;
  p.wait_ns = wait_ns;
  if (!make_map(&p.a, digits, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, NPL * n_aux_pad, n_ov_pad, FK, FT)) return -2;
  int launches = 0;
  for (int r0 = 0; r0 < n_aux_pad; r0 += b_rows) {
    const int rows = std::min(b_rows, n_aux_pad - r0);
    int tiles = 0;
    for (int iq = r0 / FT; iq < (r0 + rows) / FT; ++iq) tiles += n_pb - iq;
    for (int z0 = 0; z0 < n_zp; z0 += zps) {
      const int nz = std::min(zps, n_zp - z0);
      int* eb = reinterpret_cast<int*>(static_cast<char*>(work) + (size_t)nz * rows * n_ov_pad * 2 * NPL);
      digits_kernel<<<dim3(rows, nz), 256, 0, s>>>(o, n_aux, n_ov, n_ov_pad, r0, rows, dtab, ld_dtab, parts, z0, active,
                                                   static_cast<__nv_bfloat16*>(work), eb);
      p.eb = eb;
      p.b_row0 = r0;
      p.b_rows = rows;
      p.zp0 = z0;
      if (!make_map(&p.b, work, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, nz * NPL * rows, n_ov_pad, FK, FT)) return -2;
      fixed_gemm_kernel<<<dim3(tiles, nz), FTHREADS, FSMEM, s>>>(p);
      launches += 2;
      if (cudaPeekAtLastError() != cudaSuccess) return -1;
    }
  }
  return launches;
}

}  // namespace gwc
