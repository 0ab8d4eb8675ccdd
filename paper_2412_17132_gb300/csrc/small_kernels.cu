// Small element-wise kernels of the self-energy path: transition energies, the
// frequency factor table D_ia(z), precision copies of O_ov, right-hand-side gathers,
// the exchange self-energy and output conversion.
#include <algorithm>

#include "gwc_internal.h"

namespace gwc {

namespace {

__global__ void delta_kernel(const double* __restrict__ eps, int n_occ, int n_virt, double* __restrict__ delta) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  long long n = (long long)n_occ * n_virt;
  if (t >= n) return;
  int i = (int)(t / n_virt), a = (int)(t % n_virt);
  delta[t] = eps[n_occ + a] - eps[i];
}

// D_ia(z) = 2[1/(z - Delta) - 1/(z + Delta)] = 4 Delta / (z^2 - Delta^2), z = x + i y.
// (Sec. "Self-energy evaluation": the RI polarizability of the CD method.)
template <typename T>
__global__ void dtable_kernel(const double* __restrict__ z, int F, const double* __restrict__ delta, int n_ov, int ld,
                              T* __restrict__ out) {
  int f = blockIdx.y;
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F || k >= ld) return;
  T* re = out + (size_t)f * 2 * ld;
  T* im = re + ld;
  if (k >= n_ov) {
    re[k] = (T)0;
    im[k] = (T)0;
    return;
  }
  double x = z[2 * f], y = z[2 * f + 1], dl = delta[k];
  double a = (x - dl) * (x + dl) - y * y;  // Re(z^2 - Delta^2)
  double b = 2.0 * x * y;                  // Im(z^2 - Delta^2)
  double s = 4.0 * dl / (a * a + b * b);
  re[k] = (T)(s * a);
  im[k] = (T)(-s * b);
}

__global__ void split_o_kernel(const double* __restrict__ o, int n_aux, int n_ov, int n_aux_pad, int n_ov_pad,
                               __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo, float* __restrict__ f32) {
  long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  long long total = (long long)n_aux_pad * n_ov_pad;
  if (t >= total) return;
  int p = (int)(t / n_ov_pad), k = (int)(t % n_ov_pad);
  double v = (p < n_aux && k < n_ov) ? o[(size_t)p * n_ov + k] : 0.0;
  __nv_bfloat16 h = __double2bfloat16(v);
  double r = v - (double)__bfloat162float(h);
  hi[t] = h;
  lo[t] = __double2bfloat16(r);
  f32[t] = (float)v;
}

// A CTA converts one row for the `share` matrices from blockIdx.y * share on (share > 1: they all take the same row).
template <typename S>
__global__ void rhs_gather_kernel(const double* __restrict__ src, long long src_row_stride, const int* __restrict__ row_of,
                                  int row_f, int F, int share, int r, int n_aux, S* __restrict__ dst, long long ldr,
                                  long long rhs_stride, double* __restrict__ bnorm2) {
  const int f = blockIdx.y * share, f1 = min(F, f + share), q = blockIdx.x;
  long long row = row_of ? row_of[f * r + q] : (long long)f * row_f + q;
  const double* s = src + (size_t)row * src_row_stride;
  S* d = dst + f * rhs_stride + q * ldr;
  double acc = 0.0;
  for (int p = threadIdx.x; p < n_aux; p += blockDim.x) {
    double v = s[p];
    const S e = sfrom<S>(v, 0.0);
    S* o = d + p;
    for (int u = f; u < f1; ++u, o += rhs_stride) *o = e;
    acc += v * v;
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    for (int u = f; u < f1; ++u) bnorm2[u * r + q] = t;
  }
}

// Sigma^x_n = -sum_{i occ} (n i | i n) = -sum_{i occ} sum_P (O^P_{n i})^2  (Eq. sigma_x)
__global__ void sigma_x_kernel(const double* __restrict__ o_core, int n_occ, int n_core, int n_aux, double* __restrict__ sx) {
  int c = blockIdx.x;
  double acc = 0.0;
  long long total = (long long)n_occ * n_aux;
  for (long long t = threadIdx.x; t < total; t += blockDim.x) {
    int i = (int)(t / n_aux), p = (int)(t % n_aux);
    double v = o_core[((size_t)i * n_core + c) * n_aux + p];
    acc += v * v;
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    sx[c] = -t;
  }
}

__global__ void fill_z_pairs_kernel(const double* __restrict__ eps, const int* __restrict__ pair_m,
                                    const double* __restrict__ pair_w, int n_pairs, double eta, double* __restrict__ z) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_pairs) return;
  z[2 * p] = fabs(eps[pair_m[p]] - pair_w[p]);
  z[2 * p + 1] = eta;
}

// Lower triangle of matrix blockIdx.y to a full complex FP64 matrix, one 32 x 32 tile of the lower triangle per CTA: a tile
// is read once and written in rows on both sides of the diagonal (through shared memory; a thread per output element read the
// upper half in columns: two matrices of N_aux 4500 237 us, this 149 us).
constexpr int CTL = 32;

template <typename S>
__global__ void __launch_bounds__(256) mat_to_c128_kernel(const S* __restrict__ m, int n, long long ldm, long long stride,
                                                           double* __restrict__ out, bool pairs) {
  __shared__ S t[CTL][CTL + 1];
  int ip = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((long long)ip * (ip + 1) / 2 > (long long)blockIdx.x) --ip;
  while ((long long)(ip + 1) * (ip + 2) / 2 <= (long long)blockIdx.x) ++ip;
  const int iq = (int)((long long)blockIdx.x - (long long)ip * (ip + 1) / 2);
  const int p0 = ip * CTL, q0 = iq * CTL, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const S* a = m + blockIdx.y * stride;
  double* o = out + (size_t)blockIdx.y * n * n * 2;
  auto store = [&](size_t e, S v) {
    if (pairs) {  // 16-byte aligned output
      reinterpret_cast<double2*>(o)[e] = make_double2(sre(v), sim(v));
    } else {
      o[2 * e] = sre(v);
      o[2 * e + 1] = sim(v);
    }
  };
#pragma unroll
  for (int r = ty; r < CTL; r += 8) {
    const int p = p0 + r, q = q0 + tx;
    if (p < n && q <= p) t[r][tx] = a[(long long)p * ldm + q];
  }
  __syncthreads();
#pragma unroll
  for (int r = ty; r < CTL; r += 8) {
    const int p = p0 + r, q = q0 + tx;
    if (p < n && q < n) {  // (above the diagonal of a diagonal tile: the mirrored element)
      const S v = ip == iq && tx > r ? t[tx][r] : t[r][tx];
      store((size_t)p * n + q, v);
    }
    if (ip != iq && q0 + r < n && p0 + tx < n) {
      const S v = t[tx][r];
      store((size_t)(q0 + r) * n + p0 + tx, v);
    }
  }
}

inline int grid1(long long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

int launch_delta(const double* eps, int n_occ, int n_virt, double* delta, cudaStream_t s) {
  long long n = (long long)n_occ * n_virt;
  delta_kernel<<<grid1(n, 256), 256, 0, s>>>(eps, n_occ, n_virt, delta);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_dtable(const double* z, int F, const double* delta, int n_ov, int ld, bool fp32, void* out, cudaStream_t s) {
  dim3 g(grid1(ld, 256), F);
  if (fp32)
    dtable_kernel<float><<<g, 256, 0, s>>>(z, F, delta, n_ov, ld, (float*)out);
  else
    dtable_kernel<double><<<g, 256, 0, s>>>(z, F, delta, n_ov, ld, (double*)out);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_split_o(const double* o_ov, int n_aux, int n_ov, int n_aux_pad, int n_ov_pad, __nv_bfloat16* hi,
                   __nv_bfloat16* lo, float* f32, cudaStream_t s) {
  long long n = (long long)n_aux_pad * n_ov_pad;
  split_o_kernel<<<grid1(n, 256), 256, 0, s>>>(o_ov, n_aux, n_ov, n_aux_pad, n_ov_pad, hi, lo, f32);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_rhs_gather(MatKind kind, const double* src, long long src_row_stride, const int* row_of, int row_f, int F, int r,
                      int n_aux, void* dst, long long ldr, long long rhs_stride, double* bnorm2, cudaStream_t s) {
  // The same rows for every matrix: a CTA writes several copies of what it read (the conversions and the FP64 sum bound a
  // CTA per copy: 33 nodes of 340 states with 6 cores, N_aux 1190, 394 -> 68 us), as long as some 16 CTAs per SM remain.
  const int share = (!row_of && row_f == 0) ? std::max(1, (int)std::min<long long>(F, (long long)F * r / (16 * 152))) : 1;
  dim3 g(r, (F + share - 1) / share);
  switch (kind) {
    case MatKind::RealF32:
      rhs_gather_kernel<float><<<g, 128, 0, s>>>(src, src_row_stride, row_of, row_f, F, share, r, n_aux, (float*)dst, ldr, rhs_stride, bnorm2);
      break;
    case MatKind::CplxF32:
      rhs_gather_kernel<float2><<<g, 128, 0, s>>>(src, src_row_stride, row_of, row_f, F, share, r, n_aux, (float2*)dst, ldr, rhs_stride, bnorm2);
      break;
    case MatKind::RealF64:
      rhs_gather_kernel<double><<<g, 128, 0, s>>>(src, src_row_stride, row_of, row_f, F, share, r, n_aux, (double*)dst, ldr, rhs_stride, bnorm2);
      break;
    case MatKind::CplxF64:
      rhs_gather_kernel<double2><<<g, 128, 0, s>>>(src, src_row_stride, row_of, row_f, F, share, r, n_aux, (double2*)dst, ldr, rhs_stride, bnorm2);
      break;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_sigma_x(const double* o_core, int n_occ, int n_core, int n_aux, double* sx, cudaStream_t s) {
  sigma_x_kernel<<<n_core, 256, 0, s>>>(o_core, n_occ, n_core, n_aux, sx);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_fill_z_pairs(const double* eps, const int* pair_m, const double* pair_w, int n_pairs, double eta, double* z,
                        cudaStream_t s) {
  if (n_pairs <= 0) return 0;
  fill_z_pairs_kernel<<<grid1(n_pairs, 128), 128, 0, s>>>(eps, pair_m, pair_w, n_pairs, eta, z);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_mat_to_c128(MatKind kind, const void* mats, int n, long long ldm, long long stride, int F, double* out,
                       cudaStream_t s) {
  const long long nt = (n + CTL - 1) / CTL;
  dim3 g((unsigned)(nt * (nt + 1) / 2), F);
  const bool pairs = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  switch (kind) {
    case MatKind::RealF32: mat_to_c128_kernel<float><<<g, 256, 0, s>>>((const float*)mats, n, ldm, stride, out, pairs); break;
    case MatKind::CplxF32: mat_to_c128_kernel<float2><<<g, 256, 0, s>>>((const float2*)mats, n, ldm, stride, out, pairs); break;
    case MatKind::RealF64: mat_to_c128_kernel<double><<<g, 256, 0, s>>>((const double*)mats, n, ldm, stride, out, pairs); break;
    case MatKind::CplxF64: mat_to_c128_kernel<double2><<<g, 256, 0, s>>>((const double2*)mats, n, ldm, stride, out, pairs); break;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace gwc
