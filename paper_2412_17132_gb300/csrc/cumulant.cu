// Retarded-cumulant spectral function (Sec. "Numerical GW+C scheme").
//
//   beta_j = |Im Sigma_n(eps_n + w_j)| / pi
//   C~(t)  = sum_j q_j beta_j / w_j^2 (e^{-i w_j t} - 1)        (Eq. landau_cumulant_truncated)
//   G^C(t) = G^QP(t) e^{C~(t)}                                   (Eq. cumulant_propagator_numerical_time)
//   A(eps^QP + nu) = (1/pi) Re int_0^T e^{i nu t - eta t} e^{C~(t)} dt    (Eq. eq:AGWC)
//
// The transform of e^{C~(t)} followed by the convolution with G^QP (Eqs.
// cumulant_propagator_fourier, cumulant_propagator_convolution) is done as ONE damped
// transform (convolution theorem): g_k = w_k e^{C~(t_k) - eta t_k}, t_k = k dt, w_0 = 1/2,
// X_j = dt sum_k g_k e^{2 pi i jk/n}, A_j = Re X_j / pi on nu_j = 2 pi j/(n dt).
// The sum over k is a batched Stockham FFT in FP64 (Stockham autosort form as in
// E. Bainville, "OpenCL Fast Fourier Transform", 2010), four radix-2 levels per kernel.
#include <algorithm>
#include <utility>

#include "gwc_internal.h"

namespace gwc {

namespace {

// ---- C~(t) on blocks of times ---------------------------------------------------------------------
// C~ is band-limited by its grid (|w_j| <= w_max), and the times are far denser than its Nyquist step (30 eV
// windows: w_max dt = 0.03 at n_t = 2^16, t_max = 2000). So on a block of B consecutive times, t = t_b + h s with
// |s| <= 1 and h = B dt / 2, sum_j c_j e^{-i w_j t} is a polynomial of degree 31 in s to FP64 rounding as long as
// w_max h <= 8 (the interpolation error of e^{-i x s} at 32 Chebyshev nodes is at most 2 J_32(x), 9e-17 at x = 8).
// Its values at the 32 nodes +-s_m cost 2 FMAs per (node, j) (E_j cos and E_j sin of the 16 positive nodes,
// E_j = c_j e^{-i w_j t_b}), the Chebyshev coefficients a 16 x 16 cosine transform per parity, and every time one
// 32-term Chebyshev sum: 100 + 48 FMAs per time instead of 6 N_w at N_w = 800, B = 512. FP64 runs at 1/64 of the
// FP32 rate here, so the FP64 instruction count is what bounds the path.
// The coefficients c_j = q_j beta_j / w_j^2 grow without bound towards w = 0 while c_j (e^{-i w_j t} - 1) does not, so nothing may
// be formed as sum c_j e^{-i w_j t} - sum c_j. With p_j = c_j (e^{-i w_j t_b} - 1) from half angles (-2 c_j sin^2, -2 c_j sin cos),
//   sum_j c_j (e^{-i w_j t} - 1) = sum_j p_j + sum_j E_j (cos(w_j h s) - 1) - i sum_j E_j sin(w_j h s),  E_j = p_j + c_j,
// whose terms are all of the size of what they add; the first sum belongs to the block. (Formed with the difference, every time
// carried a few ulp of sum |c_j|: 1e-11 of the peak at 1.6e4, which a grid point within 3e-4 Ha of zero gives.)
// Points next to zero (a window's rounding error, 1.1e-16 where 0 was meant), |w_j| t_max <= 2^-10, stay out of the blocks and
// are added time by time as the direct sum adds them, up to MAXN of them; a core with more, or whose other coefficients sum
// to more than 2^30, takes the direct sum. Measured (n_t = 2^16), the whole spectrum with the direct
// sum below and with this: 6.66 and 0.156 ms for one core at 400 points, 26.5 and 0.856 ms for 22 cores.
constexpr int NP = 32;       // Chebyshev nodes of a block, NH of them positive
constexpr int NH = NP / 2;
constexpr int MAXB = 1024;   // times per block, a power of two in NP .. MAXB
constexpr int MAXG = 4;      // consecutive blocks of one work item
constexpr int CT = 256;      // threads
constexpr int MAXN = 8;      // points next to zero of a core on blocks
constexpr double kNear = 0x1p-10;
constexpr float kMaxSum = 0x1p30f;

// the bits of |x|, in the order of |x| (integers and FP32 here: at the FP64 rate each comparison of a CTA takes 128 cycles)
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; }
// |x| as FP32, rounded down; infinite from 2^128 on and for NaN
__device__ __forceinline__ float abs_f32(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff, e = (hi >> 20) - 1023 + 127;
  return e >= 255 ? __int_as_float(0x7f800000) : e <= 0 ? 0.f : __int_as_float((e << 23) | (hi & 0xfffff) << 3);
}
__device__ __forceinline__ bool next_to_zero(double w, long long near_bits) { return abs_bits(w) <= near_bits; }

// (w_j, c_j) of the points next to zero, in the order of the grid
struct NearPoints {
  int n;
  int j[MAXN];
  double w[MAXN], c[MAXN];
};

// Times per block for core c's grid: the largest power of two with w_max B dt / 2 <= 8; 0 where not even NP times fit
// (a grid beyond w_max dt = 1/2, or one that is not finite): that core takes the direct sum. With coef given, 0 also where the
// points next to zero are too many or the others' coefficients too large (or not finite), and the points next to zero go
// to `near` (shared memory). CT threads; every one gets the result, the same in every kernel.
__device__ int block_times(const double* __restrict__ w, const double* __restrict__ coef, int n_w, int n_t, double dt,
                           NearPoints* near) {
  __shared__ long long wm[CT / 32];
  __shared__ float cm[CT / 32];
  const long long near_bits = abs_bits(kNear / (dt * n_t));
  if (coef) {
    if (threadIdx.x == 0) near->n = 0;
    __syncthreads();
  }
  long long top = 0;
  float s = 0.f;
  for (int j = threadIdx.x; j < n_w; j += CT) {
    const double a = w[j], c = coef ? coef[j] : 0.0;
    top = max(top, abs_bits(a));
    if (abs_bits(c) == 0) continue;
    if (next_to_zero(a, near_bits)) {
      const int q = atomicAdd(&near->n, 1);
      if (q < MAXN) near->j[q] = j;
    } else {
      s += abs_f32(c);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if ((threadIdx.x & 31) == 0) {
    wm[threadIdx.x >> 5] = top;
    cm[threadIdx.x >> 5] = s;
  }
  __syncthreads();
  s = 0.f;
  for (int k = 0; k < CT / 32; ++k) {
    top = max(top, wm[k]);
    s += cm[k];
  }
  const double m = top < abs_bits(1e300) ? __longlong_as_double(top) : 1e300;  // (infinities and NaN lie above)
  if (coef) {
    if (near->n > MAXN || !(s <= kMaxSum)) return 0;
    if (threadIdx.x == 0) {
      for (int q = 1; q < near->n; ++q)  // the order of the grid, whichever thread came first
        for (int r = q; r > 0 && near->j[r] < near->j[r - 1]; --r) {
          const int x = near->j[r];
          near->j[r] = near->j[r - 1];
          near->j[r - 1] = x;
        }
      for (int q = 0; q < near->n; ++q) {
        near->w[q] = w[near->j[q]];
        near->c[q] = coef[near->j[q]];
      }
    }
    __syncthreads();
  }
  int b = 0;
  for (int t = NP; t <= MAXB && t <= n_t && m * dt * (0.5 * t) <= 8.0; t <<= 1) b = t;
  return b;
}

// coef[c][j] = q_j beta_j / w_j^2 with trapezoid weights q_j of the per-core grid, and (tab given, core on blocks)
// tab[c][j][m] = cos(w_j h s_m) - 1, tab[c][j][NH + m] = sin(w_j h s_m), s_m = cos(pi (2 m + 1) / (2 NP)). The last row of the grid
// writes the transform's factors tw[m] = e^{+2 pi i m / n_t}, m < n_t / 2.
__global__ void __launch_bounds__(CT) cumulant_coef_kernel(const double* __restrict__ omega_rel, int n_w,
                                                            const double* __restrict__ im_sigma, int n_t, double dt,
                                                            double* __restrict__ coef, double* __restrict__ tab,
                                                            double2* __restrict__ tw) {
  const int c = blockIdx.y;
  if (c == (int)gridDim.y - 1) {
    for (int m = blockIdx.x * CT + threadIdx.x; m < n_t / 2; m += gridDim.x * CT) {
      double sn, cs;
      sincospi(2.0 * (double)m / (double)n_t, &sn, &cs);
      tw[m] = make_double2(cs, sn);
    }
    return;
  }
  const double* w = omega_rel + (size_t)c * n_w;
  const int b = tab ? block_times(w, nullptr, n_w, n_t, dt, nullptr) : 0;
  const int e = blockIdx.x * CT + threadIdx.x, j = e / NH, m = e % NH;
  if (j >= n_w) return;
  const double wj = w[j];
  if (m == 0) {
    double q = 0.0;
    if (j > 0) q += 0.5 * (w[j] - w[j - 1]);
    if (j < n_w - 1) q += 0.5 * (w[j + 1] - w[j]);
    const double beta = fabs(im_sigma[(size_t)c * n_w + j]) * (1.0 / 3.14159265358979323846);
    coef[(size_t)c * n_w + j] = wj == 0.0 ? 0.0 : q * beta / (wj * wj);
  }
  if (b == 0) return;
  double sn, cs;
  sincos(0.5 * (wj * ((0.5 * b * dt) * cospi((2 * m + 1) * (0.5 / NP)))), &sn, &cs);
  double* o = tab + ((size_t)c * n_w + j) * NP;
  o[m] = -2.0 * sn * sn;
  o[NH + m] = 2.0 * sn * cs;
}

// One work item: G consecutive blocks from block b0 of core c (all of its times).
template <int G>
__device__ void cumulant_blocks(const double* __restrict__ w, const double* __restrict__ coef, const double* __restrict__ tab,
                                int n_w, int B, int b0, double dt, long long near_bits, double eta, double2 (*es)[CT] /*[MAXG][CT]*/,
                                double2 (*cf)[NP] /*[MAXG][NP]*/, const double* cosn, double2 (*s0sh)[CT / 32] /*[MAXG][CT / 32]*/, const NearPoints& near,
                                double2* __restrict__ g) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double step = B * dt, tc = dt * ((double)b0 * B + 0.5 * (B - 1));  // centre of the first block
  double ar[G], ai[G];
  double2 s0[G];  // sum_j p_j of every block
#pragma unroll
  for (int u = 0; u < G; ++u) {
    ar[u] = ai[u] = 0.0;
    s0[u] = make_double2(0.0, 0.0);
  }
  for (int j0 = 0; j0 < n_w; j0 += CT) {
    const int j = j0 + tid;
    double2 p = make_double2(0.0, 0.0), r = make_double2(0.0, 0.0);  // p_j; e^{-i w_j B dt} - 1
    double cj = 0.0;
    if (j < n_w) {
      cj = next_to_zero(w[j], near_bits) ? 0.0 : coef[j];
      if (cj != 0.0) {
        double sn, cs;
        sincos(0.5 * (w[j] * tc), &sn, &cs);
        const double a = -2.0 * (cj * sn);
        p = make_double2(a * sn, a * cs);
        if (G > 1) {
          sincos(0.5 * (w[j] * step), &sn, &cs);
          r = make_double2(-2.0 * sn * sn, -2.0 * sn * cs);
        }
      }
    }
    __syncthreads();  // the previous chunk (or item) has been read
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const double2 e = make_double2(p.x + cj, p.y);
      es[u][tid] = e;
      s0[u].x += p.x;
      s0[u].y += p.y;
      if (u + 1 < G) p = make_double2(fma(e.x, r.x, fma(-e.y, r.y, p.x)), fma(e.x, r.y, fma(e.y, r.x, p.y)));
    }
    __syncthreads();
    const int jn = min(CT, n_w - j0);
    const double* t = tab + (size_t)j0 * NP + lane;
#pragma unroll 4
    for (int q = warp; q < jn; q += CT / 32) {
      const double v = t[(size_t)q * NP];
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const double2 x = es[u][q];
        ar[u] = fma(x.x, v, ar[u]);
        ai[u] = fma(x.y, v, ai[u]);
      }
    }
  }
  // sums over the warps (es holds them), then the node values and sum_j p_j
  __syncthreads();
  double2* part = &es[0][0];  // [warp][u][node]
#pragma unroll
  for (int u = 0; u < G; ++u) part[(warp * G + u) * 32 + lane] = make_double2(ar[u], ai[u]);
#pragma unroll
  for (int u = 0; u < G; ++u) {
    for (int o = 16; o > 0; o >>= 1) {
      s0[u].x += __shfl_down_sync(0xffffffffu, s0[u].x, o);
      s0[u].y += __shfl_down_sync(0xffffffffu, s0[u].y, o);
    }
    if (lane == 0) s0sh[u][warp] = s0[u];
  }
  __syncthreads();
  for (int e = tid; e < G * 32; e += CT) {
    double2 a = part[e];
#pragma unroll
    for (int k = 1; k < CT / 32; ++k) {
      const double2 x = part[k * G * 32 + e];
      a.x += x.x;
      a.y += x.y;
    }
    part[e] = a;  // read by this thread alone so far
  }
  __syncthreads();
  // Chebyshev coefficients: even ones from E (cos - 1), with sum_j p_j on the constant, odd ones from -i E sin
  for (int e = tid; e < G * NP; e += CT) {
    const int u = e / NP, p = e % NP;
    const double2* v = part + u * 32 + (p & 1) * NH;
    double2 a = make_double2(0.0, 0.0);
#pragma unroll
    for (int m = 0; m < NH; ++m) {
      const double k = cosn[(p * (2 * m + 1)) & (4 * NP - 1)];
      a.x = fma(v[m].x, k, a.x);
      a.y = fma(v[m].y, k, a.y);
    }
    const double f = p == 0 ? 2.0 / NP : 4.0 / NP;
    a = (p & 1) ? make_double2(f * a.y, -f * a.x) : make_double2(f * a.x, f * a.y);
    if (p == 0) {
      double2 s = s0sh[u][0];
#pragma unroll
      for (int k = 1; k < CT / 32; ++k) {
        s.x += s0sh[u][k].x;
        s.y += s0sh[u][k].y;
      }
      a.x += s.x;
      a.y += s.y;
    }
    cf[u][p] = a;
  }
  __syncthreads();
  for (int q = tid; q < B / 2; q += CT) {  // the times at +-s of every block
    const double s = (2 * q + 1) / (double)B;
    double t0 = 1.0, t1 = s;
    double er[G], ei[G], dr[G], di[G];  // even and odd sums
#pragma unroll
    for (int u = 0; u < G; ++u) er[u] = ei[u] = dr[u] = di[u] = 0.0;
#pragma unroll 4
    for (int p = 0; p < NP; p += 2) {
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const double2 x = cf[u][p], y = cf[u][p + 1];
        er[u] = fma(x.x, t0, er[u]);
        ei[u] = fma(x.y, t0, ei[u]);
        dr[u] = fma(y.x, t1, dr[u]);
        di[u] = fma(y.y, t1, di[u]);
      }
      t0 = fma(2.0 * s, t1, -t0);
      t1 = fma(2.0 * s, t0, -t1);
    }
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const int kc = (b0 + u) * B + B / 2;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int k = side ? kc - 1 - q : kc + q;
        double re = side ? er[u] - dr[u] : er[u] + dr[u], im = side ? ei[u] - di[u] : ei[u] + di[u];
        double sn, cs;
        for (int a = 0; a < near.n; ++a) {
          sincos(near.w[a] * (dt * k), &sn, &cs);
          re += near.c[a] * (cs - 1.0);
          im -= near.c[a] * sn;
        }
        const double mag = exp(re - eta * (dt * k)) * (k == 0 ? 0.5 : 1.0);
        sincos(im, &sn, &cs);
        g[k] = make_double2(mag * cs, mag * sn);
      }
    }
  }
}

// g[c][k] = w_k exp(C~(t_k) - eta t_k), w_0 = 1/2, for the cores whose grid fits the blocks. gridDim.y = cores; an item is G
// consecutive blocks (the rotation e^{-i w_j B dt} replaces a sincos per block and j), G the largest of 4, 2, 1 that
// still gives four items per SM.
__global__ void __launch_bounds__(CT) cumulant_block_kernel(const double* __restrict__ omega_rel, int n_w,
                                                             const double* __restrict__ coef, const double* __restrict__ tab,
                                                             int n_t, double dt, double eta, int n_sm, double2* __restrict__ g) {
  __shared__ double2 es[MAXG][CT];
  __shared__ double2 cf[MAXG][NP];
  __shared__ double cosn[4 * NP];  // cos(pi k / (2 NP))
  __shared__ double2 s0sh[MAXG][CT / 32];
  __shared__ NearPoints near;
  static_assert((CT / 32) * 32 <= CT, "the warps' partial sums fit in es");
  const int c = blockIdx.y;
  const double* w = omega_rel + (size_t)c * n_w;
  const long long near_bits = abs_bits(kNear / (dt * n_t));
  const int B = block_times(w, coef + (size_t)c * n_w, n_w, n_t, dt, &near);
  if (B == 0) return;
  if (threadIdx.x < 4 * NP) cosn[threadIdx.x] = cospi(threadIdx.x * (0.5 / NP));
  __syncthreads();
  const int nb = n_t / B;
  const double* k = coef + (size_t)c * n_w;
  const double* t = tab + (size_t)c * n_w * NP;
  double2* o = g + (size_t)c * n_t;
  const long long all = (long long)nb * gridDim.y, want = 4LL * n_sm;
  if (nb >= 4 && all / 4 >= want) {
    for (int b = 4 * blockIdx.x; b < nb; b += 4 * gridDim.x)
      cumulant_blocks<4>(w, k, t, n_w, B, b, dt, near_bits, eta, es, cf, cosn, s0sh, near, o);
  } else if (nb >= 2 && all / 2 >= want) {
    for (int b = 2 * blockIdx.x; b < nb; b += 2 * gridDim.x)
      cumulant_blocks<2>(w, k, t, n_w, B, b, dt, near_bits, eta, es, cf, cosn, s0sh, near, o);
  } else {
    for (int b = blockIdx.x; b < nb; b += gridDim.x)
      cumulant_blocks<1>(w, k, t, n_w, B, b, dt, near_bits, eta, es, cf, cosn, s0sh, near, o);
  }
}

// The direct sum over the grid, for the cores that do not go by blocks (all of them without `blocks`). Each thread
// takes KT consecutive times: per grid point one sincos at its first time and one for the step w_j dt, then the phase
// advances by that rotation (the rotation drifts by ~KT ulp over a block).
constexpr int KT = 32;

__global__ void __launch_bounds__(CT) cumulant_time_kernel(const double* __restrict__ omega_rel, int n_w, const double* __restrict__ coef,
                                     int n_core, int n_t, double dt, double eta, int blocks, double2* __restrict__ g) {
  extern __shared__ double sh[];  // [2][n_w]
  double* sw = sh;
  double* sc = sh + n_w;
  const int c = blockIdx.y;
  __shared__ NearPoints near;
  if (blocks && block_times(omega_rel + (size_t)c * n_w, coef + (size_t)c * n_w, n_w, n_t, dt, &near) > 0) return;
  for (int j = threadIdx.x; j < n_w; j += blockDim.x) {
    sw[j] = omega_rel[(size_t)c * n_w + j];
    sc[j] = coef[(size_t)c * n_w + j];
  }
  __syncthreads();
  const int k0 = (blockIdx.x * blockDim.x + threadIdx.x) * KT;
  if (k0 >= n_t) return;
  double re[KT], im[KT];
#pragma unroll
  for (int q = 0; q < KT; ++q) re[q] = im[q] = 0.0;
  const double t0 = dt * k0;
  for (int j = 0; j < n_w; ++j) {
    const double cj = sc[j];
    if (cj == 0.0) continue;
    double sn, cs, sd, cd;
    sincos(sw[j] * t0, &sn, &cs);
    sincos(sw[j] * dt, &sd, &cd);
#pragma unroll
    for (int q = 0; q < KT; ++q) {
      re[q] += cj * (cs - 1.0);
      im[q] -= cj * sn;
      const double c2 = cs * cd - sn * sd;  // angle + w_j dt
      sn = sn * cd + cs * sd;
      cs = c2;
    }
  }
#pragma unroll
  for (int q = 0; q < KT; ++q) {
    const int k = k0 + q;
    if (k >= n_t) break;
    const double t = dt * k;
    const double mag = exp(re[q] - eta * t) * (k == 0 ? 0.5 : 1.0);
    double sn, cs;
    sincos(im[q], &sn, &cs);
    g[(size_t)c * n_t + k] = make_double2(mag * cs, mag * sn);
  }
}

// Only Re X_j is wanted, the transform of the Hermitian part h_k = (g_k + conj g_{n-k}) / 2, whose result is real. Its even and
// odd outputs are the real and imaginary parts of ONE complex transform of half the length N = n / 2:
//   x_2j + i x_2j+1 = sum_{k<N} Z_k e^{2 pi i jk/N},  Z_k = (h_k + h_{k+N}) + i e^{2 pi i k/n} (h_k - h_{k+N}).
__device__ __forceinline__ double2 half_input(const double2* __restrict__ g, int n, int k, const double2* __restrict__ tw) {
  const int N = n >> 1;
  const double2 a = g[k], b = g[k ? n - k : 0], c = g[k + N], d = g[N - k];
  const double2 h0 = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
  const double2 h1 = make_double2(0.5 * (c.x + d.x), 0.5 * (c.y - d.y));
  const double2 e = make_double2(h0.x - h1.x, h0.y - h1.y), w = tw[k];
  return make_double2((h0.x + h1.x) - (e.x * w.y + e.y * w.x), (h0.y + h1.y) + (e.x * w.x - e.y * w.y));
}

// 2^LR-point Stockham pass of the half-length transform with span p (1, 2^LR, ...): LR radix-2 levels in registers, so a
// transform of 2^15 points takes four passes over memory and four launches. FIRST forms Z from g, LAST writes
// the spectrum: A on ascending nu, o = 0 <-> the most negative. 22 transforms for n_t = 2^16: 134 us (FP64
// instructions and L2) against 221 us for one full-length radix-2 level per launch; the whole spectrum 0.935 -> 0.831 ms (blocks as then),
// and for one core, where 18 launches became 5, 0.164 -> 0.154 ms.
template <int LR, bool FIRST, bool LAST>
__global__ void __launch_bounds__(64) stockham_pass_kernel(const double2* __restrict__ x, double2* __restrict__ y, int n, int p,
                                                            const double2* __restrict__ tw, double dt, double* __restrict__ a,
                                                            double* __restrict__ nu) {
  constexpr int R = 1 << LR;
  const int N = n >> 1, c = blockIdx.y;
  const int i = blockIdx.x * 64 + threadIdx.x;
  if (i >= N / R) return;
  double2 v[R];
#pragma unroll
  for (int r = 0; r < R; ++r)
    v[r] = FIRST ? half_input(x + (size_t)c * n, n, i + r * (N / R), tw) : x[(size_t)c * N + i + r * (N / R)];
  const int k = i & (p - 1);
  // level l joins the blocks r and r + R / 2 of the autosort order; its spans are p 2^l
#pragma unroll
  for (int l = 0; l < LR; ++l) {
    double2 u[R];
#pragma unroll
    for (int r = 0; r < R / 2; ++r) {
      const int q = r & ((1 << l) - 1);  // position inside the span beyond k: k + p q
      const double2 w = tw[(size_t)(k + p * q) * (size_t)(N / (p << l))];  // e^{+i pi (k + p q) / (p 2^l)}
      const double2 u0 = v[r], u1 = v[r + R / 2];
      const double2 t = make_double2(u1.x * w.x - u1.y * w.y, u1.x * w.y + u1.y * w.x);
      const int o = 2 * r - q;
      u[o] = make_double2(u0.x + t.x, u0.y + t.y);
      u[o + (1 << l)] = make_double2(u0.x - t.x, u0.y - t.y);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = u[r];
  }
  const int j = ((i - k) << LR) + k;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (!LAST) {
      y[(size_t)c * N + j + r * p] = v[r];
    } else {
      const int o = (2 * (j + r * p) + N) & (n - 1);
      double* ao = a + (size_t)c * n + o;
      ao[0] = dt * v[r].x * (1.0 / 3.14159265358979323846);
      ao[1] = dt * v[r].y * (1.0 / 3.14159265358979323846);
      if (nu && c == 0) {
        nu[o] = 2.0 * 3.14159265358979323846 * (double)(o - N) / ((double)n * dt);
        nu[o + 1] = 2.0 * 3.14159265358979323846 * (double)(o + 1 - N) / ((double)n * dt);
      }
    }
  }
}

template <int LR>
void launch_pass(const double2* x, double2* y, int n, int p, const double2* tw, double dt, double* a, double* nu, int n_core,
                 bool last, cudaStream_t s) {
  const int per = (n >> 1) >> LR;
  const dim3 g((per + 63) / 64, n_core);
  if (p == 1 && last)
    stockham_pass_kernel<LR, true, true><<<g, 64, 0, s>>>(x, y, n, p, tw, dt, a, nu);
  else if (p == 1)
    stockham_pass_kernel<LR, true, false><<<g, 64, 0, s>>>(x, y, n, p, tw, dt, a, nu);
  else if (last)
    stockham_pass_kernel<LR, false, true><<<g, 64, 0, s>>>(x, y, n, p, tw, dt, a, nu);
  else
    stockham_pass_kernel<LR, false, false><<<g, 64, 0, s>>>(x, y, n, p, tw, dt, a, nu);
}

}  // namespace

int launch_cumulant_spectrum(const double* omega_rel, int n_w, const double* im_sigma, int n_core, int n_t, double t_max,
                             double eta, double* work_a, double* work_b, double* coef, double* twiddle, double* a_out,
                             double* nu_out, double* table, int n_sm, cudaStream_t s) {
  int launches = 0;
  const double dt = t_max / n_t;
  cumulant_coef_kernel<<<dim3((n_w * NH + CT - 1) / CT, n_core + 1), CT, 0, s>>>(omega_rel, n_w, im_sigma, n_t, dt, coef, table,
                                                                                 (double2*)twiddle);
  ++launches;
  if (table) {
    const int per = std::max(1, std::min(n_t / NP, (6 * n_sm + n_core - 1) / n_core));
    cumulant_block_kernel<<<dim3(per, n_core), CT, 0, s>>>(omega_rel, n_w, coef, table, n_t, dt, eta, n_sm, (double2*)work_a);
    ++launches;
  }
  // beyond 48 KB with the kernel's own shared memory (272 bytes), from 3056 grid points on, a larger limit has to be asked for
  const size_t sm = sizeof(double) * 2 * (size_t)n_w;
  if (sm > 47 * 1024) {
    if (cudaFuncSetAttribute(cumulant_time_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             std::max((int)sm, 16 * 8192)) != cudaSuccess)  // (8192 points: the largest grid of the entry points)
      return -1;
  }
  dim3 g((n_t + CT * KT - 1) / (CT * KT), n_core);
  cumulant_time_kernel<<<g, CT, sm, s>>>(omega_rel, n_w, coef, n_core, n_t, dt, eta, table ? 1 : 0, (double2*)work_a);
  ++launches;
  double2* src = (double2*)work_a;
  double2* dst = (double2*)work_b;
  const double2* tw = (const double2*)twiddle;
  int levels = 0;
  while ((2 << levels) < n_t) ++levels;  // n_t / 2 = 2^levels points
  for (int done = 0; done < levels;) {
    const int lr = std::min(4, levels - done);
    const bool last = done + lr == levels;
    const int p = 1 << done;
    switch (lr) {
      case 1: launch_pass<1>(src, dst, n_t, p, tw, dt, a_out, nu_out, n_core, last, s); break;
      case 2: launch_pass<2>(src, dst, n_t, p, tw, dt, a_out, nu_out, n_core, last, s); break;
      case 3: launch_pass<3>(src, dst, n_t, p, tw, dt, a_out, nu_out, n_core, last, s); break;
      default: launch_pass<4>(src, dst, n_t, p, tw, dt, a_out, nu_out, n_core, last, s); break;
    }
    ++launches;
    done += lr;
    std::swap(src, dst);
  }
  return cudaPeekAtLastError() == cudaSuccess ? launches : -1;
}

}  // namespace gwc
