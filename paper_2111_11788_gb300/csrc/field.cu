// Lognormal coefficient kappa = exp(Phi xi) at element centroids.
//
// Phi is the full tensor basis of the 1D exponential-covariance KLE
// eigenfunctions (Sec. 5.2 "eigenfunctions in each dimension"):
//   Phi[e, k] = sqrt(sigma^2) prod_a sqrt(theta_{k_a}) f_{k_a}(c_a(e)),
// k = (k_z m + k_y) m + k_x. Because Phi is a Kronecker product of per-axis
// tables F[i, k] = sqrt(theta_k) f_k((i + 1/2) h), the contraction Phi xi is
// evaluated axis by axis (sum factorisation) in FP64: for each sample a
// small x-contraction into shared memory, then per element the last axis's
// sum (over the even and odd modes of a mirrored pair of elements) and one
// exp. On GB300 the FP64 exp and FMAs bound the kernel, not the write of
// kappa (8 B per element).
#include <algorithm>
#include <cmath>

#include "mlmc_internal.cuh"

namespace mlmc {
namespace {

// exp in FP64 by the table-driven reduction of P. T. P. Tang ("Table-driven
// implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15(2), 1989), written from the mathematics, for a
// log-field x that is formed as t = x 64 / ln 2 (the factor goes into the small
// contracted table, not into a multiply per element):
//   t = N + f, N = 64 k + j, |f| <= 1/2, 0 <= j < 64,
//   exp(x) = 2^(t/64) = 2^k 2^(j/64) (1 + p), r = f ln2 / 64,
//   p = r + r^2 / 2 + r^3 / 6 + r^4 / 24 + r^5 / 120
// (the next Taylor term, r^6 / 720, is below 4e-17), evaluated in f with the
// powers of ln2 / 64 in its coefficients. N comes from adding 1.5 2^52 (the
// low word of the sum holds N, taking it off again gives N, and t - N is
// exact), 2^(j/64) from a table made on the host, and 2^k is added to the
// exponent field: 9 FP64 operations per element; reducing x itself with ln2 /
// 64 in two parts, with conversions through the FP64 pipe and a multiply by
// 2^k, took 13. About 1 ulp beside the rounding of t. Outside the normal
// range of the result, and for NaN, the library's exp.
constexpr int EXP_TAB = 64;
__device__ double g_exp2_tab[EXP_TAB];
constexpr double kInvLn2x64 = 92.332482616893658071;   // 64 / ln 2
constexpr double kR = 0x1.62e42fefa39efp-7;            // ln 2 / 64 = 0.0108304246962491454596...
constexpr double kRound = 6755399441055744.0;          // 1.5 2^52
constexpr int kBig = 0x40ef0000;                       // high word of |t| = 64 * 992 (|x| = 687.6)

__device__ __forceinline__ double kle_exp(double t, const double* tab) {
  if ((__double2hiint(t) & 0x7fffffff) >= kBig) return exp(t * kR);
  const double y = t + kRound;
  const int N = __double2loint(y);
  const double f = t - (y - kRound);
  double q = fma(f, kR * kR * kR * kR * kR / 120.0, kR * kR * kR * kR / 24.0);
  q = fma(f, q, kR * kR * kR / 6.0);
  q = fma(f, q, kR * kR / 2.0);
  q = fma(f, q, kR);
  const double T = tab[N & (EXP_TAB - 1)];
  const double v = fma(T, f * q, T);
  return __hiloint2double(__double2hiint(v) + ((N >> 6) << 20), __double2loint(v));
}

// F[i * m + k] = sqrt(theta_k) f_k(x_i), x_i = (i + 1/2) / n, centred t = x - 1/2:
// even k: cos(w t) / sqrt(1/2 + sin(w) / (2w)); odd k: sin(w t) / sqrt(1/2 - sin(w) / (2w)).
__global__ void k_kle_table(int n, int m, const double* __restrict__ omega,
                            const double* __restrict__ theta, const int32_t* __restrict__ even,
                            double* __restrict__ table) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * m) return;
  const int i = idx / m;
  const int k = idx - i * m;
  const double w = omega[k];
  const double t = ((double)i + 0.5) / (double)n - 0.5;
  const double s2 = sin(w) / (2.0 * w);   // sin(2 w a) / (2 w) with a = 1/2
  double f;
  if (even[k]) {
    f = cos(w * t) / sqrt(0.5 + s2);
  } else {
    f = sin(w * t) / sqrt(0.5 - s2);
  }
  table[idx] = sqrt(theta[k]) * f;
}

// Row pairs per thread in 2D. The eigenfunctions are even or odd about the
// centre, so element rows iy and n - 1 - iy share the sums over the even and
// over the odd modes, E and O: their fields are E + O and E - O, m / 2 + 1
// FP64 operations per element instead of m. A CTA covers 32 columns x 8 *
// KAP_ROWS row pairs, so the x-contraction of its columns (m^2 FMAs per
// column) is shared by 64 rows.
constexpr int KAP_ROWS = 4;

// The sample's KLE coefficients in the full tensor layout (m^dim entries) in
// shared memory: a copy, or under total-order truncation the kept
// coefficients scattered to their full-basis slots and zeros elsewhere.
template <class V>
__device__ __forceinline__ void load_coefs(const double* __restrict__ xs, int M_xi,
                                           const int32_t* __restrict__ slot, int M_full,
                                           V* s_xi, int tid, int nthreads) {
  if (!slot) {
    for (int k = tid; k < M_full; k += nthreads) s_xi[k] = (V)xs[k];
    return;
  }
  for (int k = tid; k < M_full; k += nthreads) s_xi[k] = V(0);
  __syncthreads();
  for (int t = tid; t < M_xi; t += nthreads) s_xi[slot[t]] = (V)xs[t];
}

// 2D: CTA covers 32 columns x (8 * KAP_ROWS) row pairs of one sample. Bound by
// the FP64 pipe: m / 2 + 10 operations per element (64 samples of 512^2, m = 8:
// 674 us with m + 13, 479 us now).
__global__ void __launch_bounds__(TX2* TY2)
    k_kappa2d(int n, int m, double sqrt_sigma2, const double* __restrict__ table,
              const double* __restrict__ xi, int M_xi, const int32_t* __restrict__ slot,
              int64_t es, double* __restrict__ kappa, Prof prof) {
  __shared__ double s_xi[MAX_MODES_1D * MAX_MODES_1D];
  __shared__ double s_t[TX2][MAX_MODES_1D + 1];          // T[ix][k_y] 64 / ln 2
  __shared__ double s_fy[TY2 * KAP_ROWS][MAX_MODES_1D + 1];
  __shared__ double s_tab[EXP_TAB];
  const int b = blockIdx.z;
  const int tid = threadIdx.y * TX2 + threadIdx.x;
  const int nthreads = TX2 * TY2;
  const int x0 = blockIdx.x * TX2;
  const int y0 = blockIdx.y * TY2 * KAP_ROWS;
  const int half = (n + 1) / 2;                          // row pairs (the middle row of an odd n is its own)
  for (int j = tid; j < EXP_TAB; j += nthreads) s_tab[j] = g_exp2_tab[j];
  load_coefs(xi + (int64_t)b * M_xi, M_xi, slot, m * m, s_xi, tid, nthreads);
  for (int idx = tid; idx < TY2 * KAP_ROWS * m; idx += nthreads) {
    const int r = idx / m, k = idx - r * m;
    const int iy = y0 + r;
    s_fy[r][k] = (iy < half) ? table[iy * m + k] : 0.0;
  }
  __syncthreads();
  // T[ix][ky] = sum_kx F[ix][kx] xi[ky * m + kx]
  const double scale = sqrt_sigma2 * kInvLn2x64;
  for (int idx = tid; idx < TX2 * m; idx += nthreads) {
    const int c = idx / m, ky = idx - c * m;
    const int ix = x0 + c;
    double acc = 0.0;
    if (ix < n) {
      const double* fx = table + ix * m;
      for (int kx = 0; kx < m; ++kx) acc = fma(fx[kx], s_xi[ky * m + kx], acc);
    }
    s_t[c][ky] = scale * acc;
  }
  __syncthreads();
  const int ix = x0 + threadIdx.x;
  if (ix < n) {
    double* out = kappa + (int64_t)b * es + ix;
    const double* tx = s_t[threadIdx.x];
#pragma unroll 2
    for (int r = 0; r < KAP_ROWS; ++r) {
      const int rl = threadIdx.y + TY2 * r;
      const int iy = y0 + rl;
      if (iy >= half) break;
      const double* fy = s_fy[rl];
      double e = fy[0] * tx[0], o = 0.0;
      int ky = 1;
      for (; ky + 1 < m; ky += 2) {
        o = fma(fy[ky], tx[ky], o);
        e = fma(fy[ky + 1], tx[ky + 1], e);
      }
      if (ky < m) o = fma(fy[ky], tx[ky], o);
      out[(int64_t)iy * n] = kle_exp(e + o, s_tab);
      const int my = n - 1 - iy;
      if (my != iy) out[(int64_t)my * n] = kle_exp(e - o, s_tab);
    }
  }
  if (prof.acc && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) atomicAdd(prof.acc, prof.per_sample);
}

// 3D: CTA covers 32 (x) x 4 (y) elements for all z of one sample column
// block; per (ix, iy): T2[kz] = sum_ky F[iy][ky] sum_kx F[ix][kx] xi[kz][ky][kx],
// then the layers iz and n - 1 - iz from the even and odd sums over kz of
// F[iz][kz] T2[kz], as in 2D. T2 sits in shared memory (a column per thread):
// as a local array its run-time index would put it in local memory.
constexpr int K3_TY = 4;
__global__ void __launch_bounds__(TX2* K3_TY)
    k_kappa3d(int n, int m, double sqrt_sigma2, const double* __restrict__ table,
              const double* __restrict__ xi, int M_xi, const int32_t* __restrict__ slot,
              int64_t es, double* __restrict__ kappa, Prof prof) {
  extern __shared__ double smem[];
  const int M = m * m * m;
  double* s_xi = smem;                              // M
  double* s_t1 = s_xi + M;                          // [TX2][m*m]  T1[ix][kz*m+ky]
  double* s_t2 = s_t1 + TX2 * m * m;                // [m][threads]
  __shared__ double s_tab[EXP_TAB];
  const int b = blockIdx.z;
  const int tid = threadIdx.y * TX2 + threadIdx.x;
  const int nthreads = TX2 * K3_TY;
  const int x0 = blockIdx.x * TX2;
  const int iy = blockIdx.y * K3_TY + threadIdx.y;
  for (int j = tid; j < EXP_TAB; j += nthreads) s_tab[j] = g_exp2_tab[j];
  load_coefs(xi + (int64_t)b * M_xi, M_xi, slot, M, s_xi, tid, nthreads);
  __syncthreads();
  const int mm = m * m;
  const double scale = sqrt_sigma2 * kInvLn2x64;
  for (int idx = tid; idx < TX2 * mm; idx += nthreads) {
    const int c = idx / mm, kk = idx - c * mm;     // kk = kz * m + ky
    const int ix = x0 + c;
    double acc = 0.0;
    if (ix < n) {
      const double* fx = table + ix * m;
      for (int kx = 0; kx < m; ++kx) acc = fma(fx[kx], s_xi[kk * m + kx], acc);
    }
    s_t1[c * mm + kk] = scale * acc;
  }
  __syncthreads();
  const int ix = x0 + threadIdx.x;
  if (ix >= n || iy >= n) return;
  const double* fy = table + iy * m;
  double* t2 = s_t2 + tid;
  for (int kz = 0; kz < m; ++kz) {
    double acc = 0.0;
    for (int ky = 0; ky < m; ++ky) acc = fma(fy[ky], s_t1[threadIdx.x * mm + kz * m + ky], acc);
    t2[kz * nthreads] = acc;
  }
  double* out = kappa + (int64_t)b * es + (int64_t)iy * n + ix;
  const int64_t plane = (int64_t)n * n;
#pragma unroll 2
  for (int iz = 0; iz < (n + 1) / 2; ++iz) {
    const double* fz = table + iz * m;
    double e = fz[0] * t2[0], o = 0.0;
    int kz = 1;
    for (; kz + 1 < m; kz += 2) {
      o = fma(fz[kz], t2[kz * nthreads], o);
      e = fma(fz[kz + 1], t2[(kz + 1) * nthreads], e);
    }
    if (kz < m) o = fma(fz[kz], t2[kz * nthreads], o);
    out[iz * plane] = kle_exp(e + o, s_tab);
    const int mz = n - 1 - iz;
    if (mz != iz) out[mz * plane] = kle_exp(e - o, s_tab);
  }
  if (prof.acc && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) atomicAdd(prof.acc, prof.per_sample);
}

// kappa in FP32 for the mixed form's inner solves: the same sum factorisation
// and mirrored pairs with FP32 sums, kappa32 = 2^t by the hardware
// approximation (ex2.approx, relative error about 2^-22), t = x / ln 2. A
// thread takes K32_P consecutive row (layer) pairs of one column at a time,
// so a mode costs it one load of the column's contraction and one 16-byte
// load of the axis table for K32_P multiply-adds. Bound by instruction issue
// (80% of the slots in 2D, 77% in 3D): 100 samples of 1024^2 with m = 8 take 137
// us, 46% of the copy bandwidth, and 16 of 128^3 with m = 5 32 us, 63%. On small
// meshes the setup of a CTA's tables comes before its first store. A dense
// contraction over all M modes, on the tensor cores or not, does M multiply-adds
// per element where this does m / 2 + 1.
constexpr int K32_P = 4;
constexpr int K32_Y = 8;          // warps per CTA
constexpr int K32_ROWS = 128;     // 2D: row pairs per CTA

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// even and odd sums over the modes of K32_P consecutive pairs: t the column's
// contraction (stride ts), f the axis table, f[k * fs + pair]
__device__ __forceinline__ void even_odd(int m, const float* t, int ts, const float* f, int fs, float (&e)[K32_P],
                                         float (&o)[K32_P]) {
#pragma unroll
  for (int q = 0; q < K32_P; ++q) e[q] = o[q] = 0.f;
  auto add = [&](int k, float (&a)[K32_P]) {
    const float tv = t[k * ts];
    const float4 fv = *reinterpret_cast<const float4*>(f + k * fs);
    a[0] = fmaf(fv.x, tv, a[0]);
    a[1] = fmaf(fv.y, tv, a[1]);
    a[2] = fmaf(fv.z, tv, a[2]);
    a[3] = fmaf(fv.w, tv, a[3]);
  };
  int k = 0;
  for (; k + 1 < m; k += 2) {
    add(k, e);
    add(k + 1, o);
  }
  if (k < m) add(k, e);
}

__global__ void __launch_bounds__(TX2* K32_Y)
    k_kappa32_2d(int n, int m, float scale, const double* __restrict__ table, const double* __restrict__ xi, int M_xi,
                 const int32_t* __restrict__ slot, int64_t es, float* __restrict__ kappa) {
  __shared__ float s_xi[MAX_MODES_1D * MAX_MODES_1D];
  __shared__ float s_t[TX2][MAX_MODES_1D + 1];                      // T[ix][k_y] / ln 2
  __shared__ __align__(16) float s_f[MAX_MODES_1D][K32_ROWS];       // F[iy][k_y]
  __shared__ float s_fx[TX2][MAX_MODES_1D + 1];                     // F[ix][k_x]
  const int b = blockIdx.z, nthreads = TX2 * K32_Y;
  const int tid = threadIdx.y * TX2 + threadIdx.x;
  const int x0 = blockIdx.x * TX2, y0 = blockIdx.y * K32_ROWS, half = (n + 1) / 2;
  load_coefs(xi + (int64_t)b * M_xi, M_xi, slot, m * m, s_xi, tid, nthreads);
  for (int idx = tid; idx < K32_ROWS * m; idx += nthreads) {
    const int r = idx / m, k = idx - r * m;
    s_f[k][r] = y0 + r < half ? (float)table[(y0 + r) * m + k] : 0.f;
  }
  for (int idx = tid; idx < TX2 * m; idx += nthreads) {
    const int c = idx / m, k = idx - c * m;
    s_fx[c][k] = x0 + c < n ? (float)table[(x0 + c) * m + k] : 0.f;
  }
  __syncthreads();
  for (int idx = tid; idx < TX2 * m; idx += nthreads) {
    const int c = idx / m, ky = idx - c * m;
    float acc = 0.f;
    for (int kx = 0; kx < m; ++kx) acc = fmaf(s_fx[c][kx], s_xi[ky * m + kx], acc);
    s_t[c][ky] = scale * acc;
  }
  __syncthreads();
  const int ix = x0 + threadIdx.x;
  if (ix >= n) return;
  float* out = kappa + (int64_t)b * es + ix;
  for (int p = threadIdx.y * K32_P; p < K32_ROWS && y0 + p < half; p += K32_Y * K32_P) {
    float e[K32_P], o[K32_P];
    even_odd(m, s_t[threadIdx.x], 1, &s_f[0][p], K32_ROWS, e, o);
#pragma unroll
    for (int q = 0; q < K32_P; ++q) {
      const int iy = y0 + p + q, my = n - 1 - iy;
      if (iy < half) {
        out[(int64_t)iy * n] = ex2_approx(e[q] + o[q]);
        if (my != iy) out[(int64_t)my * n] = ex2_approx(e[q] - o[q]);
      }
    }
  }
}

// half (rounded up to K32_P) of the layers' table in shared memory
inline int k32_half(int n) { return ((n + 1) / 2 + K32_P - 1) / K32_P * K32_P; }
inline size_t k32_smem3(int n, int m) {
  return sizeof(float) * ((size_t)m * k32_half(n) + (size_t)m * m * m + (size_t)TX2 * (m * m + 1) +
                          (size_t)m * TX2 * K32_Y + (size_t)TX2 * (m + 1) + (size_t)K32_Y * m);
}

__global__ void __launch_bounds__(TX2* K32_Y)
    k_kappa32_3d(int n, int m, int fs, float scale, const double* __restrict__ table, const double* __restrict__ xi,
                 int M_xi, const int32_t* __restrict__ slot, int64_t es, float* __restrict__ kappa) {
  extern __shared__ __align__(16) float sm32[];
  const int mm = m * m, M = mm * m, half = (n + 1) / 2, nthreads = TX2 * K32_Y;
  float* s_f = sm32;                       // [m][fs] F[iz][k_z] of the first half of the layers
  float* s_xi = s_f + m * fs;              // [M]
  float* s_t1 = s_xi + M;                  // [TX2][mm + 1] T1[ix][k_z m + k_y] / ln 2
  float* s_t2 = s_t1 + TX2 * (mm + 1);     // [m][threads] T2[k_z] of each column
  float* s_fx = s_t2 + m * nthreads;       // [TX2][m + 1] F[ix][k_x]
  float* s_fy = s_fx + TX2 * (m + 1);      // [K32_Y][m] F[iy][k_y]
  const int b = blockIdx.z;
  const int tid = threadIdx.y * TX2 + threadIdx.x;
  const int x0 = blockIdx.x * TX2, iy = blockIdx.y * K32_Y + threadIdx.y;
  load_coefs(xi + (int64_t)b * M_xi, M_xi, slot, M, s_xi, tid, nthreads);
  for (int idx = tid; idx < fs * m; idx += nthreads) {
    const int r = idx / m, k = idx - r * m;
    s_f[k * fs + r] = r < half ? (float)table[r * m + k] : 0.f;
  }
  for (int idx = tid; idx < TX2 * m; idx += nthreads) {
    const int c = idx / m, k = idx - c * m;
    s_fx[c * (m + 1) + k] = x0 + c < n ? (float)table[(x0 + c) * m + k] : 0.f;
  }
  for (int idx = tid; idx < K32_Y * m; idx += nthreads) {
    const int r = idx / m, k = idx - r * m, y = blockIdx.y * K32_Y + r;
    s_fy[r * m + k] = y < n ? (float)table[y * m + k] : 0.f;
  }
  __syncthreads();
  for (int idx = tid; idx < TX2 * mm; idx += nthreads) {
    const int c = idx & (TX2 - 1), kk = idx / TX2;   // lanes along x: the coefficient is a broadcast
    float acc = 0.f;
    for (int kx = 0; kx < m; ++kx) acc = fmaf(s_fx[c * (m + 1) + kx], s_xi[kk * m + kx], acc);
    s_t1[c * (mm + 1) + kk] = scale * acc;
  }
  __syncthreads();
  const int ix = x0 + threadIdx.x;
  if (ix >= n || iy >= n) return;
  float* t2 = s_t2 + tid;
  const float* t1 = s_t1 + threadIdx.x * (mm + 1);
  for (int kz = 0; kz < m; ++kz) {
    float acc = 0.f;
    for (int ky = 0; ky < m; ++ky) acc = fmaf(s_fy[threadIdx.y * m + ky], t1[kz * m + ky], acc);
    t2[kz * nthreads] = acc;
  }
  float* out = kappa + (int64_t)b * es + (int64_t)iy * n + ix;
  const int64_t plane = (int64_t)n * n;
  for (int p = 0; p < half; p += K32_P) {
    float e[K32_P], o[K32_P];
    even_odd(m, t2, nthreads, s_f + p, fs, e, o);
#pragma unroll
    for (int q = 0; q < K32_P; ++q) {
      const int iz = p + q, mz = n - 1 - iz;
      if (iz < half) {
        out[iz * plane] = ex2_approx(e[q] + o[q]);
        if (mz != iz) out[mz * plane] = ex2_approx(e[q] - o[q]);
      }
    }
  }
}

template <class T>
__global__ void k_coarsen2d(int nc, const T* __restrict__ kf, T* __restrict__ kc,
                            int64_t esf, int64_t esc, Prof prof) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y;
  const int b = blockIdx.z;
  if (I >= nc) return;
  const int nf = 2 * nc;
  const T* f = kf + (int64_t)b * esf + (int64_t)(2 * J) * nf + 2 * I;
  kc[(int64_t)b * esc + (int64_t)J * nc + I] = T(0.25) * ((f[0] + f[1]) + (f[nf] + f[nf + 1]));
  if (prof.acc && I == 0 && J == 0) atomicAdd(prof.acc, prof.per_sample);
}

template <class T>
__global__ void k_coarsen3d(int nc, const T* __restrict__ kf, T* __restrict__ kc,
                            int64_t esf, int64_t esc, Prof prof) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y % nc;
  const int K = blockIdx.y / nc;
  const int b = blockIdx.z;
  if (I >= nc) return;
  const int nf = 2 * nc;
  const int64_t pl = (int64_t)nf * nf;
  const T* f = kf + (int64_t)b * esf + (int64_t)(2 * K) * pl + (int64_t)(2 * J) * nf + 2 * I;
  const T s0 = (f[0] + f[1]) + (f[nf] + f[nf + 1]);
  const T s1 = (f[pl] + f[pl + 1]) + (f[pl + nf] + f[pl + nf + 1]);
  kc[(int64_t)b * esc + ((int64_t)K * nc + J) * nc + I] = T(0.125) * (s0 + s1);
  if (prof.acc && I == 0 && J == 0 && K == 0) atomicAdd(prof.acc, prof.per_sample);
}

__global__ void k_cast_kappa(int64_t ne, int64_t es, const double* __restrict__ k64,
                             float* __restrict__ k32) {
  const int64_t b = blockIdx.y;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne;
       e += (int64_t)gridDim.x * blockDim.x)
    k32[b * es + e] = (float)k64[b * es + e];
}

}  // namespace

// 2^(j/64), j < 64, for kle_exp: set once per device (not under stream capture).
cudaError_t init_kle_exp() {
  static std::atomic<uint64_t> done{0};
  return once_per_device(done, [] {
    double tab[EXP_TAB];
    for (int j = 0; j < EXP_TAB; ++j) tab[j] = (double)std::exp2((long double)j / EXP_TAB);
    return cudaMemcpyToSymbol(g_exp2_tab, tab, sizeof(tab));
  });
}

cudaError_t launch_cast_kappa(cudaStream_t s, const Grid& g, const double* k64, float* k32,
                              int64_t B) {
  if (B == 0) return cudaSuccess;
  const int64_t ne = ipow(g.n, g.dim);
  const int64_t blocks = std::min<int64_t>((ne + 255) / 256, 4096);
  k_cast_kappa<<<dim3((unsigned)blocks, (unsigned)B), 256, 0, s>>>(ne, g.es, k64, k32);
  return cudaGetLastError();
}

cudaError_t launch_kle_table(cudaStream_t s, int n, int m, const double* omega,
                             const double* theta, const int32_t* even, double* table) {
  const int total = n * m;
  k_kle_table<<<(total + 255) / 256, 256, 0, s>>>(n, m, omega, theta, even, table);
  return cudaGetLastError();
}

cudaError_t launch_kappa(cudaStream_t s, const Grid& g, int m, double sqrt_sigma2,
                         const double* table, const double* xi, int M_xi, const int32_t* slot,
                         int64_t B, double* kappa, Prof p) {
  if (B == 0) return cudaSuccess;
  if (g.dim == 2) {
    const int half = (g.n + 1) / 2;
    dim3 grid((g.n + TX2 - 1) / TX2, (half + TY2 * KAP_ROWS - 1) / (TY2 * KAP_ROWS), (unsigned)B);
    k_kappa2d<<<grid, dim3(TX2, TY2), 0, s>>>(g.n, m, sqrt_sigma2, table, xi, M_xi, slot, g.es, kappa, p);
  } else {
    const int M = m * m * m;
    const size_t smem = sizeof(double) * ((size_t)M + (size_t)TX2 * m * m + (size_t)TX2 * K3_TY * m);
    static std::atomic<uint64_t> opted{0};
    const cudaError_t attr = once_per_device(opted, [] {
      return cudaFuncSetAttribute(k_kappa3d, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    });
    if (attr != cudaSuccess) return attr;
    dim3 grid((g.n + TX2 - 1) / TX2, (g.n + K3_TY - 1) / K3_TY, (unsigned)B);
    k_kappa3d<<<grid, dim3(TX2, K3_TY), smem, s>>>(g.n, m, sqrt_sigma2, table, xi, M_xi, slot, g.es,
                                                   kappa, p);
  }
  return cudaGetLastError();
}

cudaError_t launch_kappa32(cudaStream_t s, const Grid& g, int m, double sqrt_sigma2, const double* table,
                           const double* xi, int M_xi, const int32_t* slot, int64_t B, float* kappa32) {
  if (B == 0) return cudaSuccess;
  const float scale = (float)(sqrt_sigma2 * 1.4426950408889634074);   // 1 / ln 2
  const dim3 block(TX2, K32_Y);
  if (g.dim == 2) {
    const dim3 grid((g.n + TX2 - 1) / TX2, ((g.n + 1) / 2 + K32_ROWS - 1) / K32_ROWS, (unsigned)B);
    k_kappa32_2d<<<grid, block, 0, s>>>(g.n, m, scale, table, xi, M_xi, slot, g.es, kappa32);
  } else {
    static std::atomic<uint64_t> opted{0};
    const cudaError_t attr = once_per_device(opted, [] {
      return cudaFuncSetAttribute(k_kappa32_3d, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    });
    if (attr != cudaSuccess) return attr;
    const dim3 grid((g.n + TX2 - 1) / TX2, (g.n + K32_Y - 1) / K32_Y, (unsigned)B);
    k_kappa32_3d<<<grid, block, k32_smem3(g.n, m), s>>>(g.n, m, k32_half(g.n), scale, table, xi, M_xi, slot, g.es,
                                                        kappa32);
  }
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_coarsen(cudaStream_t s, const Grid& fine, const Grid& coarse,
                           const T* kf, T* kc, int64_t B, Prof p) {
  if (B == 0) return cudaSuccess;
  const int nc = coarse.n;
  const int threads = nc < 128 ? ((nc + 31) / 32) * 32 : 128;
  if (fine.dim == 2) {
    dim3 grid((nc + threads - 1) / threads, nc, (unsigned)B);
    k_coarsen2d<T><<<grid, threads, 0, s>>>(nc, kf, kc, fine.es, coarse.es, p);
  } else {
    dim3 grid((nc + threads - 1) / threads, nc * nc, (unsigned)B);
    k_coarsen3d<T><<<grid, threads, 0, s>>>(nc, kf, kc, fine.es, coarse.es, p);
  }
  return cudaGetLastError();
}

template cudaError_t launch_coarsen<double>(cudaStream_t, const Grid&, const Grid&, const double*,
                                            double*, int64_t, Prof);
template cudaError_t launch_coarsen<float>(cudaStream_t, const Grid&, const Grid&, const float*,
                                           float*, int64_t, Prof);

}  // namespace mlmc
