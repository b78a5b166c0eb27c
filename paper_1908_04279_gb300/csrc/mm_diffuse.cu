// Filament diffusion (the -D_t grad ln psi and -D_r d_theta ln psi fluxes of
// Eq. 2-3: d_t psi = D_t lap_x psi + D_r d_theta^2 psi) by Crank-Nicolson, the
// scheme Sec. 2 / Alg. 1 use for the diffusive terms of the psi update, taken
// one direction at a time (theta, x, y). Each direction is a batch of
// constant-coefficient periodic tridiagonal systems
//   (I - a/2 L) psi' = (I + a/2 L) psi,  (L psi)_i = psi_{i-1} - 2 psi_i + psi_{i+1},
// one per line. Arithmetic in float64, storage in the state precision, in place.
//
// k_cn_block uses I + a/2 L = 2 I - (I - a/2 L): psi' = 2 q - psi with
// (I - a/2 L) q = psi, which keeps the right side positive (with L psi formed
// first, a stiff step, a = 16000, lost a digit more), and solves for q by two
// first-order cyclic recursions. With S the cyclic shift, I - a/2 L = kappa (I -
// r S)(I - r S^-1) where r = a / (1 + a + sqrt(1 + 2 a)) (0 < r < 1) and kappa =
// a / (2 r): solve y_i = d_i + r y_{i-1}, then q_i = y_i + r q_{i+1}, both cyclic,
// d = psi / kappa. There are no factors to compute or to read, and a recursion
// splits: a block takes 32 lines (a lane each, so that neighbouring lanes read
// neighbouring addresses) and cuts them into one segment per warp; a segment's
// value at its end from a zero start is known at once, and the true starts
// follow from the other segments' ends and powers of r. The lines live in shared
// memory between the passes, and psi is rounded to the state precision once per
// direction. Bound by the float64 pipe (8 operations a value) and latency: 128^2 x
// 32, three directions, 321 (a thread per line, and the factors on one thread)
// -> 51 us.
//
// k_cn_lines, a thread per line with a Thomas sweep and the corners by the
// Sherman-Morrison formula, stays for lines too long for shared memory.
#include <cmath>

#include "mm_internal.cuh"

namespace mm {

namespace {

// Factors of one periodic direction of n >= 2 points with a = D dt / h^2
// (one thread per direction): the matrix I - a/2 L (diagonal b = 1 + a,
// off-diagonals and corners c = -a/2) is T + u v^T with T tridiagonal
// (corners removed, T_00 = b - gamma, T_{n-1,n-1} = b - c^2 / gamma,
// gamma = -b), u = (gamma, 0, .., 0, c), v = (1, 0, .., 0, c / gamma).
// tab: cp[n], 1/m[n] of T's Thomas elimination, z[n] = T^{-1} u, then
// r = c / gamma and vzf = 1 / (1 + v.z).
__global__ void k_cn_factors(double* tab0, int n0, double a0, double* tab1, int n1, double a1,
                             double* tab2, int n2, double a2) {
  const int d = threadIdx.x;
  if (d > 2 || blockIdx.x != 0) return;
  double* tab = d == 0 ? tab0 : d == 1 ? tab1 : tab2;
  const int n = d == 0 ? n0 : d == 1 ? n1 : n2;
  const double a = d == 0 ? a0 : d == 1 ? a1 : a2;
  if (!(a > 0.0) || n < 2) return;
  const double b = 1.0 + a, c = -0.5 * a, gamma = -b;
  double* cp = tab;
  double* im = tab + n;
  double* z = tab + 2 * n;
  for (int i = 0; i < n; ++i) {
    double diag = b;
    if (i == 0) diag = b - gamma;
    if (i == n - 1) diag = b - c * c / gamma;
    const double m = i == 0 ? diag : diag - c * cp[i - 1];
    im[i] = 1.0 / m;
    cp[i] = c / m;
  }
  for (int i = 0; i < n; ++i) {  // T z = u
    const double ui = i == 0 ? gamma : (i == n - 1 ? c : 0.0);
    z[i] = (ui - (i == 0 ? 0.0 : c * z[i - 1])) * im[i];
  }
  for (int i = n - 2; i >= 0; --i) z[i] -= cp[i] * z[i + 1];
  const double r = c / gamma;
  tab[3 * n] = r;
  tab[3 * n + 1] = 1.0 / (1.0 + z[0] + r * z[n - 1]);
}

// One direction for every line: c = -a/2, ha = a/2, the factors in tab.
template <typename T>
__global__ void k_cn_lines(T* psi, int mode, int nx, int ny, int nth, const double* tab, int n,
                           double c, double ha, const double* scale) {
  const long long nlines = mode == 0 ? (long long)nx * ny : mode == 1 ? (long long)ny * nth
                                                                      : (long long)nx * nth;
  const double g = scale ? *scale : 1.0;
  const double* cp = tab;
  const double* im = tab + n;
  const double* z = tab + 2 * n;
  const double r = tab[3 * n], vzf = tab[3 * n + 1];
  for (long long L = blockIdx.x * (long long)blockDim.x + threadIdx.x; L < nlines;
       L += (long long)gridDim.x * blockDim.x) {
    size_t base, stride;
    if (mode == 0) {  // theta: a row of the cell, contiguous
      base = (size_t)L * nth;
      stride = 1;
    } else if (mode == 1) {  // x: line (y, k), stride nth
      const long long y = L / nth, k = L - y * nth;
      base = (size_t)y * nx * nth + (size_t)k;
      stride = (size_t)nth;
    } else {  // y: line (x, k), stride nx nth
      const long long x = L / nth, k = L - x * nth;
      base = (size_t)x * nth + (size_t)k;
      stride = (size_t)nx * nth;
    }
    T* p = psi + base;
    // forward sweep with the explicit half step as right-hand side
    const double first = g * (double)p[0];
    double prev = g * (double)p[(size_t)(n - 1) * stride], cur = first, yp = 0.0;
    for (int i = 0; i < n; ++i) {
      const double next = i + 1 < n ? g * (double)p[(size_t)(i + 1) * stride] : first;
      const double d = fma(ha, prev + next, (1.0 - 2.0 * ha) * cur);
      yp = (d - c * yp) * im[i];
      p[(size_t)i * stride] = (T)yp;
      prev = cur;
      cur = next;
    }
    // back substitution (y_{n-1} = y'_{n-1})
    const double ylast = yp;
    double y = yp;
    for (int i = n - 2; i >= 0; --i) {
      y = (double)p[(size_t)i * stride] - cp[i] * y;
      p[(size_t)i * stride] = (T)y;
    }
    // periodic corners: x = y - (v.y) / (1 + v.z) z, v = (1, 0, .., 0, r)
    const double beta = (y + r * ylast) * vzf;
    for (int i = 0; i < n; ++i)
      p[(size_t)i * stride] = (T)((double)p[(size_t)i * stride] - beta * z[i]);
  }
}

constexpr int kCnPitch = 33;   // shared-memory row of 32 lines, padded
constexpr int kCnWarps = 16;   // segments of a line at most

// One direction for 32 lines per block: ik = 1 / kappa; rl and re: r to the
// segment length and to the last segment's; wrap = 1 / (1 - r^n). len: points
// per segment.
template <typename T>
__global__ void __launch_bounds__(32 * kCnWarps)
    k_cn_block(T* psi, int mode, int nx, int ny, int nth, int n, int len, double r, double ik,
               double rl, double re, double wrap, const double* scale) {
  extern __shared__ __align__(16) double cn_t[];  // [n][kCnPitch], then [2][warps][32]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double* ends = cn_t + (size_t)n * kCnPitch;
  const long long nlines = mode == 0 ? (long long)nx * ny : mode == 1 ? (long long)ny * nth
                                                                      : (long long)nx * nth;
  const long long L0 = blockIdx.x * 32LL, Ln = L0 + lane;
  const bool on = Ln < nlines;
  const long long La = on ? Ln : nlines - 1;
  // first value and stride of the lane's line
  size_t base, stride;
  if (mode == 0) {
    base = (size_t)La * nth;
    stride = 1;
  } else if (mode == 1) {
    const long long y = La / nth;
    base = (size_t)y * nx * nth + (size_t)(La - y * nth);
    stride = (size_t)nth;
  } else {
    base = (size_t)La;
    stride = (size_t)nx * nth;
  }
  const double g = scale ? *scale : 1.0;
  const double gk = ik * g;
  const int i0 = w * len, i1 = min(n, i0 + len);
  // a theta line is contiguous: the block's lines as one run, transposed
  // through shared memory
  if (mode == 0) {
    const int cnt = (int)min(32LL, nlines - L0) * nth;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
      const int l = e / nth, i = e - l * nth;
      cn_t[i * kCnPitch + l] = (double)psi[(size_t)L0 * nth + e];
    }
    __syncthreads();
  }
  // d, and the segment's end of the forward recursion from a zero start
  double acc = 0.0;
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    const double d =
        gk * (mode == 0 ? cn_t[i * kCnPitch + lane] : (double)psi[base + (size_t)i * stride]);
    cn_t[i * kCnPitch + lane] = d;
    acc = fma(r, acc, d);
  }
  ends[w * 32 + lane] = acc;
  __syncthreads();
  // the value before the segment: one turn over all segments, closed by wrap
  double y = 0.0;
  for (int q = 0; q < nw; ++q) {
    const int s = w + q < nw ? w + q : w + q - nw;
    y = fma(s == nw - 1 ? re : rl, y, ends[s * 32 + lane]);
  }
  y *= wrap;
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    y = fma(r, y, cn_t[i * kCnPitch + lane]);
    cn_t[i * kCnPitch + lane] = y;
  }
  // the backward recursion in the same way
  acc = 0.0;
#pragma unroll 4
  for (int i = i1 - 1; i >= i0; --i) acc = fma(r, acc, cn_t[i * kCnPitch + lane]);
  ends[(nw + w) * 32 + lane] = acc;
  __syncthreads();
  double x = 0.0;
  for (int q = 0; q < nw; ++q) {
    const int s = w - q >= 0 ? w - q : w - q + nw;
    x = fma(s == nw - 1 ? re : rl, x, ends[(nw + s) * 32 + lane]);
  }
  x *= wrap;
#pragma unroll 4
  for (int i = i1 - 1; i >= i0; --i) {
    x = fma(r, x, cn_t[i * kCnPitch + lane]);
    if (mode == 0)
      cn_t[i * kCnPitch + lane] = x;
    else if (on) {
      T* p = psi + base + (size_t)i * stride;
      *p = (T)fma(2.0, x, -g * (double)*p);
    }
  }
  if (mode == 0) {
    __syncthreads();
    const int cnt = (int)min(32LL, nlines - L0) * nth;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
      const int l = e / nth, i = e - l * nth;
      T* p = psi + (size_t)L0 * nth + e;
      *p = (T)fma(2.0, cn_t[i * kCnPitch + l], -g * (double)*p);
    }
  }
}

__global__ void k_set_scale_one(double* scale) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *scale = 1.0;
}

}  // namespace

cudaError_t launch_cn_factors(double* tab0, int n0, double a0, double* tab1, int n1, double a1,
                              double* tab2, int n2, double a2, cudaStream_t s) {
  k_cn_factors<<<1, 32, 0, s>>>(tab0, n0, a0, tab1, n1, a1, tab2, n2, a2);
  return cudaGetLastError();
}

// Shared memory of k_cn_block for lines of n points in `warps` segments.
size_t cn_block_smem(int n, int warps) {
  return ((size_t)n * kCnPitch + 2 * (size_t)warps * 32) * sizeof(double);
}
bool cn_block_fits(int n) { return cn_block_smem(n, kCnWarps) <= 227 * 1024; }

// One direction of n >= 2 points, a = D dt / h^2 > 0, by k_cn_block.
template <typename T>
cudaError_t launch_cn_block(T* psi, int mode, int nx, int ny, int nth, int n, double a,
                            const double* scale, cudaStream_t s) {
  const long long nlines = mode == 0 ? (long long)nx * ny : mode == 1 ? (long long)ny * nth
                                                                      : (long long)nx * nth;
  // segments of at least 8 points
  int warps = n / 8 < 1 ? 1 : n / 8 > kCnWarps ? kCnWarps : n / 8;
  const int len = (n + warps - 1) / warps;
  warps = (n + len - 1) / len;
  const size_t smem = cn_block_smem(n, warps);
  if (smem > 48 * 1024) {
    const cudaError_t e = raise_smem_limit(k_cn_block<T>, smem);
    if (e != cudaSuccess) return e;
  }
  const double r = a / (1.0 + a + sqrt(1.0 + 2.0 * a)), kappa = 0.5 * a / r;
  const double rl = pow(r, len), re = pow(r, n - (warps - 1) * len);
  const double wrap = 1.0 / (-expm1(n * log(r)));
  k_cn_block<T><<<(unsigned)((nlines + 31) / 32), 32 * warps, smem, s>>>(
      psi, mode, nx, ny, nth, n, len, r, 1.0 / kappa, rl, re, wrap, scale);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cn_lines(T* psi, int mode, int nx, int ny, int nth, const double* tab, int n,
                            double c, double ha, const double* scale, cudaStream_t s) {
  const long long nlines = mode == 0 ? (long long)nx * ny : mode == 1 ? (long long)ny * nth
                                                                      : (long long)nx * nth;
  long long g = (nlines + 127) / 128;
  if (g > 152LL * 32) g = 152LL * 32;
  k_cn_lines<T><<<(int)g, 128, 0, s>>>(psi, mode, nx, ny, nth, tab, n, c, ha, scale);
  return cudaGetLastError();
}

cudaError_t launch_set_scale_one(double* scale, cudaStream_t s) {
  k_set_scale_one<<<1, 32, 0, s>>>(scale);
  return cudaGetLastError();
}

template cudaError_t launch_cn_block<float>(float*, int, int, int, int, int, double,
                                            const double*, cudaStream_t);
template cudaError_t launch_cn_block<double>(double*, int, int, int, int, int, double,
                                             const double*, cudaStream_t);
template cudaError_t launch_cn_lines<float>(float*, int, int, int, int, const double*, int, double,
                                            double, const double*, cudaStream_t);
template cudaError_t launch_cn_lines<double>(double*, int, int, int, int, const double*, int,
                                             double, double, const double*, cudaStream_t);

}  // namespace mm
