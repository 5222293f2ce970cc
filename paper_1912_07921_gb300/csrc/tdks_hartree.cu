// Hartree potential of the density (the density-dependent potential beside exchange in the
// Kohn-Sham Hamiltonian, which CFM4 of Sec. "New propagators for real-time TDDFT"
// extrapolates as part of Hxc):
//   finite box:     v_H(r_i) = h^3 sum_j K(r_i - r_j) n_j,  K(d) = 1/|d|,  K(0) = c0 / h,
//                   c0 = 3 ln(2 + sqrt 3) - pi/2 (the Coulomb integral of a cell over itself);
//                   a linear convolution, computed exactly by a zero-padded FFT (Hockney):
//                   v = IFFT(FFT(n padded) FFT(K padded)) on a grid of >= 2n - 1 points per axis;
//   periodic cell:  v_H(G) = 4 pi n(G) / |G|^2 on the grid's plane waves (G the alias nearest
//                   zero), G = 0 dropped (neutralising background).
//
// Five launches per solve, all FP64: x forward, y forward, z (forward, times the kernel, inverse),
// y inverse, x inverse.
//   * The density is real: two x lines are transformed as one complex line, and only the
//     hx = px/2 + 1 columns of the half spectrum go on.  The kernel's transform is real (K is real
//     and even on the padded grid).
//   * Padding is never stored in z nor read in x and y: lines of zeros are skipped (a quarter of the
//     x lines, half of the y lines of a box are transformed), zeros enter in shared memory, and
//     each inverse transform writes the box's points only.  The spectrum buffer is hx py nz values.
//   * Line transforms are mixed-radix Stockham passes in shared memory (Govindaraju et al., SC 2008:
//     each pass takes R values N/R apart, twiddles them, does an R-point DFT and stores them in
//     autosorted order), radices 8, 4, 2, 3, 5, 7, 11, 13, twiddles from a table.  A CTA takes LB
//     adjacent lines, value-major ([i][line]), so that strided axes are read in runs of LB values and,
//     with LB = 8 (lengths up to 512), no pass has a bank conflict.
// Bound by the FP64 pipe (2 instructions per clock per SM) and, at small grids, by five launches: a
// 128^3 padded transform pair is ~8e7 FP64 instructions, 0.13 ms.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "tdks_system.h"

using namespace tdks;
using namespace tdks_host;

namespace {

constexpr int FFT_THREADS = 128;
constexpr int FFT_MAXR = 13;      // largest radix (prime factor of a line length)
constexpr int FFT_MAXN = 1024;    // longest line

struct FftPlan {
  int n;                // line length
  int nrad, rad[12];    // radices, in the order the passes take them
  const double2 *tw;    // (cos, sin) of 2 pi j / n
};

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// e^{sign i angle} from the table's (cos, sin)
template <int SIGN> __device__ __forceinline__ double2 tw_of(double2 t) { return make_double2(t.x, SIGN < 0 ? -t.y : t.y); }
// SIGN i a
template <int SIGN> __device__ __forceinline__ double2 muli(double2 a) {
  return SIGN < 0 ? make_double2(a.y, -a.x) : make_double2(-a.y, a.x);
}

// R-point DFTs in place, v[q] <- sum_r v[r] e^{SIGN 2 pi i r q / R}
template <int R, int SIGN> struct Dft {  // odd prime R: pairs r, R - r
  static __device__ __forceinline__ void run(double2 *v, const double2 *tw, int n) {
    double2 s[(R - 1) / 2], d[(R - 1) / 2], o[R];
#pragma unroll
    for (int r = 1; r <= (R - 1) / 2; r++) {
      s[r - 1] = cadd(v[r], v[R - r]);
      d[r - 1] = muli<SIGN>(csub(v[r], v[R - r]));
    }
    o[0] = v[0];
#pragma unroll
    for (int r = 0; r < (R - 1) / 2; r++) o[0] = cadd(o[0], s[r]);
    const int st = n / R;
#pragma unroll
    for (int q = 1; q <= (R - 1) / 2; q++) {
      double2 c = v[0], e = make_double2(0.0, 0.0);
#pragma unroll
      for (int r = 1; r <= (R - 1) / 2; r++) {
        const double2 w = tw[((r * q) % R) * st];
        c.x += w.x * s[r - 1].x;
        c.y += w.x * s[r - 1].y;
        e.x += w.y * d[r - 1].x;
        e.y += w.y * d[r - 1].y;
      }
      o[q] = cadd(c, e);
      o[R - q] = csub(c, e);
    }
#pragma unroll
    for (int q = 0; q < R; q++) v[q] = o[q];
  }
};
template <int SIGN> struct Dft<2, SIGN> {
  static __device__ __forceinline__ void run(double2 *v, const double2 *, int) {
    const double2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};
template <int SIGN> struct Dft<4, SIGN> {
  static __device__ __forceinline__ void run(double2 *v, const double2 *, int) {
    const double2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = muli<SIGN>(csub(v[1], v[3]));
    v[0] = cadd(a, c);
    v[1] = cadd(b, d);
    v[2] = csub(a, c);
    v[3] = csub(b, d);
  }
};
template <int SIGN> struct Dft<8, SIGN> {
  static __device__ __forceinline__ void run(double2 *v, const double2 *, int) {
    double2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4, SIGN>::run(e, nullptr, 0);
    Dft<4, SIGN>::run(o, nullptr, 0);
    constexpr double h = 0.70710678118654752440;  // sqrt(1/2)
    // o[k] e^{SIGN i pi k / 4}
    const double2 i1 = muli<SIGN>(o[1]), i3 = muli<SIGN>(o[3]);
    o[1] = make_double2(h * (o[1].x + i1.x), h * (o[1].y + i1.y));
    o[2] = muli<SIGN>(o[2]);
    o[3] = make_double2(h * (i3.x - o[3].x), h * (i3.y - o[3].y));
#pragma unroll
    for (int k = 0; k < 4; k++) {
      v[k] = cadd(e[k], o[k]);
      v[k + 4] = csub(e[k], o[k]);
    }
  }
};

// One Stockham pass of radix R over LB lines: a -> b.
template <int R, int SIGN, int LB>
__device__ __forceinline__ void fft_pass(const double2 *a, double2 *b, const FftPlan &p, int Ns) {
  const int m = p.n / R, step = p.n / (Ns * R);
  for (int t = threadIdx.x; t < m * LB; t += FFT_THREADS) {
    const int l = t % LB, j = t / LB;
    const int jn = j / Ns, k = j - jn * Ns;
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = a[(j + r * m) * LB + l];
    if (k != 0) {
#pragma unroll
      for (int r = 1; r < R; r++) v[r] = cmul(v[r], tw_of<SIGN>(p.tw[k * r * step]));
    }
    Dft<R, SIGN>::run(v, p.tw, p.n);
    double2 *o = b + (jn * Ns * R + k) * LB + l;
#pragma unroll
    for (int q = 0; q < R; q++) o[q * Ns * LB] = v[q];
  }
}

// Transform of the LB lines in a (b: as much scratch); the result is in a again on return.
// BIG: lengths with prime factors above 5 (periodic cells); the others' kernels keep half the registers.
template <int SIGN, int LB, bool BIG>
__device__ __forceinline__ void fft_lines(double2 *&a, double2 *&b, const FftPlan &p) {
  int Ns = 1;
  for (int i = 0; i < p.nrad; i++) {
    __syncthreads();
    switch (p.rad[i]) {
      case 2: fft_pass<2, SIGN, LB>(a, b, p, Ns); break;
      case 3: fft_pass<3, SIGN, LB>(a, b, p, Ns); break;
      case 4: fft_pass<4, SIGN, LB>(a, b, p, Ns); break;
      case 5: fft_pass<5, SIGN, LB>(a, b, p, Ns); break;
      case 8: fft_pass<8, SIGN, LB>(a, b, p, Ns); break;
      default:
        if constexpr (BIG) {
          if (p.rad[i] == 7) fft_pass<7, SIGN, LB>(a, b, p, Ns);
          else if (p.rad[i] == 11) fft_pass<11, SIGN, LB>(a, b, p, Ns);
          else fft_pass<13, SIGN, LB>(a, b, p, Ns);
        }
    }
    Ns *= p.rad[i];
    double2 *t = a;
    a = b;
    b = t;
  }
  __syncthreads();
}

// Real x lines -> half spectrum.  Line l = z ny + y of src (nx values, zeros beyond) goes to row
// z py + y of buf (hx values); lines 2q and 2q + 1 are one complex line.
template <int LB, bool BIG>
__global__ void __launch_bounds__(FFT_THREADS, BIG ? 1 : 6)
fft_x_forward(const double *src, double2 *buf, const FftPlan p, int nx, int ny, int py, long lines) {
  extern __shared__ double2 sm[];
  double2 *a = sm, *b = sm + p.n * LB;
  const int n = p.n, hx = n / 2 + 1;
  const long l0 = blockIdx.x * 2L * LB;
  for (int t = threadIdx.x; t < n * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    const long la = l0 + 2 * l, lb = la + 1;
    double2 v = make_double2(0.0, 0.0);
    if (i < nx) {
      if (la < lines) v.x = src[la * nx + i];
      if (lb < lines) v.y = src[lb * nx + i];
    }
    a[t] = v;
  }
  fft_lines<-1, LB, BIG>(a, b, p);
  for (int t = threadIdx.x; t < hx * LB; t += FFT_THREADS) {
    const int l = t % LB, k = t / LB;
    const long la = l0 + 2 * l, lb = la + 1;
    const double2 z = a[k * LB + l], y = a[(k ? n - k : 0) * LB + l];
    // A = (Z[k] + conj Z[-k]) / 2, B = (Z[k] - conj Z[-k]) / 2i
    if (la < lines) buf[((la / ny) * py + la % ny) * hx + k] = make_double2(0.5 * (z.x + y.x), 0.5 * (z.y - y.y));
    if (lb < lines) buf[((lb / ny) * py + lb % ny) * hx + k] = make_double2(0.5 * (z.y + y.y), 0.5 * (y.x - z.x));
  }
}

// The inverse of fft_x_forward: half spectra -> real lines, times scale.
template <int LB, bool BIG>
__global__ void __launch_bounds__(FFT_THREADS, BIG ? 1 : 6)
fft_x_inverse(const double2 *buf, double *dst, const FftPlan p, int nx, int ny, int py, long lines, double scale) {
  extern __shared__ double2 sm[];
  double2 *a = sm, *b = sm + p.n * LB;
  const int n = p.n, hx = n / 2 + 1;
  const long l0 = blockIdx.x * 2L * LB;
  for (int t = threadIdx.x; t < hx * LB; t += FFT_THREADS) {
    const int l = t % LB, k = t / LB;
    const long la = l0 + 2 * l, lb = la + 1;
    double2 A = make_double2(0.0, 0.0), B = A;
    if (la < lines) A = buf[((la / ny) * py + la % ny) * hx + k];
    if (lb < lines) B = buf[((lb / ny) * py + lb % ny) * hx + k];
    // a real line's spectrum: imaginary parts at 0 and n/2 are zero up to rounding and drop out
    if (k == 0 || 2 * k == n) A.y = B.y = 0.0;
    a[k * LB + l] = make_double2(A.x - B.y, A.y + B.x);
    if (k > 0 && 2 * k < n) a[(n - k) * LB + l] = make_double2(A.x + B.y, B.x - A.y);
  }
  fft_lines<1, LB, BIG>(a, b, p);
  for (int t = threadIdx.x; t < nx * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    const long la = l0 + 2 * l, lb = la + 1;
    const double2 v = a[i * LB + l];
    if (la < lines) dst[la * nx + i] = scale * v.x;
    if (lb < lines) dst[lb * nx + i] = scale * v.y;
  }
}

// Lines along y (SIGN -1: n_in = ny values in, py out; +1: py in, ny out) of LB adjacent columns.
template <int SIGN, int LB, bool BIG>
__global__ void __launch_bounds__(FFT_THREADS, BIG ? 1 : 6) fft_y(double2 *buf, const FftPlan p, int hx, int n_in, int n_out) {
  extern __shared__ double2 sm[];
  double2 *a = sm, *b = sm + p.n * LB;
  const int n = p.n, x0 = blockIdx.x * LB;
  double2 *base = buf + (long)blockIdx.y * n * hx + x0;
  for (int t = threadIdx.x; t < n * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    a[t] = i < n_in && x0 + l < hx ? base[(long)i * hx + l] : make_double2(0.0, 0.0);
  }
  fft_lines<SIGN, LB, BIG>(a, b, p);
  for (int t = threadIdx.x; t < n_out * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    if (x0 + l < hx) base[(long)i * hx + l] = a[t];
  }
}

// Lines along z: forward, times the kernel's transform, inverse (nz values in and out).
// kout: forward only, the real part of the transform of a kernel's lines (pz values in) to kout.
template <int LB, bool BIG>
__global__ void __launch_bounds__(FFT_THREADS, BIG ? 1 : 6)
fft_z(double2 *buf, const FftPlan p, int hx, int nz, const double *kern, double *kout) {
  extern __shared__ double2 sm[];
  double2 *a = sm, *b = sm + p.n * LB;
  const int n = p.n, x0 = blockIdx.x * LB;
  const long stride = (long)gridDim.y * hx, at = (long)blockIdx.y * hx + x0;
  for (int t = threadIdx.x; t < n * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    a[t] = i < nz && x0 + l < hx ? buf[at + i * stride + l] : make_double2(0.0, 0.0);
  }
  fft_lines<-1, LB, BIG>(a, b, p);
  for (int t = threadIdx.x; t < n * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    if (x0 + l >= hx) continue;
    if (kout) {
      kout[at + i * stride + l] = a[t].x;
    } else {
      const double k = kern[at + i * stride + l];
      a[t] = make_double2(k * a[t].x, k * a[t].y);
    }
  }
  if (kout) return;
  fft_lines<1, LB, BIG>(a, b, p);
  for (int t = threadIdx.x; t < nz * LB; t += FFT_THREADS) {
    const int l = t % LB, i = t / LB;
    if (x0 + l < hx) buf[at + i * stride + l] = a[t];
  }
}

// the sampled kernel on the padded grid: offsets 0..n-1 at indices 0..n-1, offsets -(n-1)..-1
// at indices P-(n-1)..P-1, zero in between (never met by a linear convolution of n points)
__global__ void hartree_kernel_box(int nx, int ny, int nz, int px, int py, int pz, double h, double self,
                                   double *kern) {
  const long P = (long)px * py * pz;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < P; i += (long)gridDim.x * blockDim.x) {
    const int x = (int)(i % px), y = (int)((i / px) % py), z = (int)(i / ((long)px * py));
    const int dx = x < nx ? x : (x > px - nx ? x - px : INT32_MAX);
    const int dy = y < ny ? y : (y > py - ny ? y - py : INT32_MAX);
    const int dz = z < nz ? z : (z > pz - nz ? z - pz : INT32_MAX);
    double v = 0.0;
    if (dx != INT32_MAX && dy != INT32_MAX && dz != INT32_MAX) {
      if (dx == 0 && dy == 0 && dz == 0) v = self / h;
      else v = 1.0 / (h * sqrt((double)dx * dx + (double)dy * dy + (double)dz * dz));
    }
    kern[i] = v;
  }
}

// periodic cell: 4 pi / |G|^2 with G the alias of each index nearest zero, 0 at G = 0, over
// the number of points (the inverse transform is unscaled), on the half spectrum
__global__ void hartree_kernel_cell(int nx, int ny, int nz, double Lx, double Ly, double Lz, double *kern) {
  const long N = (long)nx * ny * nz;
  const int hx = nx / 2 + 1;
  const long H = (long)hx * ny * nz;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < H; i += (long)gridDim.x * blockDim.x) {
    const int x = (int)(i % hx), y = (int)((i / hx) % ny), z = (int)(i / ((long)hx * ny));
    const int ay = y <= ny / 2 ? y : y - ny, az = z <= nz / 2 ? z : z - nz;
    const double gx = 2.0 * M_PI * x / Lx, gy = 2.0 * M_PI * ay / Ly, gz = 2.0 * M_PI * az / Lz;
    const double g2 = gx * gx + gy * gy + gz * gz;
    kern[i] = i == 0 ? 0.0 : 4.0 * M_PI / g2 / (double)N;
  }
}

// radices of a line length: 8, 4 and 2 for its powers of two, then its odd primes (<= 13).  (At most six
// for lengths up to FFT_MAXN; longer ones, which have no room for theirs, are refused first.)
bool factor(int n, FftPlan &p) {
  p.n = n;
  p.nrad = 0;
  if (n > FFT_MAXN) return false;
  int m = n;
  const int rad[] = {8, 4, 2, 3, 5, 7, 11, 13};
  for (int r : rad)
    while (m % r == 0) {
      // (16 = 4 * 4 rather than 8 * 2)
      if (r == 8 && m % 16 == 0 && m % 32 != 0) break;
      p.rad[p.nrad++] = r;
      m /= r;
    }
  return m == 1;
}

// smallest length >= m whose prime factors are 2 and 3
int smooth_at_least(int m) {
  for (int c = m;; c++) {
    int r = c;
    while (r % 2 == 0) r /= 2;
    while (r % 3 == 0) r /= 3;
    if (r == 1) return c;
  }
}

int grid_blocks(long n) {
  const long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 152L * 16 ? 152L * 16 : b));
}

// the three axes' plans of a padded array (twiddle tables after one another at tw)
bool plans(const int hp[3], const double2 *tw, FftPlan p[3]) {
  for (int a = 0; a < 3; a++) {
    if (!factor(hp[a], p[a])) return false;
    p[a].tw = tw;
    if (tw) tw += hp[a];
  }
  return true;
}

// lines per CTA of transforms of length n: two buffers of 16 n bytes per line, 128 KB at most
int lines_of(int n) { return n <= 512 ? 8 : 4; }
size_t smem_of(int n) { return 2ul * lines_of(n) * n * sizeof(double2); }

template <auto K>
cudaError_t big_smem() {
  static std::atomic<unsigned> done{0};  // (one per kernel)
  return ensure_smem_attr(K, 2ul * 8 * 512 * sizeof(double2), done);
}

// f(LB, BIG) as compile-time constants for a line length
template <class F>
cudaError_t by_length(const FftPlan &p, F f) {
  const bool big = p.n > 1 && p.rad[p.nrad - 1] > 5 && p.rad[p.nrad - 1] != 8;
  if (lines_of(p.n) == 8)
    return big ? f(std::integral_constant<int, 8>{}, std::true_type{}) : f(std::integral_constant<int, 8>{}, std::false_type{});
  return big ? f(std::integral_constant<int, 4>{}, std::true_type{}) : f(std::integral_constant<int, 4>{}, std::false_type{});
}

cudaError_t x_forward(const double *src, double2 *buf, const FftPlan &p, int nx, int ny, int nz, int py, cudaStream_t s) {
  return by_length(p, [&](auto lb, auto big) {
    constexpr int LB = decltype(lb)::value;
    constexpr auto k = fft_x_forward<LB, decltype(big)::value>;
    const long lines = (long)ny * nz;
    if (cudaError_t e = big_smem<k>()) return e;
    k<<<(unsigned)((lines + 2 * LB - 1) / (2 * LB)), FFT_THREADS, smem_of(p.n), s>>>(src, buf, p, nx, ny, py, lines);
    return cudaGetLastError();
  });
}

cudaError_t x_inverse(const double2 *buf, double *dst, const FftPlan &p, int nx, int ny, int nz, int py, double scale,
                      cudaStream_t s) {
  return by_length(p, [&](auto lb, auto big) {
    constexpr int LB = decltype(lb)::value;
    constexpr auto k = fft_x_inverse<LB, decltype(big)::value>;
    const long lines = (long)ny * nz;
    if (cudaError_t e = big_smem<k>()) return e;
    k<<<(unsigned)((lines + 2 * LB - 1) / (2 * LB)), FFT_THREADS, smem_of(p.n), s>>>(buf, dst, p, nx, ny, py, lines,
                                                                                 scale);
    return cudaGetLastError();
  });
}

template <int SIGN>
cudaError_t y_lines(double2 *buf, const FftPlan &p, int hx, int nz, int n_in, int n_out, cudaStream_t s) {
  return by_length(p, [&](auto lb, auto big) {
    constexpr int LB = decltype(lb)::value;
    constexpr auto k = fft_y<SIGN, LB, decltype(big)::value>;
    if (cudaError_t e = big_smem<k>()) return e;
    k<<<dim3((hx + LB - 1) / LB, nz), FFT_THREADS, smem_of(p.n), s>>>(buf, p, hx, n_in, n_out);
    return cudaGetLastError();
  });
}

cudaError_t z_lines(double2 *buf, const FftPlan &p, int hx, int py, int nz, const double *kern, double *kout,
                    cudaStream_t s) {
  return by_length(p, [&](auto lb, auto big) {
    constexpr int LB = decltype(lb)::value;
    constexpr auto k = fft_z<LB, decltype(big)::value>;
    if (cudaError_t e = big_smem<k>()) return e;
    k<<<dim3((hx + LB - 1) / LB, py), FFT_THREADS, smem_of(p.n), s>>>(buf, p, hx, nz, kern, kout);
    return cudaGetLastError();
  });
}

}  // namespace

namespace tdks_host {

void hartree_free(tdks_system *s) {
  cudaFree(s->d_hbuf); cudaFree(s->d_hkern); cudaFree(s->d_htw); cudaFree(s->d_vh);
  s->d_hbuf = s->d_htw = nullptr;
  s->d_hkern = nullptr;
  s->d_vh = nullptr;
}

// Workspace, twiddle tables and the transformed kernel of the system's grid.
static int hartree_build(tdks_system *s) {
  int hp[3];
  const int n[3] = {s->nx, s->ny, s->nz};
  const bool box = s->bc == TDKS_BC_ZERO;
  for (int a = 0; a < 3; a++) hp[a] = box ? smooth_at_least(2 * n[a] - 1) : n[a];
  FftPlan p[3];
  if (!plans(hp, nullptr, p))
    return fail(TDKS_EINVAL, "Hartree term: grid edges need prime factors <= 13 and transforms of <= 1024 points");
  for (int a = 0; a < 3; a++) s->hp[a] = hp[a];
  const int hx = hp[0] / 2 + 1;
  const long P = (long)hp[0] * hp[1] * hp[2], row = (long)hx * hp[1];
  std::vector<double2> tw;
  for (int a = 0; a < 3; a++)
    for (int j = 0; j < hp[a]; j++) {
      // (angles reduced to the first octant's neighbourhood: j and hp - j share a cosine)
      const double ang = 2.0 * M_PI * (double)(2 * j <= hp[a] ? j : j - hp[a]) / (double)hp[a];
      tw.push_back(make_double2(std::cos(ang), std::sin(ang)));
    }
  CU(cudaMalloc((void **)&s->d_htw, tw.size() * sizeof(double2)));
  CU(to_device(s->d_htw, tw.data(), tw.size() * sizeof(double2), s->stream));
  CU(cudaMalloc((void **)&s->d_hbuf, row * s->nz * sizeof(double2)));
  CU(cudaMalloc((void **)&s->d_hkern, row * hp[2] * sizeof(double)));
  CU(cudaMalloc((void **)&s->d_vh, s->N * sizeof(double)));
  if (box) {
    // the sampled kernel and its half spectrum: the largest allocations here, for the length of this call
    const double self = 3.0 * std::log(2.0 + std::sqrt(3.0)) - 0.5 * M_PI;
    plans(hp, s->d_htw, p);
    double *k = nullptr;
    double2 *kb = nullptr;
    cudaError_t e = cudaMalloc((void **)&k, P * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void **)&kb, row * hp[2] * sizeof(double2));
    if (e == cudaSuccess) {
      hartree_kernel_box<<<grid_blocks(P), 256, 0, s->stream>>>(s->nx, s->ny, s->nz, hp[0], hp[1], hp[2], s->h, self, k);
      e = x_forward(k, kb, p[0], hp[0], hp[1], hp[2], hp[1], s->stream);
    }
    if (e == cudaSuccess) e = y_lines<-1>(kb, p[1], hx, hp[2], hp[1], hp[1], s->stream);
    if (e == cudaSuccess) e = z_lines(kb, p[2], hx, hp[1], hp[2], nullptr, s->d_hkern, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFree(k);
    cudaFree(kb);
    if (e != cudaSuccess)
      return fail(e == cudaErrorMemoryAllocation ? TDKS_ENOMEM : TDKS_EDEVICE,
                  std::string("Hartree kernel transform: ") + cudaGetErrorString(e));
  } else {
    hartree_kernel_cell<<<grid_blocks(P), 256, 0, s->stream>>>(s->nx, s->ny, s->nz, s->nx * s->h, s->ny * s->h,
                                                               s->nz * s->h, s->d_hkern);
    CU(cudaGetLastError());
    CU(cudaStreamSynchronize(s->stream));
  }
  if (!s->n_total) CU(cudaMalloc((void **)&s->n_total, (size_t)s->N * sizeof(double)));
  return TDKS_OK;
}

// Once, when the Hartree term is turned on: d_vh says that all of it is there, so a set-up that fails
// leaves nothing behind and is done from the beginning the next time.
int hartree_setup(tdks_system *s) {
  if (s->d_vh) return TDKS_OK;
  const int rc = hartree_build(s);
  if (rc) {
    hartree_free(s);
    cudaGetLastError();  // (reported by rc)
  }
  return rc;
}

// v_H of the density in n_total (FP64, N points) into d_vh.
int hartree_solve(tdks_system *s) {
  FftPlan p[3];
  plans(s->hp, s->d_htw, p);
  const int hx = s->hp[0] / 2 + 1, py = s->hp[1];
  const double h3 = s->h * s->h * s->h;
  // box: the unscaled inverse transform is P times the convolution; cell: the kernel holds 1/N
  const double scale = s->bc == TDKS_BC_ZERO ? h3 / ((double)s->hp[0] * s->hp[1] * s->hp[2]) : 1.0;
  cudaError_t e = x_forward(s->n_total, s->d_hbuf, p[0], s->nx, s->ny, s->nz, py, s->stream);
  if (e == cudaSuccess) e = y_lines<-1>(s->d_hbuf, p[1], hx, s->nz, s->ny, py, s->stream);
  if (e == cudaSuccess) e = z_lines(s->d_hbuf, p[2], hx, py, s->nz, s->d_hkern, nullptr, s->stream);
  if (e == cudaSuccess) e = y_lines<1>(s->d_hbuf, p[1], hx, s->nz, py, s->ny, s->stream);
  if (e == cudaSuccess) e = x_inverse(s->d_hbuf, s->d_vh, p[0], s->nx, s->ny, s->nz, py, scale, s->stream);
  s->launches += 5;
  if (e != cudaSuccess) return fail(TDKS_EDEVICE, std::string("Hartree: ") + cudaGetErrorString(e));
  return TDKS_OK;
}

}  // namespace tdks_host
