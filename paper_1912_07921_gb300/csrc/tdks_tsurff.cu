// t-SURFF photoelectron amplitudes (Sec. "t-SURFF"): the amplitude of orbital i on the
// Volkov state of momentum p is the time integral of the current of chi_p and phi_i through
// a surface S between the inner region and the outer one,
//   b_i(p, T) = int_0^T dt oint_S ds n . <chi_p| j |phi_i>,
//   <chi_p| j |phi> = 1/2 chi_p^* (k_p phi - i grad_h phi)   (length gauge),
//   chi_p(r, t) = (2 pi)^(-3/2) exp(i k_p(t).r - i Phi_p(t)),  k_p = p + a(t),  a = -int E,
//   Phi_p = 1/2 (|p|^2 t + 2 p.alpha + beta),  alpha = int a,  beta = int |a|^2,
// with S the surface of a box of grid planes (each face by the two-dimensional trapezoid rule,
// outward normal), the gradient the central difference of order 2M, and the time integral
// the trapezoid rule over the configured steps.  The section notes that the method only
// needs the gradient on the surface points: per step a gather kernel forms, at every surface
// entry and orbital, w n.(phi, -i grad_h phi), and a flux kernel contracts them with the
// Volkov factors of every momentum (products of one factor per axis), the entries split over CTAs
// whose sums are added in order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "tdks_system.h"

using namespace tdks;
using namespace tdks_host;

namespace {

struct TsGather {
  int prec, BS, n_orb, ax_unused;
  long N;
  long stride[3];          // point strides along x, y, z
  const void *psi, *psi_lo;
  const TsEntry *ent;
  int n_e, M;
  double d[MAXM + 1];      // gradient weights over h
  double2 *G0, *G1;        // [n_e][n_orb]
};

// value of orbital o at point pt, in FP64 (complex64 systems: hi + lo of the state)
__device__ __forceinline__ double2 ts_value(const TsGather &g, int o, long pt) {
  const long i = ((long)(o / g.BS) * g.N + pt) * g.BS + (o % g.BS);
  if (g.prec == P_C128) return reinterpret_cast<const double2 *>(g.psi)[i];
  const float2 hi = reinterpret_cast<const float2 *>(g.psi)[i], lo = reinterpret_cast<const float2 *>(g.psi_lo)[i];
  return make_double2((double)hi.x + (double)lo.x, (double)hi.y + (double)lo.y);
}

__global__ void tsurff_gather_kernel(const TsGather g) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= (long)g.n_e * g.n_orb) return;
  const int e = (int)(t / g.n_orb), o = (int)(t % g.n_orb);
  const TsEntry en = g.ent[e];
  const long st = g.stride[en.ax];
  const double2 phi = ts_value(g, o, en.cell);
  double gx = 0.0, gy = 0.0;
  for (int m = 1; m <= g.M; m++) {
    const double2 a = ts_value(g, o, en.cell + m * st), b = ts_value(g, o, en.cell - m * st);
    gx += g.d[m] * (a.x - b.x);
    gy += g.d[m] * (a.y - b.y);
  }
  // w n (phi) and w n (-i grad phi); -i (gx + i gy) = gy - i gx
  g.G0[t] = make_double2(en.ws * phi.x, en.ws * phi.y);
  g.G1[t] = make_double2(en.ws * gy, -en.ws * gx);
}

// Volkov factors along each axis: E[p][i] = exp(-i k_p,a x_i) for the nx + ny + nz coordinates of a
// momentum's three axes, so that a surface point's factor is a product of three (a sine and cosine
// per momentum and point cost more than the contraction of a few orbitals).
__global__ void tsurff_factor_kernel(const double *p, double ax, double ay, double az, int n_p, int nx, int ny,
                                     int nz, double h, double2 *E) {
  const int nt = nx + ny + nz;
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= (long)n_p * nt) return;
  const int i = (int)(t % nt), pi = (int)(t / nt);
  const int a = i < nx ? 0 : (i < nx + ny ? 1 : 2);
  const int j = a == 0 ? i : (a == 1 ? i - nx : i - nx - ny), n = a == 0 ? nx : (a == 1 ? ny : nz);
  const double k = p[3 * pi + a] + (a == 0 ? ax : (a == 1 ? ay : az));
  double sn, cs;
  sincos(k * ((j - 0.5 * (n - 1)) * h), &sn, &cs);
  E[t] = make_double2(cs, -sn);
}

struct TsFlux {
  int n_e, n_orb, n_p, nt, off1, off2;  // nt = nx + ny + nz, off1 = nx, off2 = nx + ny
  int splits, tile;        // CTAs along the entries; entries per shared-memory tile
  const TsEntry *ent;
  const double2 *G0, *G1, *E;
  const double *p;         // [n_p][3]
  double a[3], alpha[3], beta, t_rel, weight;
  double2 *part;           // [splits][n_p][n_orb]
  double2 *b;              // [n_orb][n_p]
};

constexpr int TS_THREADS = 256;
constexpr int TS_WMAX = 1024;  // Volkov factors of one shared-memory tile (momenta of the CTA x entries)

// Contraction sum_e W_pe (k_p,ax G0_eo + G1_eo) of one split of the entries, one (momentum, orbital)
// pair per thread: 6 FP64 multiply-adds per entry and pair on GB300's 2-per-clock FP64 pipe, which
// bounds it, so every lane holds a pair (pairs are numbered through, orbital fastest) and the entries
// are split over enough CTAs to fill the GPU.  The tile's factors are formed once per CTA; G is read
// through L1 in runs of orbitals.  One CTA per momentum with a thread per orbital, as before, left
// 112 of 128 threads idle with 16 orbitals: 64^3 grid, 400 momenta, 6.3 ms per flux
// against 1.05; the multiply-adds alone take 0.85.
__global__ void __launch_bounds__(TS_THREADS) tsurff_flux_kernel(const TsFlux f) {
  __shared__ double2 sW[TS_WMAX];
  __shared__ int sAx[TS_WMAX];
  const long pairs = (long)f.n_p * f.n_orb, q0 = (long)blockIdx.x * TS_THREADS, q = q0 + threadIdx.x;
  const bool live = q < pairs;
  const int p0 = (int)(q0 / f.n_orb);
  const int np = (int)(min(pairs - 1, q0 + TS_THREADS - 1) / f.n_orb) - p0 + 1;  // momenta of this CTA
  const int pi = live ? (int)(q / f.n_orb) : p0, o = live ? (int)(q % f.n_orb) : 0, pl = pi - p0;
  const double k0 = f.p[3 * pi] + f.a[0], k1 = f.p[3 * pi + 1] + f.a[1], k2 = f.p[3 * pi + 2] + f.a[2];
  const int e_lo = (int)((long)f.n_e * blockIdx.y / f.splits), e_hi = (int)((long)f.n_e * (blockIdx.y + 1) / f.splits);
  double ar = 0.0, ai = 0.0;
  for (int e0 = e_lo; e0 < e_hi; e0 += f.tile) {
    const int ne = min(f.tile, e_hi - e0);
    __syncthreads();
    for (int t = threadIdx.x; t < ne * np; t += TS_THREADS) {
      const int j = t / np, m = t - j * np;
      const TsEntry &en = f.ent[e0 + j];
      const double2 *E = f.E + (long)(p0 + m) * f.nt;
      const double2 x = E[en.i[0]], y = E[f.off1 + en.i[1]], z = E[f.off2 + en.i[2]];
      const double2 xy = make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x);
      sW[t] = make_double2(xy.x * z.x - xy.y * z.y, xy.x * z.y + xy.y * z.x);
      if (m == 0) sAx[j] = en.ax;
    }
    __syncthreads();
    if (live) {
      const double2 *g0 = f.G0 + (long)e0 * f.n_orb + o, *g1 = f.G1 + (long)e0 * f.n_orb + o;
#pragma unroll 4
      for (int j = 0; j < ne; j++) {
        const double2 x = g0[(long)j * f.n_orb], y = g1[(long)j * f.n_orb], w = sW[j * np + pl];
        const int ax = sAx[j];
        const double k = ax == 0 ? k0 : (ax == 1 ? k1 : k2);
        const double tr = fma(k, x.x, y.x), ti = fma(k, x.y, y.y);
        ar = fma(w.x, tr, ar);  // (as written with + and -, a product and a sum more)
        ai = fma(w.x, ti, ai);
        ar = fma(-w.y, ti, ar);
        ai = fma(w.y, tr, ai);
      }
    }
  }
  if (live) f.part[(long)blockIdx.y * pairs + q] = make_double2(ar, ai);
}

// b += the splits' sums in order, times the time weight and the Volkov phase.
__global__ void __launch_bounds__(TS_THREADS) tsurff_add_kernel(const TsFlux f) {
  const long pairs = (long)f.n_p * f.n_orb, q = blockIdx.x * (long)TS_THREADS + threadIdx.x;
  if (q >= pairs) return;
  const int pi = (int)(q / f.n_orb), o = (int)(q % f.n_orb);
  double ar = 0.0, ai = 0.0;
  for (int s = 0; s < f.splits; s++) {
    const double2 v = f.part[(long)s * pairs + q];
    ar += v.x;
    ai += v.y;
  }
  const double px = f.p[3 * pi], py = f.p[3 * pi + 1], pz = f.p[3 * pi + 2];
  const double phase = 0.5 * ((px * px + py * py + pz * pz) * f.t_rel +
                              2.0 * (px * f.alpha[0] + py * f.alpha[1] + pz * f.alpha[2]) + f.beta);
  double sn, cs;
  sincos(phase, &sn, &cs);
  const double pref = 0.5 * f.weight * 0.063493635934240969;  // (2 pi)^(-3/2)
  double2 &bo = f.b[(long)o * f.n_p + pi];
  bo.x += pref * (cs * ar - sn * ai);
  bo.y += pref * (cs * ai + sn * ar);
}

// CTAs along the entries: with the pair tiles, four to an SM, in whole rounds.
int flux_splits(long pairs, int n_e) {
  const long tiles = (pairs + TS_THREADS - 1) / TS_THREADS;
  return (int)std::max(1L, std::min(std::min(64L, (long)n_e), 152L * 4 / tiles));
}

}  // namespace

namespace tdks_host {

void tsurff_free(tdks_system *s) {
  cudaFree(s->d_ts_p); cudaFree(s->d_ts_ent); cudaFree(s->d_ts_G); cudaFree(s->d_ts_b);
  cudaFree(s->d_ts_E); cudaFree(s->d_ts_part);
  s->d_ts_E = s->d_ts_part = nullptr;
  s->d_ts_p = nullptr; s->d_ts_ent = nullptr; s->d_ts_G = nullptr; s->d_ts_b = nullptr;
  s->ts_np = 0;
  s->ts_ne = 0;
}

// The flux of the current state with trapezoid weight `weight` (dt or dt/2) into b.
int tsurff_accumulate(tdks_system *s, double weight) {
  double c[MAXM + 1], d[MAXM + 1];
  fd_weights(s->M, c, d);
  TsGather g{};
  g.prec = s->prec; g.BS = s->BS; g.n_orb = s->n_orb; g.N = s->N;
  g.stride[0] = 1; g.stride[1] = s->nx; g.stride[2] = (long)s->nx * s->ny;
  g.psi = s->psi; g.psi_lo = s->psi_lo; g.ent = s->d_ts_ent; g.n_e = s->ts_ne; g.M = s->M;
  for (int m = 0; m <= MAXM; m++) g.d[m] = m <= s->M ? d[m] / s->h : 0.0;
  g.G0 = s->d_ts_G;
  g.G1 = s->d_ts_G + (size_t)s->ts_ne * s->n_orb;
  const long n = (long)s->ts_ne * s->n_orb;
  tsurff_gather_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(g);
  TsFlux f{};
  f.n_e = s->ts_ne; f.n_orb = s->n_orb; f.n_p = s->ts_np; f.ent = s->d_ts_ent;
  f.G0 = g.G0; f.G1 = g.G1; f.p = s->d_ts_p;
  for (int x = 0; x < 3; x++) { f.a[x] = s->ts_vol[x]; f.alpha[x] = s->ts_vol[3 + x]; }
  f.beta = s->ts_vol[6];
  f.t_rel = s->ts_trel;
  f.weight = weight;
  f.b = s->d_ts_b;
  f.E = s->d_ts_E; f.part = s->d_ts_part;
  f.nt = s->nx + s->ny + s->nz; f.off1 = s->nx; f.off2 = s->nx + s->ny;
  const long pairs = (long)s->ts_np * s->n_orb;
  f.splits = flux_splits(pairs, s->ts_ne);
  // (a CTA's 256 pairs belong to at most 255 / n_orb + 2 momenta, and to no more than there are)
  f.tile = TS_WMAX / std::min(s->ts_np, (TS_THREADS - 1) / s->n_orb + 2);
  const long nf = (long)s->ts_np * f.nt;
  const unsigned tiles = (unsigned)((pairs + TS_THREADS - 1) / TS_THREADS);
  tsurff_factor_kernel<<<(unsigned)((nf + 127) / 128), 128, 0, s->stream>>>(s->d_ts_p, f.a[0], f.a[1], f.a[2], s->ts_np,
                                                                           s->nx, s->ny, s->nz, s->h, s->d_ts_E);
  tsurff_flux_kernel<<<dim3(tiles, f.splits), TS_THREADS, 0, s->stream>>>(f);
  tsurff_add_kernel<<<tiles, TS_THREADS, 0, s->stream>>>(f);
  s->launches += 4;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(TDKS_EDEVICE, std::string("t-SURFF flux: ") + cudaGetErrorString(e));
  return TDKS_OK;
}

// a, alpha, beta from t to t + dt: the classical Runge-Kutta method on a' = -E (length
// gauge; zero otherwise), alpha' = a, beta' = |a|^2.
void tsurff_advance(tdks_system *s, double t, double dt) {
  auto rhs = [&](double tt, const double *y, double *f) {
    double E[3], A[3];
    field_at(s, tt, E, A);
    for (int x = 0; x < 3; x++) {
      f[x] = s->gauge == TDKS_GAUGE_LENGTH ? -E[x] : 0.0;
      f[3 + x] = y[x];
    }
    f[6] = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
  };
  double *y = s->ts_vol, k1[7], k2[7], k3[7], k4[7], tmp[7];
  rhs(t, y, k1);
  for (int i = 0; i < 7; i++) tmp[i] = y[i] + 0.5 * dt * k1[i];
  rhs(t + 0.5 * dt, tmp, k2);
  for (int i = 0; i < 7; i++) tmp[i] = y[i] + 0.5 * dt * k2[i];
  rhs(t + 0.5 * dt, tmp, k3);
  for (int i = 0; i < 7; i++) tmp[i] = y[i] + dt * k3[i];
  rhs(t + dt, tmp, k4);
  for (int i = 0; i < 7; i++) y[i] += dt / 6.0 * (k1[i] + 2.0 * k2[i] + 2.0 * k3[i] + k4[i]);
  s->ts_trel += dt;
}

}  // namespace tdks_host

extern "C" int tdks_set_tsurff(tdks_sys s, const int *box, int n_p, const double *p) {
  if (!s) return fail(TDKS_EINVAL, "NULL system");
  if (n_p < 0) return fail(TDKS_EINVAL, "n_p < 0");
  CU(cudaStreamSynchronize(s->stream));
  tsurff_free(s);
  if (n_p == 0) return TDKS_OK;
  if (!box || !p) return fail(TDKS_EINVAL, "NULL argument");
  if (s->bc != TDKS_BC_ZERO || s->n_k != 1) return fail(TDKS_EINVAL, "t-SURFF needs a finite box with one k-point");
  const int n[3] = {s->nx, s->ny, s->nz};
  for (int a = 0; a < 3; a++)
    if (box[2 * a] < s->M || box[2 * a] >= box[2 * a + 1] || box[2 * a + 1] > n[a] - 1 - s->M)
      return fail(TDKS_EINVAL, "t-SURFF box planes must satisfy M <= lo < hi <= n - 1 - M on every axis");
  for (int i = 0; i < 3 * n_p; i++)
    if (!std::isfinite(p[i])) return fail(TDKS_EINVAL, "momenta must be finite");
  // surface entries: every grid point of each face (trapezoid weight h^2, halved on the face's
  // edges) with the face's outward normal; points on edges and corners belong to each face
  std::vector<TsEntry> ent;
  for (int face = 0; face < 6; face++) {
    const int ax = face / 2, ua = (ax + 1) % 3, va = (ax + 2) % 3;
    const double sgn = (face % 2) ? 1.0 : -1.0;
    for (int u = box[2 * ua]; u <= box[2 * ua + 1]; u++)
      for (int v = box[2 * va]; v <= box[2 * va + 1]; v++) {
        int ii[3];
        ii[ax] = box[2 * ax + (face % 2)];
        ii[ua] = u;
        ii[va] = v;
        double w = s->h * s->h;
        if (u == box[2 * ua] || u == box[2 * ua + 1]) w *= 0.5;
        if (v == box[2 * va] || v == box[2 * va + 1]) w *= 0.5;
        TsEntry e{};
        e.cell = ((long)ii[2] * s->ny + ii[1]) * s->nx + ii[0];
        e.ax = ax;
        e.ws = sgn * w;
        for (int q = 0; q < 3; q++) e.i[q] = ii[q];
        ent.push_back(e);
      }
  }
  s->ts_ne = (int)ent.size();
  CU(cudaMalloc((void **)&s->d_ts_ent, ent.size() * sizeof(TsEntry)));
  CU(to_device(s->d_ts_ent, ent.data(), ent.size() * sizeof(TsEntry), s->stream));
  CU(cudaMalloc((void **)&s->d_ts_p, (size_t)n_p * 3 * sizeof(double)));
  CU(to_device(s->d_ts_p, p, (size_t)n_p * 3 * sizeof(double), s->stream));
  CU(cudaMalloc((void **)&s->d_ts_G, 2 * ent.size() * (size_t)s->n_orb * sizeof(double2)));
  CU(cudaMalloc((void **)&s->d_ts_b, (size_t)s->n_orb * n_p * sizeof(double2)));
  CU(cudaMemsetAsync(s->d_ts_b, 0, (size_t)s->n_orb * n_p * sizeof(double2), s->stream));
  const long pairs = (long)s->n_orb * n_p;
  CU(cudaMalloc((void **)&s->d_ts_E, (size_t)n_p * (s->nx + s->ny + s->nz) * sizeof(double2)));
  CU(cudaMalloc((void **)&s->d_ts_part, (size_t)flux_splits(pairs, s->ts_ne) * pairs * sizeof(double2)));
  s->ts_np = n_p;
  for (int i = 0; i < 7; i++) s->ts_vol[i] = 0.0;
  s->ts_trel = 0.0;
  s->ts_started = false;
  return TDKS_OK;
}

extern "C" int tdks_get_tsurff(tdks_sys s, double *b, double *t_rel) {
  if (!s) return fail(TDKS_EINVAL, "NULL system");
  if (s->ts_np == 0) return fail(TDKS_ESTATE, "t-SURFF is not set");
  CU(cudaStreamSynchronize(s->stream));
  if (int rc = check_err(s)) return rc;
  if (b) CU(cudaMemcpy(b, s->d_ts_b, (size_t)s->n_orb * s->ts_np * sizeof(double2), cudaMemcpyDeviceToHost));
  if (t_rel) *t_rel = s->ts_trel;
  return TDKS_OK;
}
