// Internal declarations of the GB300 TDKS library (not part of the C interface).
//
// Device layout of one system ("packed batches", the paper's Sec. "Memory layout": the
// state index is innermost so every thread of a warp runs the same stencil on
// neighbouring orbitals):
//
//   orbitals  [k][batch][z][y][x][j],  orbital o = batch * BS + j,  BS orbitals per batch
//   vectors   one thread owns one 16-byte vector: complex128 -> 1 orbital,
//             complex64 -> 2 orbitals; OVC = 4 vectors per (point, batch), i.e. 64 B.
//
// complex128 systems: BS = 4, the state and the Taylor terms are complex128.
// complex64  systems: BS = 8, the Taylor terms are complex64; the state (the running sum
//                     of the series) is a double-float pair hi + lo of two complex64
//                     arrays (~48-bit significand), updated with error-free FP32
//                     transformations, because GB300 runs FP64 at a small fraction of its
//                     FP32 rate; density, potentials and reductions are FP64.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

namespace tdks {

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per device for kernel k; `done`
// (one per kernel instantiation) records the devices already set, safely across host
// threads that drive systems at the same time.
template <typename K>
inline cudaError_t ensure_smem_attr(K k, size_t smem, std::atomic<unsigned> &done) {
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned bit = dev < 32 ? 1u << dev : 0u;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

// Launch with thread-block clusters of `cluster` CTAs along x.  (An error is returned and, as by a
// cudaGetLastError() after a launch, no longer pending.)
template <typename... Par, typename... Arg>
inline cudaError_t launch_cluster(void (*k)(Par...), dim3 grid, dim3 block, cudaStream_t s, int cluster, Arg &&...arg) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k, std::forward<Arg>(arg)...);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

constexpr int OVC = 4;        // 16-byte vectors per (point, batch)
constexpr int MAXM = 4;       // largest FD half-width (8th order)

enum Mode { MODE_FIRST = 0, MODE_MID = 1, MODE_LAST = 2 };
// Compute precisions of the sweeps.  P_C64S is complex64 storage computed with one complex
// value per thread vector (8 bytes, 8 vectors per (point, batch)) instead of two (16 bytes,
// 4 vectors): the tile shapes that use it keep more points per thread in registers.
enum Prec { P_C128 = 0, P_C64 = 1, P_C64S = 2 };

// Per-entry projector data (one grid point of one atom's sphere).
struct ProjEntry {
  int cell;        // flat grid index of the (wrapped) point
  int atom;
  float beta[4];   // beta_aj at the point (c64 path)
  double betad[4]; // same, double (c128 path)
  double T[3];     // lattice translation of the unwrapped point
  double d[3];     // unwrapped point minus atom centre
};

// One point of one face of the t-SURFF surface: its flat grid index, the face's normal
// axis, its grid indices, and the trapezoid weight times the sign of the outward normal.
struct TsEntry {
  long cell;
  int ax;
  int i[3];
  double ws;
};

// Per-point record read by the sweeps (16 bytes): the diagonal of H, V_eff + w0 with w0 the stencil's
// centre weight, summed in the compute precision (double for complex128 systems; float in the first 4
// bytes for complex64 systems; formed once per point here, not once per value in the sweeps), and the point's
// range [r0, r1) in the point-major projector entry list.
struct __align__(16) PointAux {
  double veff;
  int r0, r1;
};

struct SweepParams {
  int nx, ny, nz;
  int n_tx, n_ty, n_zc, zc;   // x/y tiles and z chunks
  int n_kb, n_batches;        // kb = k * n_batches + batch
  long n_items;
  // stencil: H = w0 c + sum_m w[m] (sum of the 6 neighbours at distance m) + ...
  double w[MAXM + 1];         // w[0] = -3 c_0 / (2 h^2), w[m] = -c_m / (2 h^2)
  double gw[MAXM + 1];        // gradient weights d_m / h
  double coef;                // out = coef H in, or i coef H in (coef_im)
  int coef_im;
  float wf[MAXM + 1];         // w rounded to FP32 (complex64 sweeps)
  float coeff;                // coef rounded to FP32
  const void *in;             // stencil input (psi storage in MODE_FIRST, term storage else)
  void *out;                  // term output (MODE_FIRST / MODE_MID)
  void *psi;                  // MODE_LAST: state (complex128, or the hi part of a complex64
                              // system's double-float state), read and written in place
  void *psi_lo;               // MODE_LAST, complex64 systems: lo part of the state
  const void *t1, *t2;        // MODE_LAST: earlier terms
  const PointAux *aux;        // [N] V_eff and projector entry ranges
  // projectors
  int has_proj;               // the system has projector entries
  const void *nl;             // [kb][n_ent + 1][OVC] vectors: sum_aj beta_aj(r) phase q_aj at the
                              // sphere point whose entries start at r0; row n_ent is zero
  int n_ent;                  // projector entries
  // Bloch boundary
  int bloch;                  // periodic cell: values across a face carry exp(i k.L) per wrap
  const double *kvec;         // [n_k][3]
  const double2 *kphase;      // [n_k][3] e^{i k_a L_a} in the compute precision
  double L[3];
  double A[3];                // vector potential (velocity gauge)
  int grad_mask;              // bit a: add -i A_a grad_a; bit 3: observables need all grads
  // reductions
  int do_obs;
  double *obs_part;           // [n_items][4]: <psi|H psi> weighted, current x,y,z
  const double *wocc;         // [n_k] k-weight times occupation
  double *dens_part;          // [n_kb][N] (MODE_LAST): w_k f sum |psi|^2 (complex128); for
                              // complex64, the unweighted sum as a (float hi, float lo) pair
  int *err;                   // device error word (bounded waits that ran out set it)
  int withhold;               // failure injection (tests): the producer makes no claim and no
                              // copy, so every other warp's first wait runs out
  unsigned int *work;         // work-item counter of the warp-specialised TMA sweep (zero
                              // between launches: the launch's last claim resets it)
};

// Sets the coefficient cr + i ci, one of which is zero (H itself, or -i tau/k of a Taylor term), with
// its FP32 copy.
inline void set_coef(SweepParams &p, double cr, double ci) {
  p.coef_im = cr == 0.0;
  p.coef = p.coef_im ? ci : cr;
  p.coeff = (float)p.coef;
}

struct GatherParams {
  int n_kb, n_batches, n_atoms;
  long N;
  const void *in;             // stencil input (state or hi part of the state, or a term)
  const int *atom_begin;      // [n_atoms+1] entry ranges (atom-major)
  const ProjEntry *ent;
  const float4 *ent_beta;     // [n_ent] beta_aj of each entry in FP32 (complex64 kernels)
  const int2 *ent_ca;         // [n_ent] (cell, atom) of each entry
  const double *D;            // [n_atoms][4]
  double h3;
  double A[3];
  void *q;                    // [kb][atom][4][OVC] vectors
  int n_chunks;               // CTAs per (atom, kb): each sums a contiguous share of the sphere
  double2 *qpart;             // [kb][atom][chunk][4][OVC][2] partial sums (FP64)
  // scatter side: the non-local term at every sphere point
  const int2 *sp;             // [n_sp] entry range [r0, r1) of each point inside a sphere
  int n_sp;
  const int *rowent;          // entry indices, point-major
  int n_ent;
  void *nl;                   // [kb][n_ent + 1][OVC] vectors, row r0 of each sphere point
  const void *phase;          // [k][n_ent] (cos, sin) of k.T + A.d as float2 or double2; null: no phases
};

// The projectors' share of a periodic cell's current (record time): partial records
// out[(kb * n_atoms + a) * BS + o][4] for every atom, k-batch and orbital of the batch.
struct NlCurrentParams {
  int prec, BS, n_batches, n_kb, n_atoms;
  long N;
  const void *psi, *psi_lo;   // the state (complex64: hi and lo parts)
  const int *atom_begin;      // [n_atoms + 1] entry ranges
  const ProjEntry *ent;
  const double *D;            // [n_atoms][4]
  const void *phase;          // [k][n_ent] entry phases (GatherParams)
  int n_ent;
  const double *wocc;         // [n_k] k-weight times occupation
  double h3;
  int n_chunks;               // CTAs per (atom, kb), set by the launcher
  double *out;
};
cudaError_t launch_nl_current(const NlCurrentParams &p, cudaStream_t s);

// Per-system data of a batch (device copies), for the batched LDA and finalise kernels.
struct BatchAux {
  long N;
  int nx, ny, nz, n_kb, n_batches, xc;
  double h, occ, w0;
  const double *wocc;       // [n_k] k-weight times occupation
  int gauge, envelope;
  double pol[3], amp, omega, t_total;
  const double *dens_part;
  const double *vloc;
  PointAux *aux;
  double *lda_part;
  int n_lda;
  double *obs_part;
  long n_items;
  double *ring;
  long long ring_len;
};

// Device clock of a batched system: state time t of the current step, step length dt,
// sub-steps per step, current sub-step j, steps completed.
struct BatchClock {
  double t, dt;
  long long step;
  int substeps, j;
};

// Tensor maps of one TMA sweep launch: the stencil input with halo (z depth = planes per
// copy), the stencil input as tiles without halo (same depth), the per-point records (tile
// box, same depth) and, for the last Taylor term, the four own-point operands state hi,
// state lo, t1, t2 (tile boxes, depth 1).
struct SweepMaps {
  CUtensorMap in, ctr, aux, op[4];
  CUtensorMap sx, sy;  // periodic cells: the input as M x (TY + 2M) and TX x M strip boxes
};

// Batched stencil sweep over many systems (tdks_sweep_tma.cu): params[s] and
// maps[4*s + which] of system s; item_begin[s] = first work item of system s.
struct BatchSweepArgs {
  const SweepParams *params;
  const SweepMaps *maps;  // 4 per system (one per Taylor term)
  int which;
  const long *item_begin;
  int n_sys;
  long total_items;
  unsigned int *work;     // work-item counter (zero between launches)
  const int *item_sys;    // the system of every work item
};


// Launchers (tdks_sweep.cu)
cudaError_t launch_sweep(int M, int prec, int mode, int bloch, int tx, int ty,
                         const SweepParams &p, int grid, cudaStream_t s);
int sweep_threads(int tx, int ty);
size_t sweep_smem(int M, int tx, int ty);

// Launchers (tdks_aux.cu).  The projector step of a system alone is two kernels: the gather-dot (a cluster per
// unit) and the non-local term at every sphere point (skipped when no point is in a sphere); a batch's gather
// has a second stage as a launch of its own.
constexpr int NL_THREADS = 256;
cudaError_t launch_gather(int prec, int bloch, const GatherParams &p, cudaStream_t s);
// out[3 k + a] = e^{i k_a L_a} from FP32 functions (complex64 sweeps)
cudaError_t launch_face_phase(int n_k, const double *kvec, const double L[3], double2 *out, cudaStream_t s);
// out[k * n_ent + e] = (cos, sin) of A.d_e (+ k.T_e in a periodic cell): float2 (complex64) or double2
cudaError_t launch_phase_table(int prec, const ProjEntry *ent, int n_ent, int n_k, const double *kvec,
                               const double A[3], int bloch, void *out, cudaStream_t s);
// chunks per (atom, k-batch) that fill the GPU for n_atoms * n_kb units; those of a system alone
int gather_chunks(long units);
int gather_chunks_alone(int prec, long units);
cudaError_t launch_density(int prec, long N, int n_kb, int n_batches, const void *psi, const void *psi_lo,
                           const double *wocc, double *dens_part, cudaStream_t s);
cudaError_t launch_lda(int prec, int bloch, long N, int nx, int ny, int nz, double h,
                       int n_kb, int n_batches, const double *wocc, const double *dens_part,
                       const double *vloc, int xc,
                       const double E[3], double half_A2, double w0, PointAux *aux, double *lda_part,
                       int n_blocks, cudaStream_t s, const double *n_in = nullptr, const double *vh = nullptr,
                       int sums = 1);
// Classical Runge-Kutta stage update over n complex128 values (complex128 systems):
//   stage = psi + a k,  acc = (init ? 0 : acc) + b k,
// and the last stage's psi <- psi + acc + b k (rk4_finish).
cudaError_t launch_rk4_stage(long n, const void *psi, const void *k, double a, void *stage, void *acc, double b,
                             int init, cudaStream_t s);
cudaError_t launch_rk4_finish(long n, void *psi, const void *acc, const void *k, double b, cudaStream_t s);
// n_out[r] = sum over this system's states of w_k f |psi_ik(r)|^2 (FP64), from dens_part
cudaError_t launch_density_sum(int prec, long N, int n_kb, int n_batches, const double *wocc,
                               const double *dens_part, double *n_out, cudaStream_t s);
// CFM4 exchange history: v[j] is v_x at the start of the j-th latest sub-step (v[0] the
// newest), w[j] its weight in an exponential's effective potential, nh the points in use.
struct CfmHist {
  double *v[4];
  double w[4];
  int nh;
};
cudaError_t launch_cfm_veff(int prec, int bloch, long N, int nx, int ny, int nz, double h, int n_kb, int n_batches,
                            const double *wocc, const double *dens_part, const double *vloc, int xc, int push,
                            const CfmHist &hist, const double E[3], double w0, PointAux *aux, cudaStream_t s,
                            const double *vh = nullptr, const double *n_in = nullptr);
cudaError_t launch_finalize(const double *obs_part, long n_items, const double *lda_part,
                            int n_lda_blocks, double *record, double t_state, double h3,
                            double occ, int bloch, double omega_cell, const double A[3],
                            double field_val, cudaStream_t s);
// The same record in two parts, for state-parallel runs: the 10 sums into sums[0..9]
// (sums[0..3]: this rank's band energy and current; sums[4..9]: from the summed density),
// then, once the caller has summed sums[0..3] over the ranks, the record from sums.
cudaError_t launch_finalize_sums(const double *obs_part, long n_items, const double *lda_part, int n_lda_blocks,
                                 double *sums, cudaStream_t s);
cudaError_t launch_record_from_sums(const double *sums, double *record, double t_state, double h3, double occ,
                                    int bloch, double omega_cell, const double A[3], double field_val,
                                    cudaStream_t s);
// host layout -> internal layout and density partials, points [pt0, pt0 + npts) of k-point k
cudaError_t launch_pack_in(int prec, long N, int k, long pt0, long npts, int n_orb, int n_batches,
                           const double *plain, void *internal, void *internal_lo, const double *wocc,
                           double *dens_part, cudaStream_t s);
cudaError_t launch_unpack(int prec, long N, long g0, long npts, int n_orb, int n_batches, const void *internal,
                          const void *internal_lo, double *plain, cudaStream_t s);

// TMA sweep (tdks_sweep_tma.cu).  maps.in: 8-byte words, dims {8 nx, ny, nz, n_kb}, box {8 (TX + 2M), TY + 2M,
// tma_planes(prec, mode), 1} (TX, TY: the shape's tile); maps.aux: dims {2 nx, ny, nz}, box {2 TX, TY,
// tma_planes}; maps.op[i]: dims as maps.in, box {8 TX, TY, 1, 1}; maps.ctr: as maps.op with tma_planes planes.
// (A tile row is one run of the innermost dimension: with a dimension of its own per point the copies moved 64
// bytes at a time, last term of the medium molecule 653 -> 620 us.)  Default: the warp-specialised kernel;
// lockstep: the variant in which all warps of a CTA advance plane by plane together.
cudaError_t launch_sweep_tma(int M, int prec, int mode, int tx, int ty, const SweepMaps &maps,
                             const SweepParams &p, int grid, cudaStream_t s, bool lockstep = false,
                             int shape = 0);
// Tile shapes of the warp-specialised sweep: shape s covers tx x ty points of one orbital
// block with `warps` consumer warps, each thread computing `rows` points of a 16-byte vector.
// Null outputs are skipped; false for a shape out of range.
constexpr int WS_SHAPES = 9;
bool ws_shape_info(int shape, int *tx, int *ty, int *rows, int *warps);
// The shape whose kernel a sweep of `shape` runs: some shapes exist for some systems only, the others run one
// that does.  Tiles, tensor maps and record counts follow the result.
// last: the sweep of the last Taylor term.
int ws_kernel_shape(int shape, int M, int prec, int bloch, int nx, int ny, bool last);
// The shape a sweep takes until one is set or tuned.  complex64, terms 1 to 3: shape 6 once the grid has
// work for its larger tile (medium molecule 0.316 -> 0.250 ms, 48^3 with 16 orbitals 18.4 -> 17.2 us; at
// 24^3 shape 0 is still ahead, 9.6 against 10.4 us, and in cells up to 32^3); last term: shape 3 while the
// sweep is short (64^3, 24 orbitals 96 -> 82 us), shape 2 for long ones (medium molecule 0.54 -> 0.48 ms).
// complex128 is bound by the FP64 pipe in every shape (96^3, 16 orbitals 1.513 ms with shape 0, 1.531 with 2) and
// takes the tile that leaves fewer of its points outside the grid (cell of 30 x 36 x 32, 3 k-points, 10 orbitals:
// 16 x 12 has 6% and 16 x 8 18% outside, 0.175 against 0.193 ms); short sweeps keep the smaller one.  Of both
// orders: in cells of order 8 shape 2's kernels spill beside four service warps and shape 0's do not, and it is
// still the faster one wherever this rule takes it (middle term, 8 orbitals, 2 k-points: 30 x 36 x 32 168 against
// 173 us, 64 x 36 x 40 376 against 430, 60^3 854 against 927; where both fit as well, 48^3, 430 against 437).
// A small complex64 cell also goes by the fit (first and middle term, 40^3 with 2 k-batches, 20% more of 16 x 12
// tiles outside: 20.8 and 18.4 us with shape 0, 23.0 and 19.2 with 6; 48^3 with 1: 16.6 and 14.5, 15.6 and 14.6;
// 36 x 30 x 32 with 2, 12.5% more outside: 18.7 and 16.3, 15.5 and 14.4).
inline int ws_default_shape(int prec, int bloch, int nx, int ny, long points, bool last) {
  const long wx = (nx + 15) / 16 * 16L, a0 = wx * ((ny + 7) / 8 * 8), a2 = wx * ((ny + 11) / 12 * 12);
  if (prec != P_C64) return points >= 60000 && 51 * a2 < 50 * a0 ? 2 : 0;
  if (last) return points < 1500000 ? 3 : 2;
  if (bloch && points < 150000 && 20 * a2 > 23 * a0) return 0;
  return points >= (bloch ? 60000 : 30000) ? 6 : 0;
}
// planes a shape's kernel takes per iteration
int ws_shape_planes(int shape, int M, int bloch);
bool tma_supported(int M, int tx, int ty);
int tma_planes(int prec, int mode, bool lockstep = false);
int lda_blocks(long N);
cudaError_t launch_sweep_tma_batch(int M, int prec, int mode, const BatchSweepArgs &a, cudaStream_t s,
                                   int shape = 0);
// begin: prefix sums of n_atoms * n_kb * n_chunks (stage 1 CTAs); ubegin: of n_atoms * n_kb;
// nbegin: of the non-local kernel's CTAs (nl_batch_blocks).  gsys, usys,
// nsys: the system of each stage-1 CTA, unit and non-local CTA (one table load instead of a
// binary search over the prefix sums in every CTA).
cudaError_t launch_gather_batch(int prec, const GatherParams *gp, const long *begin, const long *ubegin,
                                const long *nbegin, const int *gsys, const int *usys, const int *nsys,
                                long total, long total_units, long total_nl, cudaStream_t s);
// CTAs of one system in a batch's non-local kernel: each covers NL_BATCH_RUNS runs of NL_THREADS (sphere
// point, vector) pairs, so that its setup is paid once per several runs
constexpr int NL_BATCH_RUNS = 2;
inline long nl_batch_blocks(int n_sp) {
  return ((long)n_sp * OVC + NL_THREADS * NL_BATCH_RUNS - 1) / (NL_THREADS * NL_BATCH_RUNS);
}
cudaError_t launch_lda_batch(int prec, const BatchAux *aux, const BatchClock *clk, const long *begin, int n_sys,
                             long total, cudaStream_t s);
// which = 0: observable records (first sub-step of a step); 1: advance the clocks
cudaError_t launch_batch_tail(const BatchAux *aux, BatchClock *clk, int n_sys, int which, cudaStream_t s);

}  // namespace tdks
