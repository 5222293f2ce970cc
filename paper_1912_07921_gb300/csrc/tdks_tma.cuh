// Shared pieces of the TMA-fed stencil sweeps: mbarrier and bulk-tensor-copy wrappers,
// the ring geometry, work sources (one system or a batch), the producer's load cursors
// and the warp-specialised sweep body, whose tile shape (rows of 16 points, points per
// consumer thread, consumer warps) is a template parameter so that each shape can be
// compiled in a translation unit of its own.
#pragma once
#include <cuda.h>

#include <type_traits>

#include "tdks_internal.cuh"
#include "tdks_sweep_common.cuh"

namespace tdks {

namespace {

constexpr long long WAIT_LIMIT_CYCLES = 4000000000LL;  // ~2 s at 2 GHz
constexpr long long DRAIN_LIMIT_CYCLES = 200000000LL;  // ~0.1 s per copy on the error path

__device__ __forceinline__ uint32_t smem_u32(const void *ptr) {
  return (uint32_t)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  long long limit = WAIT_LIMIT_CYCLES) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 16-byte asynchronous global -> shared copy (L2 only), and an arrive on an mbarrier that
// fires once every cp.async this thread has issued so far has landed (the barrier's pending
// count is raised by one at issue, so its expected count stays as initialised).
__device__ __forceinline__ void cp_async_16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
  asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Consumer wait: bounded, and gives up at once when another warp has given up.  (Reading
// the abort flag only every 16 polls, or taking the bound from shared memory, measured 1-3%
// slower sweeps: the flag's load paces the polling.)
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t *bar, uint32_t parity, const volatile int *abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > WAIT_LIMIT_CYCLES) return false;
  }
  return true;
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *tmap, uint64_t *bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *tmap, uint64_t *bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap *tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}

// Before a thread's first use of a tensor map in global memory (not needed for maps in kernel parameters): maps
// are read through a proxy of their own, which may still hold what an earlier table had at the address.
__device__ __forceinline__ void tma_acquire_map(const CUtensorMap *tmap) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(tmap))
               : "memory");
}

}  // namespace

// Compile-time loop: f(integral_constant<int, 0>) ... f(integral_constant<int, N-1>).
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// Position in a ring of S slots: slot index and the parity of the slot's current use.
struct RingPos {
  int slot = 0;
  uint32_t phase = 0;
  template <int S>
  __device__ __forceinline__ void next() {
    if (++slot == S) {
      slot = 0;
      phase ^= 1u;
    }
  }
};

// Shared-memory plan: three TMA-fed rings, each slot completed by one mbarrier.
//   centre ring (SC slots): U planes of the input tile (no halo), which feed the per-thread
//     register z-queue; a slot is free again as soon as its planes are in registers;
//   halo ring (SH slots): U output planes of the input with their x/y halo, followed by the
//     U planes' per-point records; read when those planes are computed;
//   operand ring (SO slots, last Taylor term only): the four own-point operand tiles of one
//     output plane (state hi, state lo, t1, t2).
// Keeping the z history in registers (not in the ring) lets every ring run several slots
// ahead of the plane being computed.
//   periodic cells (BL): each halo slot also holds the four periodic-image strips a boundary
//     tile needs (the M columns beyond each x face over the slot's SY rows, the M rows beyond
//     each y face over the tile's TX columns), loaded by TMA from the opposite faces, and (first
//     Taylor term) the non-local rows of the plane's sphere points (one per point, in tile
//     order), which the patcher warp copies in with cp.async so that no consumer waits on a
//     global load.
template <int M, int TX, int TY, int U, bool OPS, bool BL = false, bool NLG = false>
struct TmaGeom {
  static constexpr int SX = TX + 2 * M, SY = TY + 2 * M;
  static constexpr int PLANE = SX * SY * OVC;                        // vectors per halo plane
  static constexpr int CPLANE = TX * TY * OVC;                       // vectors per centre plane
  static constexpr uint32_t CSLOT_BYTES = (uint32_t)CPLANE * 16 * U;
  static constexpr uint32_t IN_BYTES = (uint32_t)PLANE * 16 * U;
  static constexpr uint32_t AUX_BYTES = (uint32_t)TX * TY * 16 * U;
  static constexpr uint32_t STRIPX_BYTES = (uint32_t)M * SY * OVC * 16;   // beyond x = 0 or x = nx - 1
  static constexpr uint32_t STRIPY_BYTES = (uint32_t)TX * M * OVC * 16;   // beyond y = 0 or y = ny - 1
  static constexpr uint32_t STRIP1_BYTES = BL ? 2 * (STRIPX_BYTES + STRIPY_BYTES) : 0;  // of one plane
  static constexpr uint32_t STRIP_BYTES = STRIP1_BYTES * U;
  static constexpr uint32_t OPT_BYTES = (uint32_t)CPLANE * 16;       // one operand tile
  static constexpr uint32_t OP_BYTES = 4 * OPT_BYTES;
  static constexpr int SO = OPS ? 2 : 0;
  // (the last term's 4 operand tiles leave taller tiles room for few centre slots)
  static constexpr int SC = U == 1 ? (OPS ? (TX * TY > 128 ? 2 : 4) : (TX * TY > 256 ? 3 : 6)) : (OVC * TX * TY > 512 ? 3 : 4);
  static constexpr size_t BUDGET = 227 * 1024 - 2048;                // dynamic smem available
  static constexpr size_t HALO_ROOM = BUDGET - 128 - (size_t)SO * OP_BYTES - (size_t)SC * CSLOT_BYTES;
  // periodic cells, first Taylor term (NLG): the non-local rows of the plane's sphere points,
  // gathered into the slot by the patcher warp, where two slots still fit (else the consumers
  // load them).  (The larger slot leaves fewer halo slots: the faster middle and last sweeps
  // measured slower with it, the first sweep, with its current gradients, faster.)
  static constexpr uint32_t NL_STAGE = (uint32_t)TX * TY * OVC * 16 * U;
  static constexpr bool NLS = BL && NLG && HALO_ROOM / (IN_BYTES + AUX_BYTES + STRIP_BYTES + NL_STAGE) >= 2;
  static constexpr uint32_t NL_BYTES = NLS ? NL_STAGE : 0;
  static constexpr uint32_t HSLOT_BYTES = IN_BYTES + AUX_BYTES + STRIP_BYTES + NL_BYTES;
  static constexpr int SH_FIT = (int)(HALO_ROOM / HSLOT_BYTES);
  static constexpr int SH = SH_FIT < 8 ? SH_FIT : 8;
  static constexpr size_t SMEM = (size_t)SC * CSLOT_BYTES + (size_t)SH * HSLOT_BYTES + (size_t)SO * OP_BYTES + 128;
  static_assert(SH >= 2, "halo ring too small");
};

// Work sources: a single system (parameters and tensor maps are kernel parameters), or a
// batch of systems (per-system parameters and tensor maps in device arrays; a CTA stages
// the parameters of its current item in shared memory).
struct SingleSrc {
  const SweepParams *p;
  const SweepMaps *maps;
  __device__ __forceinline__ long n_items() const { return p->n_items; }
  __device__ __forceinline__ void item(long it, const SweepParams *&pp, const SweepMaps *&mp, long &local) const {
    pp = p;
    mp = maps;
    local = it;
  }
  __device__ __forceinline__ int sys_of(long) const { return 0; }
  __device__ __forceinline__ const SweepMaps *maps_of(int) const { return maps; }
  __device__ __forceinline__ int *err0() const { return p->err; }
  __device__ __forceinline__ bool withhold() const { return p->withhold != 0; }
};

// (the system of an item comes from a table: one load where a binary search over the systems'
// item ranges took a chain of them at the start of every item, in every warp)
struct BatchSrc {
  const BatchSweepArgs *a;
  __device__ __forceinline__ long n_items() const { return a->total_items; }
  __device__ __forceinline__ void item(long it, const SweepParams *&pp, const SweepMaps *&mp, long &local) const {
    const int s = a->item_sys[it];
    pp = a->params + s;
    mp = a->maps + 4 * s + a->which;
    local = it - a->item_begin[s];
  }
  __device__ __forceinline__ int sys_of(long it) const { return a->item_sys[it]; }
  __device__ __forceinline__ const SweepMaps *maps_of(int s) const { return a->maps + 4 * s + a->which; }
  __device__ __forceinline__ int *err0() const { return a->params[0].err; }
  __device__ __forceinline__ bool withhold() const { return a->params[0].withhold != 0; }
};

// Sequential cursor over one kind of load of the CTA's items (thread 0 only).  The item's
// geometry is decoded once, when the cursor enters the item, so issuing a load costs a few
// instructions: the other threads wait for thread 0 at the next barrier.
struct LoadCursor {
  long ii;     // item index among the CTA's items (-1: not entered yet)
  int l;       // load index within the item
  int n;       // loads of this kind in the item
  int tx, ty, kb, z0;
  int sys;     // system of the item (batch)
  long issued; // loads issued so far
  int nx, ny, nz, wrap;  // periodic cell: centre planes outside [0, nz) are loaded wrapped, and
                         // the halo slots of boundary tiles get their periodic-image strips
};

// floor(i / n) for possibly negative i
__device__ __forceinline__ int floordiv_i(int i, int n) { return i >= 0 ? i / n : -((-i - 1) / n) - 1; }

// Work item -> tile (tx, ty), orbital block kb and z chunk [z0, z1).
__device__ __forceinline__ void item_geom(const SweepParams &q, long it, int &tx, int &ty, int &kb, int &z0,
                                          int &z1) {
  // z chunks fastest: consecutive items are the chunks of one column, which run at about the
  // same time on different SMs and share the planes at their boundaries through L2
  z0 = (int)(it % q.n_zc) * q.zc;
  it /= q.n_zc;
  tx = (int)(it % q.n_tx);
  it /= q.n_tx;
  ty = (int)(it % q.n_ty);
  it /= q.n_ty;
  kb = (int)it;
  z1 = min(z0 + q.zc, q.nz);
}

// Loads per item: 0 = centre (queue planes z0-M .. z1+M-1, U per load), 1 = halo (output
// planes, U per load), 2 = operands (one per output plane).
template <int M, int U>
__device__ __forceinline__ int loads_of(int kind, int z0, int z1) {
  if (kind == 0) return (z1 - z0 + 2 * M + U - 1) / U;
  if (kind == 1) return (z1 - z0 + U - 1) / U;
  return z1 - z0;
}

// The producer side of the rings (one thread).  D: planes per copy (the z depth of the maps' boxes).
template <int M, int TX, int TY, int U, int D, class G, int SC, int SH, int SO, class Src>
struct Loader {
  Src src;
  long n_my;
  unsigned char *cbase, *hbase, *obase;
  uint64_t *cfull, *hfull, *ofull;

  // move the cursor onto its next load (decoding the geometry of an item it enters)
  __device__ __forceinline__ void advance(LoadCursor &c, int kind) const {
    while (c.ii < n_my && (c.ii < 0 || c.l >= c.n)) {
      c.ii += 1;
      c.l = 0;
      c.n = 0;
      if (c.ii < n_my) {
        const SweepParams *qp = nullptr;
        const SweepMaps *mq = nullptr;
        long local = 0;
        src.item(blockIdx.x + c.ii * gridDim.x, qp, mq, local);
        int z1 = 0;
        item_geom(*qp, local, c.tx, c.ty, c.kb, c.z0, z1);
        c.sys = src.sys_of(blockIdx.x + c.ii * gridDim.x);
        c.n = loads_of<M, U>(kind, c.z0, z1);
        c.nx = qp->nx;
        c.ny = qp->ny;
        c.nz = qp->nz;
        c.wrap = qp->bloch;
      }
    }
  }

  // issue the next load of `kind`; nothing past the CTA's last item
  __device__ __forceinline__ void issue(LoadCursor &c, int kind) const {
    advance(c, kind);
    if (c.ii >= n_my) return;
    emit(c, kind);
  }

  // issue the load the cursor is positioned on
  __device__ __forceinline__ void emit(LoadCursor &c, int kind) const {
    emit_at(c, kind, (int)(c.issued % (kind == 0 ? SC : (kind == 1 ? SH : SO))));
    c.issued++;
  }

  // the same into ring slot `slot`
  __device__ __forceinline__ void emit_at(LoadCursor &c, int kind, int slot) const {
    const SweepMaps *mp = src.maps_of(c.sys);
    if (kind == 0) {
      mbar_expect_tx(&cfull[slot], G::CSLOT_BYTES);
#pragma unroll
      for (int u = 0; u < U; u += D) {
        int zc = c.z0 - M + U * c.l + u;
        if (c.wrap) zc -= floordiv_i(zc, c.nz) * c.nz;  // (D = 1 for periodic cells)
        tma_load_4d(cbase + (size_t)slot * G::CSLOT_BYTES + (size_t)u * G::CPLANE * 16, &mp->ctr, &cfull[slot],
                    8 * c.tx * TX, c.ty * TY, zc, c.kb);
      }
    } else if (kind == 1) {
      unsigned char *dst = hbase + (size_t)slot * G::HSLOT_BYTES;
      const int x0 = c.tx * TX, y0 = c.ty * TY;
      // periodic cell: the strips this tile's halo crosses (the slot holds zeros there)
      const bool sl = G::STRIP_BYTES && c.wrap && x0 - M < 0, sr = G::STRIP_BYTES && c.wrap && x0 + TX + M > c.nx;
      const bool st = G::STRIP_BYTES && c.wrap && y0 - M < 0, sb = G::STRIP_BYTES && c.wrap && y0 + TY + M > c.ny;
      const uint32_t bytes = G::IN_BYTES + G::AUX_BYTES + (uint32_t)U * ((uint32_t)(sl + sr) * G::STRIPX_BYTES +
                                                                         (uint32_t)(st + sb) * G::STRIPY_BYTES);
      mbar_expect_tx(&hfull[slot], bytes);
#pragma unroll
      for (int u = 0; u < U; u += D) {
        const int zp = c.z0 + U * c.l + u;
        tma_load_4d(dst + (size_t)u * G::PLANE * 16, &mp->in, &hfull[slot], 8 * (x0 - M), y0 - M, zp, c.kb);
        tma_load_3d(dst + G::IN_BYTES + (size_t)u * TX * TY * 16, &mp->aux, &hfull[slot], 2 * x0, y0, zp);
        if constexpr (G::STRIP_BYTES > 0) {
          unsigned char *sd = dst + G::IN_BYTES + G::AUX_BYTES + (size_t)u * G::STRIP1_BYTES;
          if (sl) tma_load_4d(sd, &mp->sx, &hfull[slot], 8 * (c.nx - M), y0 - M, zp, c.kb);
          if (sr) tma_load_4d(sd + G::STRIPX_BYTES, &mp->sx, &hfull[slot], 0, y0 - M, zp, c.kb);
          if (st) tma_load_4d(sd + 2 * G::STRIPX_BYTES, &mp->sy, &hfull[slot], 8 * x0, c.ny - M, zp, c.kb);
          if (sb) tma_load_4d(sd + 2 * G::STRIPX_BYTES + G::STRIPY_BYTES, &mp->sy, &hfull[slot], 8 * x0, 0, zp, c.kb);
        }
      }
    } else {
      unsigned char *dst = obase + (size_t)slot * G::OP_BYTES;
      mbar_expect_tx(&ofull[slot], G::OP_BYTES);
      for (int j = 0; j < 4; j++)
        tma_load_4d(dst + j * G::OPT_BYTES, &mp->op[j], &ofull[slot], 8 * c.tx * TX, c.ty * TY, c.z0 + c.l, c.kb);
    }
    c.l++;
  }
};

// ---------------------------------------------------------------------------------------
// Warp-specialised variant: service warps keep the rings full, CW consumer warps compute.  Four of them, a
// warpgroup: the centre ring (and the claims of work items), the halo ring, the last term's operand ring,
// and in periodic cells the patcher of the images (a single producer for all rings was late: a wait on one
// ring held the others up; middle term of the medium molecule 0.287 -> 0.275 ms, 24 boxes of order 4 0.424
// -> 0.374).  A ring slot is handed back by an "empty" mbarrier that each consumer warp arrives on once it
// has read the slot, so the consumer warps never wait for one another inside a work item: while some warps
// read their shared-memory neighbours, others do arithmetic or store.
//
// Shapes: a tile of TX x TY points of one orbital block; a thread owns a column of R y-adjacent points, or
// (RX = 2) a block of 2 x 2, of one vector of 16 bytes (8 in shapes 5 and 8), at U planes an iteration.  The
// points of a thread share the arm values they read.  Shared-memory reads, not HBM, bound the complex64
// middle terms of order 8: a value costs 4M + 1 loads alone, (3M + 2) with two y-adjacent points, 2M + 1 in
// a block, whose inner neighbours come from the z queues.  Threads have 65536 / (32 (CW + 4)) registers:
// 168 with 6 to 8 consumer warps, 128 with 12, 96 with 16; the kernels whose queues need more split them
// (WsWarps).  tdks_autotune times the shapes on the system's own data.
//   5: 8-byte vectors (one complex64 value), four y-adjacent points in the registers of two.
//   6: shape 2 at two planes an iteration: one wait and one release per ring and two planes, and two planes'
//      loads to overlap.  Medium molecule, middle term: 0.275 -> 0.255 ms.  complex128, bound by the FP64 pipe,
//      gains in the first term of order-4 cells only (60^3, 8 orbitals, 2 k-points: 446 against shape 2's 451 us).
//   7: blocks of 2 x 2 of 16-byte vectors on 232 registers.  The fastest in cells and boxes of order 4 (64^3
//      cell, 8 k-points, 16 orbitals: 0.184 ms, shape 6 0.206, shape 3 0.230); at order 8 its 144 queue
//      registers leave one plane an iteration and 8 warps to hide the loads' latency: 0.272 against 0.255.
//   8: blocks of 2 x 2 of 8-byte vectors, two planes: 0.254 to 0.257 at order 8, 0.342 for 24 boxes of order 4
//      where shape 6 takes 0.347.
// To keep a block's loads free of bank conflicts (a point is 64 bytes, half of the banks) the odd blocks of
// a row are mirrored: their first point is the right one and their x offsets count downwards, so that two
// blocks side by side always read different halves of the banks.  The x arm is symmetric, so mirrored values
// are the same bit for bit.
template <int SHAPE> struct WsShape;
template <> struct WsShape<0> { static constexpr int U = 1, TX = 16, TY = 8, R = 2, RX = 1; };   //  8 consumer warps
template <> struct WsShape<1> { static constexpr int U = 1, TX = 16, TY = 12, R = 4, RX = 1; };  //  6
template <> struct WsShape<2> { static constexpr int U = 1, TX = 16, TY = 12, R = 2, RX = 1; };  // 12
template <> struct WsShape<3> { static constexpr int U = 1, TX = 16, TY = 8, R = 1, RX = 1; };   // 16
template <> struct WsShape<4> { static constexpr int U = 1, TX = 14, TY = 8, R = 2, RX = 1; };   //  7
template <> struct WsShape<5> { static constexpr int U = 1, TX = 16, TY = 12, R = 4, RX = 1; };  // 12 (complex64, 8-byte vectors)
template <> struct WsShape<6> { static constexpr int U = 2, TX = 16, TY = 12, R = 2, RX = 1; };  // 12 (terms 1-3)
template <> struct WsShape<7> { static constexpr int U = 2, TX = 16, TY = 16, R = 2, RX = 2; };  //  8 (complex64, terms 1-3)
template <> struct WsShape<8> { static constexpr int U = 2, TX = 16, TY = 12, R = 2, RX = 2; };  // 12 (complex64, 8-byte vectors, terms 1-3)
// planes per iteration of a shape's kernels
template <int SHAPE, int M, int BLOCH> struct WsPlanes {
  static constexpr int U = SHAPE == 7 && (M == 4 || BLOCH) ? 1 : WsShape<SHAPE>::U;
};
template <int TX, int TY, int R, int OV = OVC, int RX = 1, bool SPL = false> struct WsWarps {
  static constexpr int CW = OV * TX * TY / (32 * R * RX);  // consumer warps
  // Blocks of 2 x 2 points, and two planes at a time, want more registers than 65536 / threads: the
  // consumer warps and the four service warps start with equal shares, all there are, and the service
  // warpgroup gives most of its share to the consumers, whose z queues would spill:
  // 384 * 152 + 128 * 56 = 512 * 128 (M = 4: queues of 72 registers), 256 * 232 + 128 * 40 = 384 * 168
  // (queues of 144).
  static constexpr bool SPLIT = RX == 2 || SPL;
  static_assert(!SPLIT || CW == 12 || CW == 8, "the register splits are for twelve or eight consumer warps");
  static constexpr int CONSUMER_REGS = CW == 12 ? 152 : 232, PRODUCER_REGS = CW == 12 ? 56 : 40;
  static constexpr int THREADS = 32 * CW + 128;            // + the four service warps
  // consumer thread t owns vector t % OV of block (t / OV) % (TX / RX) of row group t / (OV TX / RX),
  // whose R rows are y-adjacent: the row groups must fill the tile and the warps exactly
  static_assert(TY % R == 0 && TX % RX == 0 && CW * 32 == OV * (TX / RX) * (TY / R),
                "row groups must fill the tile and the warps");
  static_assert(RX == 1 || (RX == 2 && R == 2), "blocks are columns of R points or 2 x 2 points");
};

// H at R y-adjacent points (rows 0 .. R-1) of one plane, from their z queues Q[r] and
// the halo plane Sp (row 0's own vector at hs0, row stride SXO vectors).  Same terms and
// summation order as stencil_point.
template <int M, int P, int QB, int QN, int R>
__device__ __forceinline__ void stencil_rows(const typename VT<P>::S *W,
                                                   const typename VT<P>::V (*Q)[QN], const typename VT<P>::V *Sp, int hs0,
                                             int SXO, const typename VT<P>::R *ve, typename VT<P>::V *acc) {
  typedef VT<P> T;
  typedef typename T::V V;
  V col[2 * M + R];  // Sp[hs0 + k SXO], k = -M .. M+R-1
#pragma unroll
  for (int k = 0; k < 2 * M + R; k++) col[k] = Sp[hs0 + (k - M) * SXO];
#pragma unroll
  for (int r = 0; r < R; r++) acc[r] = T::mul(T::diag(ve[r]), Q[r][(QB + M) % QN]);
#pragma unroll
  for (int m = 1; m <= M; m++) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int hr = hs0 + r * SXO;
      const V s = T::add(T::add(T::add(Q[r][(QB + M - m) % QN], Q[r][(QB + M + m) % QN]),
                                T::add(Sp[hr - m * T::OV], Sp[hr + m * T::OV])),
                         T::add(col[M + r - m], col[M + r + m]));
      acc[r] = T::fma(W[m], s, acc[r]);
    }
  }
}

// Bloch phase of one wrap, e^{i k_a L_a} = c + i s, in the compute precision (from the table: a sine and
// cosine in here cost registers, and the FP64 pair is a function call).
template <int P>
__device__ __forceinline__ void bloch_phase(double2 ph, typename VT<P>::S &c, typename VT<P>::S &s) {
  c = VT<P>::bc(ph.x);
  s = VT<P>::bc(ph.y);
}
// a times the phase of w wraps, (c + i s)^w (w = +-1 except in grids smaller than the stencil)
template <int P>
__device__ __forceinline__ typename VT<P>::V apply_phase(typename VT<P>::S c, typename VT<P>::S s, int w,
                                                         typename VT<P>::V a) {
  typedef VT<P> T;
  if (w < 0) {
    if constexpr (P != P_C128) s ^= SIGN2; else s = -s;
  }
  for (int i = w < 0 ? -w : w; i > 0; i--) a = T::cmul(c, s, a);
  return a;
}

// Periodic (Bloch) cell: as stencil_rows, with the velocity-gauge gradient term -i A.grad_h
// (and, for the current, the three gradients gax) in the order of stencil_point.  The halo
// slot S already holds the phased periodic images beyond the faces (the patcher warp wrote
// them), so the neighbours are read as in a finite box.
template <int M, int P, int QB, int QN, int R>
__device__ __forceinline__ void stencil_rows_bloch(const SweepParams &p, const typename VT<P>::S *W,
                                              const typename VT<P>::V (*Q)[QN],
                                                   const typename VT<P>::V *S, int hs0, int SXO,
                                                   const typename VT<P>::R *ve, typename VT<P>::V *acc,
                                                   typename VT<P>::V (*gax)[3], bool need_grad, bool grads) {
  typedef VT<P> T;
  typedef typename T::V V;
  V col[2 * M + R];  // y = gy0 - M + k
#pragma unroll
  for (int k = 0; k < 2 * M + R; k++) col[k] = S[hs0 + (k - M) * SXO];
  // gradient term as sum_m gw_m (A . d_m): 3 + M coefficients live instead of 3 M
  typename T::S A3[3] = {};
  if (need_grad) {
#pragma unroll
    for (int a = 0; a < 3; a++) A3[a] = T::bc(p.A[a]);
  }
  V gsum[R];
#pragma unroll
  for (int r = 0; r < R; r++) {
    acc[r] = T::mul(T::diag(ve[r]), Q[r][(QB + M) % QN]);
    gsum[r] = T::zero();
    gax[r][0] = gax[r][1] = gax[r][2] = T::zero();
  }
#pragma unroll
  for (int m = 1; m <= M; m++) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const V xm = S[hs0 + r * SXO - m * T::OV], xp = S[hs0 + r * SXO + m * T::OV];
      const V zm = Q[r][(QB + M - m) % QN], zp = Q[r][(QB + M + m) % QN];
      const V ym = col[M + r - m], yp = col[M + r + m];
      const V s6 = T::add(T::add(T::add(zm, zp), T::add(xm, xp)), T::add(ym, yp));
      acc[r] = T::fma(W[m], s6, acc[r]);
      if (need_grad) {
        const V dx = T::sub(xp, xm), dy = T::sub(yp, ym), dz = T::sub(zp, zm);
        const typename T::S gm = T::bc(p.gw[m]);
        const V dA = T::fma(A3[0], dx, T::fma(A3[1], dy, T::mul(A3[2], dz)));
        gsum[r] = T::fma(gm, dA, gsum[r]);
        if (grads) {
          gax[r][0] = T::fma(gm, dx, gax[r][0]);
          gax[r][1] = T::fma(gm, dy, gax[r][1]);
          gax[r][2] = T::fma(gm, dz, gax[r][2]);
        }
      }
    }
  }
  if (need_grad) {
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = T::add(acc[r], T::negi(gsum[r]));
  }
}

// H at a 2 x 2 block of points (point q = 2 r + c: row r, column c) from their z queues Q[q] and
// the halo plane, S0 = the block's first point's vector.  sx = +-OV: the vector stride from column 0 to
// column 1 (mirrored blocks count x downwards).  Same terms and summation order as stencil_point.
// Inner neighbours come from the queues: in a finite box points of the block beyond the grid are zero
// there as in the halo plane; a periodic cell takes this shape only where nx and ny are even, so that a
// block lies inside the cell or outside it as a whole.
template <int M, int P, int BLOCH, int QB, int QN>
__device__ __forceinline__ void stencil_block(const SweepParams &p, const typename VT<P>::S *W,
                                              const typename VT<P>::V (*Q)[QN],
                                              const typename VT<P>::V *S0, int SXO, int sx,
                                              const typename VT<P>::R *ve, typename VT<P>::V *acc,
                                              typename VT<P>::V (*gax)[3], bool need_grad, bool grads) {
  typedef VT<P> T;
  typedef typename T::V V;
  typename T::S A3[3] = {};
  if (BLOCH && need_grad) {
#pragma unroll
    for (int a = 0; a < 3; a++) A3[a] = T::bc(a == 0 && sx < 0 ? -p.A[a] : p.A[a]);
  }
  V gsum[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    acc[q] = T::mul(T::diag(ve[q]), Q[q][(QB + M) % QN]);
    if (BLOCH) {
      gsum[q] = T::zero();
      gax[q][0] = gax[q][1] = gax[q][2] = T::zero();
    }
  }
  // outer neighbours of the last distance: x- of row r, x+ of row r; y- of column c, y+ of column c
  V xl[2], xh[2], yl[2], yh[2];
#pragma unroll
  for (int i = 0; i < 2; i++) {
    xl[i] = Q[2 * i][(QB + M) % QN];
    xh[i] = Q[2 * i + 1][(QB + M) % QN];
    yl[i] = Q[i][(QB + M) % QN];
    yh[i] = Q[2 + i][(QB + M) % QN];
  }
#pragma unroll
  for (int m = 1; m <= M; m++) {
    // (x arms first, then y arms: half of the neighbours live at a time)
    V xln[2], xhn[2], yln[2], yhn[2], szx[4];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      xln[i] = (S0 - m * sx)[i * SXO];
      xhn[i] = (S0 + (m + 1) * sx)[i * SXO];
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = q >> 1, c = q & 1;
      const V xm = c == 0 ? xln[r] : xl[r], xp = c == 0 ? xh[r] : xhn[r];
      szx[q] = T::add(T::add(Q[q][(QB + M - m) % QN], Q[q][(QB + M + m) % QN]), T::add(xm, xp));
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
      yln[i] = (S0 + i * sx)[-m * SXO];
      yhn[i] = (S0 + i * sx)[(m + 1) * SXO];
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = q >> 1, c = q & 1;
      const V xm = c == 0 ? xln[r] : xl[r], xp = c == 0 ? xh[r] : xhn[r];
      const V ym = r == 0 ? yln[c] : yl[c], yp = r == 0 ? yh[c] : yhn[c];
      const V zm = Q[q][(QB + M - m) % QN], zp = Q[q][(QB + M + m) % QN];
      const V s6 = T::add(szx[q], T::add(ym, yp));
      acc[q] = T::fma(W[m], s6, acc[q]);
      if (BLOCH && need_grad) {
        const V dx = T::sub(xp, xm), dy = T::sub(yp, ym), dz = T::sub(zp, zm);
        const typename T::S gm = T::bc(p.gw[m]);
        const V dA = T::fma(A3[0], dx, T::fma(A3[1], dy, T::mul(A3[2], dz)));
        gsum[q] = T::fma(gm, dA, gsum[q]);
        if (grads) {
          gax[q][0] = T::fma(sx < 0 ? T::bc(-p.gw[m]) : gm, dx, gax[q][0]);
          gax[q][1] = T::fma(gm, dy, gax[q][1]);
          gax[q][2] = T::fma(gm, dz, gax[q][2]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
      xl[i] = xln[i];
      xh[i] = xhn[i];
      yl[i] = yln[i];
      yh[i] = yhn[i];
    }
  }
  if (BLOCH && need_grad) {
#pragma unroll
    for (int q = 0; q < 4; q++) acc[q] = T::add(acc[q], T::negi(gsum[q]));
  }
}

template <int M, int P, int MODE, int TX, int TY, int R, int RX, int U, bool BATCH, int BLOCH, class Src>
__device__ __forceinline__ void ws_sweep_body(const Src &src, unsigned int *work) {
  typedef VT<P> T;
  typedef typename T::V V;
  typedef typename T::S S_;
  typedef typename T::R Rv;
  constexpr bool OPS = MODE == MODE_LAST;
  typedef TmaGeom<M, TX, TY, U, OPS, BLOCH != 0, MODE == MODE_FIRST> G;
  static_assert(M % U == 0, "M must be a multiple of U");
  static_assert(!OPS || U == 1, "the last Taylor term takes one plane per iteration");
  constexpr int OV = T::OV;       // thread vectors per (point, batch)
  constexpr int CPL = TX * TY * OV;  // thread vectors per centre plane or operand tile
  constexpr int CW = WsWarps<TX, TY, R, OV, RX>::CW;
  constexpr int NP = R * RX;      // points per consumer thread
  constexpr int SC = G::SC, SH = G::SH;
  constexpr int SO = G::SO > 0 ? G::SO : 1;
  constexpr int QN = 2 * M + U;   // z-queue entries
  constexpr int LP = 2 * M / U;   // priming centre loads per item
  // order-8 blocks of 16-byte vectors: their queues leave no registers for projector terms in flight
  constexpr bool LATE_NL = RX == 2 && M == 4 && T::OV == 4;
  constexpr int IR = 16;          // claimed-item ring (the producer runs at most a few items ahead)
  extern __shared__ unsigned char smem_raw[];
  unsigned char *cbase = smem_raw + ((0u - smem_u32(smem_raw)) & 127u);
  unsigned char *hbase = cbase + (size_t)SC * G::CSLOT_BYTES;
  unsigned char *obase = hbase + (size_t)SH * G::HSLOT_BYTES;
  __shared__ __align__(8) uint64_t cfull[SC], cempty[SC];
  __shared__ __align__(8) uint64_t hfull[SH], hempty[SH];
  __shared__ __align__(8) uint64_t hready[BLOCH ? SH : 1];  // periodic cells: face images written
  __shared__ __align__(8) uint64_t ofull[SO], oempty[SO];
  __shared__ __align__(8) uint64_t ibar[IR];  // completes when s_item[seq % IR] is written
  __shared__ long s_item[IR];                 // item of the CTA's seq-th claim (-1: no more)
  __shared__ int s_abort;
  volatile int *abort_flag = &s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const long n_items_all = src.n_items();

  if (tid == 0) {
    for (int s = 0; s < SC; s++) { mbar_init(&cfull[s], 1); mbar_init(&cempty[s], CW); }
    for (int s = 0; s < SH; s++) { mbar_init(&hfull[s], 1); mbar_init(&hempty[s], CW); }
    if (BLOCH)
      for (int s = 0; s < SH; s++) mbar_init(&hready[s], 1);
    for (int s = 0; s < SO; s++) { mbar_init(&ofull[s], 1); mbar_init(&oempty[s], CW); }
    for (int s = 0; s < IR; s++) mbar_init(&ibar[s], 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();  // the only CTA-wide barrier: from here on the warps run decoupled

  // (Records, and the last term's operands, beside the queues and face phases of order 8 in a cell spill at
  // eight warps' 168 registers: 64^3, 8 k-points, 16 orbitals 0.80 -> 0.69 and 0.81 -> 0.74 ms.  The middle
  // terms lose by the split, 0.364 -> 0.373.)
  typedef WsWarps<TX, TY, R, OV, RX, U == 2 || (BLOCH && M == 4 && CW == 8 && MODE != MODE_MID)> WW;
  if (warp >= CW) {
  if constexpr (WW::SPLIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(WW::PRODUCER_REGS));
  // ---- producers: one warp per ring (warp CW the centre planes, CW + 1 the halo planes, CW + 2 the
  // last term's operands), each refilling its ring's slots in order as they are released.  One warp
  // for all three rings polled them in turn and set the pace of the CTA: ~1450 cycles per plane with
  // the consumers' stencil taken out, whatever the tile.  The centre producer, which runs ahead of
  // the others, claims the items.
  // (failure injection: withholding producers do nothing, so the other warps' waits run out; no copy
  // is in flight and nothing needs draining)
  auto serve = [&](auto kind_c) {
    constexpr int KIND = decltype(kind_c)::value;
    constexpr int S = KIND == 0 ? SC : (KIND == 1 ? SH : SO);
    uint64_t *full = KIND == 0 ? cfull : (KIND == 1 ? hfull : ofull);
    uint64_t *empty = KIND == 0 ? cempty : (KIND == 1 ? hempty : oempty);
    const Loader<M, TX, TY, U, 1, G, SC, SH, SO, Src> ld{src, 0, cbase, hbase, obase, cfull, hfull, ofull};
    RingPos rp;
    unsigned issued = 0;
    bool gave_up = false;
    [[maybe_unused]] int mapped = -1;  // batch: the system whose maps this thread has acquired last
    for (unsigned seq = 0; !gave_up; seq++) {
      if constexpr (KIND == 0) {
        // (a CTA's first item is its own number, without a round trip to the counter; then every CTA
        // claims until one claim is past the last item: n_items claims in all, the last of which
        // returns the counter to zero for the next launch)
        long t = blockIdx.x;
        if (seq > 0) {
          const unsigned int r = atomicAdd(work, 1u);
          if ((long)r == n_items_all - 1) atomicExch(work, 0u);
          t = (long)gridDim.x + (long)r;
        }
        s_item[seq % IR] = t < n_items_all ? t : -1;
        mbar_arrive(&ibar[seq % IR]);
      } else if (!mbar_wait_or_abort(&ibar[seq % IR], (seq / IR) & 1u, abort_flag)) {
        gave_up = true;
        break;
      }
      const long it = s_item[seq % IR];
      if (it < 0) break;
      const SweepParams *qp = nullptr;
      const SweepMaps *mq = nullptr;
      long local = 0;
      src.item(it, qp, mq, local);
      LoadCursor cu{};
      int z1 = 0;
      item_geom(*qp, local, cu.tx, cu.ty, cu.kb, cu.z0, z1);
      cu.sys = src.sys_of(it);
      cu.nx = qp->nx;
      cu.ny = qp->ny;
      cu.nz = qp->nz;
      cu.wrap = qp->bloch;
      if (BATCH && cu.sys != mapped) {
        mapped = cu.sys;
        const SweepMaps *mp = src.maps_of(mapped);
        if constexpr (KIND == 0) tma_acquire_map(&mp->ctr);
        if constexpr (KIND == 1) {
          tma_acquire_map(&mp->in);
          tma_acquire_map(&mp->aux);
        }
        if constexpr (KIND == 2)
          for (int j = 0; j < 4; j++) tma_acquire_map(&mp->op[j]);
      }
      const int n = loads_of<M, U>(KIND, cu.z0, z1);
      // (sending the last term's operand tiles to L2 four or eight planes ahead of their loads made it
      // 18% and 36% slower on the medium molecule: eight streams per CTA are enough for the DRAM)
      for (cu.l = 0; cu.l < n;) {
        // the slot is free once the consumers have released its previous use (at once the first time)
        if (!mbar_wait_or_abort(&empty[rp.slot], rp.phase ^ 1u, abort_flag)) {
          gave_up = true;
          break;
        }
        // The copy writes the slot through the asynchronous proxy, the consumers read it (and the patcher warp
        // writes it) through the generic one: across the two, only this fence orders what came before the
        // release with the copy that follows it.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ld.emit_at(cu, KIND, rp.slot);
        rp.next<S>();
        issued++;
      }
    }
    if (gave_up) *abort_flag = 1;
    // copies still in flight must land before the CTA's shared memory goes away
    for (unsigned j = issued > S ? issued - S : 0; j < issued; j++)
      mbar_wait_bounded(&full[j % S], (j / S) & 1u, DRAIN_LIMIT_CYCLES);
  };
  if (warp >= CW && warp < CW + 3) {
    if (lane == 0 && !src.withhold()) {
      if constexpr (!BATCH) {
        const SweepMaps *mp = src.maps_of(0);
        if (warp == CW) tma_prefetch_map(&mp->ctr);
        if (warp == CW + 1) {
          tma_prefetch_map(&mp->in);
          tma_prefetch_map(&mp->aux);
        }
        if (OPS && warp == CW + 2)
          for (int j = 0; j < 4; j++) tma_prefetch_map(&mp->op[j]);
      }
      if (warp == CW) serve(std::integral_constant<int, 0>{});
      if (warp == CW + 1) serve(std::integral_constant<int, 1>{});
      if (OPS && warp == CW + 2) serve(std::integral_constant<int, 2>{});
    }
    return;
  }

  if (BLOCH && warp == CW + 3) {
    // ---- patcher (periodic cells): for each output plane of each item, once the halo slot
    // has landed, write the Bloch-phased periodic images of the strips beyond the cell's
    // x and y faces into the halo box (where the TMA box holds zeros), then release the
    // slot to the consumers -----------------------------------------------------------------
    RingPos rp;
    for (unsigned seq = 0;; seq++) {
      if (!mbar_wait_or_abort(&ibar[seq % IR], (seq / IR) & 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      const long item = s_item[seq % IR];
      if (item < 0) break;
      const SweepParams *pp;
      const SweepMaps *mp_unused;
      long local;
      src.item(item, pp, mp_unused, local);
      const SweepParams &p = *pp;
      int tx, ty, kb, z0, z1;
      item_geom(p, local, tx, ty, kb, z0, z1);
      const int nx = p.nx, ny = p.ny, x0 = tx * TX, y0 = ty * TY;
      const bool sl = x0 - M < 0, sr = x0 + TX + M > nx, st = y0 - M < 0, sb = y0 + TY + M > ny;
      const int kidx = kb / p.n_batches;
      S_ cx, sx, cy, sy;
      bloch_phase<P>(p.kphase[3 * kidx], cx, sx);
      bloch_phase<P>(p.kphase[3 * kidx + 1], cy, sy);
      constexpr int VB = (int)sizeof(V);  // bytes per thread vector
      constexpr int SRB = (int)(G::STRIPX_BYTES / VB);
      constexpr int STB = SRB + (int)(G::STRIPX_BYTES / VB);
      constexpr int SBB = STB + (int)(G::STRIPY_BYTES / VB);
      bool gave_up = false;
      for (int z = z0; z < z1; z += U) {
        const int hs = rp.slot;
        if (!mbar_wait_or_abort(&hfull[hs], rp.phase, abort_flag)) {
          gave_up = true;
          break;
        }
#pragma unroll 1
        for (int u = 0; u < U; u++) {
          unsigned char *slot = hbase + (size_t)hs * G::HSLOT_BYTES;
          V *box = reinterpret_cast<V *>(slot + (size_t)u * G::PLANE * 16);
          const V *strips = reinterpret_cast<const V *>(slot + G::IN_BYTES + G::AUX_BYTES + (size_t)u * G::STRIP1_BYTES);
          if (sl || sr) {
            // box columns c with grid x = x0 - M + c beyond x = 0 (c < M) or beyond x = nx - 1
            const int cr0 = nx - x0 + M;  // first box column past the last grid column
            for (int i = lane; i < 2 * G::SY * M * OV; i += 32) {
              const int v = i % OV, j = (i / OV) % M, row = (i / (OV * M)) % G::SY, side = i / (OV * M * G::SY);
              if (side == 0 ? !sl : !sr) continue;
              const int c = side == 0 ? j : cr0 + j;
              if (c >= G::SX) continue;
              const V a = strips[(side == 0 ? 0 : SRB) + (row * M + j) * OV + v];
              box[(row * G::SX + c) * OV + v] = apply_phase<P>(cx, sx, side == 0 ? -1 : 1, a);
            }
          }
          if (st || sb) {
            // box rows rr with grid y = y0 - M + rr beyond y = 0 (rr < M) or beyond y = ny - 1,
            // over the tile's columns (the star stencil never reads the corners)
            const int rb0 = ny - y0 + M;
            for (int i = lane; i < 2 * M * TX * OV; i += 32) {
              const int v = i % OV, c = (i / OV) % TX, j = (i / (OV * TX)) % M, side = i / (OV * TX * M);
              if (side == 0 ? !st : !sb) continue;
              const int rr = side == 0 ? j : rb0 + j;
              if (rr >= G::SY) continue;
              const V a = strips[(side == 0 ? STB : SBB) + (j * TX + c) * OV + v];
              box[(rr * G::SX + c + M) * OV + v] = apply_phase<P>(cy, sy, side == 0 ? -1 : 1, a);
            }
          }
          if (G::NLS && p.has_proj) {
            // the plane's non-local rows: row r0 of each sphere point (points outside every
            // sphere are never read from here), in 16-byte units whatever the size of a vector
            const PointAux *ax = reinterpret_cast<const PointAux *>(slot + G::IN_BYTES) + u * TX * TY;
            ulonglong2 *nla = reinterpret_cast<ulonglong2 *>(slot + G::IN_BYTES + G::AUX_BYTES + G::STRIP_BYTES) +
                              u * TX * TY * OVC;
            const ulonglong2 *nlk = reinterpret_cast<const ulonglong2 *>(p.nl) + (long)kb * (p.n_ent + 1) * OVC;
            for (int i = lane; i < TX * TY * OVC; i += 32) {
              const PointAux a = ax[i / OVC];
              if (a.r1 > a.r0) cp_async_16(nla + i, nlk + (long)a.r0 * OVC + i % OVC);
            }
          }
        }
        if (G::NLS && p.has_proj) cp_async_arrive(&hready[hs]);
        __syncwarp();
        if (lane == 0) mbar_arrive(&hready[hs]);
        rp.next<SH>();
      }
      if (gave_up) {
        *abort_flag = 1;
        break;
      }
    }
    cp_async_wait_all();  // no copy may land after the CTA's shared memory is gone
    return;
  }
  return;
  }
  if constexpr (WW::SPLIT) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(WW::CONSUMER_REGS));

  // ---- consumers: no barrier between warps; a warp that gives up stops, and the others
  // give up at their next wait ----------------------------------------------------------------
  // (point q = RX r + c of the thread's block: row r, column c; odd blocks of a row are mirrored)
  const int v = tid % OV;
  const int lb = (tid / OV) % (TX / RX);                      // block of the row
  const int sx = RX == 2 && (lb & 1) ? -OV : OV;              // vector stride from column 0 to column 1
  const int lx = RX * lb + (sx < 0 ? 1 : 0);                  // column 0's x
  const int ly0 = R * (tid / (OV * (TX / RX)));
  const int hs0 = ((ly0 + M) * G::SX + (lx + M)) * OV + v;   // point 0's vector in a halo plane
  const int tsl0 = ly0 * TX + lx;                             // point 0 in a tile
  const int csl0 = tsl0 * OV + v;                             // point 0's vector in a centre plane
  const int dx1 = sx < 0 ? -1 : 1;                            // points from column 0 to column 1
  constexpr int SXO = G::SX * OV;

  RingPos rc, rh, ro;  // ring positions of the next centre / halo / operand load
  bool aborted = false;
  int *errp = src.err0();  // then the current item's system's
  for (unsigned seq = 0;; seq++) {
    if (!mbar_wait_or_abort(&ibar[seq % IR], (seq / IR) & 1u, abort_flag)) {
      aborted = true;
      break;
    }
    const long item = s_item[seq % IR];
    if (item < 0) break;
    const SweepParams *pp;
    const SweepMaps *mp_unused;
    long local;
    src.item(item, pp, mp_unused, local);
    const SweepParams &p = *pp;  // (batch: read from the parameter array, once per item)
    errp = p.err;
    const int nx = p.nx, ny = p.ny;
    const long N = (long)nx * ny * p.nz;
    const long plane_pts = (long)nx * ny;
    S_ W[M + 1];
#pragma unroll
    for (int m = 0; m <= M; m++) W[m] = T::coef(p.w[m], p.wf[m]);
    const bool kim = p.coef_im != 0;
    const typename T::K KC = T::kcoef(p.coef, p.coeff, kim);
    int tx, ty, kb, z0, z1;
    item_geom(p, local, tx, ty, kb, z0, z1);
    const int kidx = kb / p.n_batches;
    const Epi epi = make_epi(p, kidx);
    const bool has_proj = p.has_proj != 0, do_obs = p.do_obs != 0;
    const V *nlk = nl_column<P>(p, kb, v);
    const int gx = tx * TX + lx, gy0 = ty * TY + ly0;
    // periodic cell: the Bloch phase of one wrap along z, e^{i k_z L_z} = cz + i sz, applied to
    // the queue planes loaded from beyond a z face (the patcher warp handles x and y)
    S_ cz{}, sz{};
    if constexpr (BLOCH) bloch_phase<P>(p.kphase[3 * kidx + 2], cz, sz);
    S_ szm = sz;  // -sz: one wrap the other way
    if constexpr (P != P_C128) szm ^= SIGN2; else szm = -szm;
    const bool need_grad = BLOCH && p.grad_mask != 0;
    const bool grads = BLOCH && MODE == MODE_FIRST && (p.grad_mask & 8);
    bool own[NP];
#pragma unroll
    for (int q = 0; q < NP; q++) own[q] = gx + (q % RX) * dx1 < nx && gy0 + q / RX < ny;
    const int nl = loads_of<M, U>(0, z0, z1);
    // vector index of point 0 in the first output plane (advances one plane per output)
    long idx = ((long)kb * N + ((long)z0 * ny + gy0) * nx + gx) * OV + v;
    const long row = (long)nx * OV;
    V Q[NP][QN];
#pragma unroll
    for (int q = 0; q < NP; q++)
#pragma unroll
      for (int j = 0; j < QN; j++) Q[q][j] = T::zero();
    ObsAcc<P> oa;

    int l = 0;
    // one centre load (and, past the priming loads, one halo load); RQ = compile-time
    // queue position of its first plane
    auto iteration = [&](auto rq) {
      constexpr int RQ = decltype(rq)::value;
      const int cs = rc.slot;
      if (!mbar_wait_or_abort(&cfull[cs], rc.phase, abort_flag)) {
        aborted = true;
        return;
      }
      const V *cslot = reinterpret_cast<const V *>(cbase + (size_t)cs * G::CSLOT_BYTES);
#pragma unroll
      for (int u = 0; u < U; u++) {
#pragma unroll
        for (int q = 0; q < NP; q++)
          Q[q][(RQ + u) % QN] = (cslot + (q % RX) * sx)[u * CPL + csl0 + (q / RX) * TX * OV];
        if constexpr (BLOCH) {
          // a plane beyond a z face was loaded from its periodic image: apply the Bloch phase
          const int zq = z0 - M + U * l + u;
          if ((unsigned)zq >= (unsigned)p.nz) {
            // (nz >= M: the planes a live output reads are one wrap away)
            const S_ s1 = zq < 0 ? szm : sz;
#pragma unroll
            for (int q = 0; q < NP; q++) Q[q][(RQ + u) % QN] = T::cmul(cz, s1, Q[q][(RQ + u) % QN]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&cempty[cs]);
      rc.next<SC>();
      if (l >= LP) {
        const int zf = z0 + U * (l - LP);
        const int hs = rh.slot;
        // periodic cells: the slot is ready once the patcher warp has written the face images
        if (!mbar_wait_or_abort(BLOCH ? &hready[hs] : &hfull[hs], rh.phase, abort_flag)) {
          aborted = true;
          return;
        }
        const unsigned char *hslot = hbase + (size_t)hs * G::HSLOT_BYTES;
        const V *xs = reinterpret_cast<const V *>(hslot);
        const PointAux *ax = reinterpret_cast<const PointAux *>(hslot + G::IN_BYTES);
        const V *ob = nullptr;  // last term: the operand slot, read row by row at the epilogue
        int os = 0;
        if constexpr (OPS) {
          os = ro.slot;
          if (!mbar_wait_or_abort(&ofull[os], ro.phase, abort_flag)) {
            aborted = true;
            return;
          }
          ob = reinterpret_cast<const V *>(obase + (size_t)os * G::OP_BYTES);
        }
        (void)ob;
        (void)os;
        auto operands = [&](int c) {
          LastOperands<P> o;
          if constexpr (OPS) {
            o.hi = ob[c];
            o.lo = ob[CPL + c];
            o.t1 = ob[2 * CPL + c];
            o.t2 = ob[3 * CPL + c];
          } else {
            (void)c;
            o.hi = o.lo = o.t1 = o.t2 = T::zero();
          }
          return o;
        };
        static_for<0, U>([&](auto uc) {
          constexpr int u = decltype(uc)::value;
          constexpr int QB = (RQ + U + u) % QN;  // queue position of plane (zf + u) - M
          Rv ve[NP];
          V nlv[NP], acc[NP];
          [[maybe_unused]] bool in_sphere = false;
#pragma unroll
          for (int q = 0; q < NP; q++) {
            const PointAux a = (ax + (q % RX) * dx1)[u * TX * TY + tsl0 + (q / RX) * TX];
            ve[q] = *reinterpret_cast<const Rv *>(&a.veff);
            if constexpr (P == P_C128) in_sphere = in_sphere || a.r1 > a.r0;
            if constexpr (LATE_NL) {
              // (loaded after the stencil, below)
            } else if constexpr (G::NLS) {
              // (gathered into the slot by the patcher warp)
              const V *nla = reinterpret_cast<const V *>(hslot + G::IN_BYTES + G::AUX_BYTES + G::STRIP_BYTES);
              nlv[q] = has_proj && a.r1 > a.r0 ? (nla + (q % RX) * sx)[(u * TX * TY + tsl0 + (q / RX) * TX) * OV + v] : T::zero();
            } else {
              nlv[q] = has_proj ? nl_term<P>(nlk, a.r0, a.r1) : T::zero();
            }
          }
          [[maybe_unused]] V gax[BLOCH ? NP : 1][3];
          if constexpr (RX == 2) {
            stencil_block<M, P, BLOCH, QB, QN>(p, W, Q, xs + u * G::SX * G::SY * OV + hs0, SXO, sx, ve, acc, gax,
                                               need_grad, grads);
          } else if constexpr (BLOCH) {
            stencil_rows_bloch<M, P, QB, QN, R>(p, W, Q, xs + u * G::SX * G::SY * OV, hs0, SXO, ve, acc, gax, need_grad, grads);
          } else {
            stencil_rows<M, P, QB, QN, R>(W, Q, xs + u * G::SX * G::SY * OV, hs0, SXO, ve, acc);
          }
          if constexpr (LATE_NL) {
#pragma unroll
            for (int q = 0; q < NP; q++) {
              const PointAux a = (ax + (q % RX) * dx1)[u * TX * TY + tsl0 + (q / RX) * TX];
              nlv[q] = has_proj ? nl_term<P>(nlk, a.r0, a.r1) : T::zero();
            }
          }
          const long iu = idx + (long)u * plane_pts * OV;
          // (complex128: two FP64 sums per value are worth a vote; most warps meet no sphere)
          const bool add_nl = has_proj && (P != P_C128 || __any_sync(0xffffffffu, in_sphere));
#pragma unroll
          for (int q = 0; q < NP; q++) {
            const bool live = own[q] && (zf + u < z1);
            if (add_nl) {
              if constexpr (P == P_C128) asm volatile("");  // (a branch: speculated, the sums are not saved)
              acc[q] = T::add(acc[q], nlv[q]);
            }
            const V c0 = Q[q][(QB + M) % QN];
            if (MODE == MODE_FIRST && do_obs && live) {
              oa.add_e(c0, acc[q]);
              if constexpr (BLOCH) {
                if (grads) {
#pragma unroll
                  for (int a = 0; a < 3; a++) oa.add_j(a, c0, gax[q][a]);
                }
              }
            }
            finish_point<P, MODE>(epi, KC, kim, live, iu + (q / RX) * row + (q % RX) * sx, v, c0, acc[q],
                                  operands(csl0 + (q / RX) * TX * OV + (q % RX) * sx));
          }
        });
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&hempty[hs]);
          if constexpr (OPS) mbar_arrive(&oempty[os]);
        }
        idx += U * plane_pts * OV;
        rh.next<SH>();
        if (OPS) ro.next<SO>();
      }
      l++;
    };
    // every item starts at queue rotation 0, so the plane loop runs in unrolled blocks of
    // QN / U iterations (one full turn of the queue), each with its compile-time rotation
    while (l < nl && !aborted) {
      static_for<0, QN / U>([&](auto j) {
        if (l < nl && !aborted) iteration(std::integral_constant<int, decltype(j)::value * U>{});
      });
    }
    if (aborted) break;
    if (MODE == MODE_FIRST && do_obs) {
      // this warp's partials of the item: record local * CW + warp
      double vals[4] = {oa.get_e(), oa.get_j(0), oa.get_j(1), oa.get_j(2)};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        double x = vals[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) p.obs_part[(local * CW + warp) * 4 + i] = epi.wocc * x;
      }
    }
  }
  if (aborted) {
    *abort_flag = 1;
    if (lane == 0 && errp) atomicExch(errp, 1);
  }
}

template <int M, int P, int MODE, int TX, int TY, int R, int RX, int U, int BLOCH>
__global__ void __launch_bounds__(WsWarps<TX, TY, R, VT<P>::OV, RX>::THREADS, 1)
ws_sweep_kernel(const __grid_constant__ SweepMaps maps, const __grid_constant__ SweepParams p) {
  const SingleSrc src{&p, &maps};
  ws_sweep_body<M, P, MODE, TX, TY, R, RX, U, false, BLOCH>(src, p.work);
}

template <int M, int P, int MODE, int TX, int TY, int R, int RX, int U>
__global__ void __launch_bounds__(WsWarps<TX, TY, R, VT<P>::OV, RX>::THREADS, 1)
ws_sweep_batch_kernel(const __grid_constant__ BatchSweepArgs a) {
  const BatchSrc src{&a};
  ws_sweep_body<M, P, MODE, TX, TY, R, RX, U, true, 0>(src, a.work);
}

// Launch of the warp-specialised sweep of shape SHAPE for one system (one plane per
// iteration; grid <= 0: one CTA per SM, at most one per work item).
template <int SHAPE, int M, int P, int MODE, int BLOCH>
static cudaError_t launch_ws_t(const SweepMaps &maps, const SweepParams &p, int grid, cudaStream_t s) {
  constexpr int TX = WsShape<SHAPE>::TX, TY = WsShape<SHAPE>::TY, R = WsShape<SHAPE>::R, RX = WsShape<SHAPE>::RX;
  constexpr int U = WsPlanes<SHAPE, M, BLOCH>::U;
  typedef TmaGeom<M, TX, TY, U, MODE == MODE_LAST, BLOCH != 0, MODE == MODE_FIRST> G;
  auto k = ws_sweep_kernel<M, P, MODE, TX, TY, R, RX, U, BLOCH>;
  static std::atomic<unsigned> attr_done{0};
  if (cudaError_t e = ensure_smem_attr(k, G::SMEM, attr_done)) return e;
  if (grid <= 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = (int)(p.n_items < sms ? p.n_items : sms);
  }
  k<<<grid, WsWarps<TX, TY, R, VT<P>::OV, RX>::THREADS, G::SMEM, s>>>(maps, p);
  return cudaGetLastError();
}

// Launch of the batched warp-specialised sweep of shape SHAPE: 152 persistent CTAs (one per
// SM, at most one per work item) walk the items of every system of the batch.
template <int SHAPE, int M, int P, int MODE>
static cudaError_t launch_ws_batch_t(const BatchSweepArgs &a, cudaStream_t s) {
  constexpr int TX = WsShape<SHAPE>::TX, TY = WsShape<SHAPE>::TY, R = WsShape<SHAPE>::R, RX = WsShape<SHAPE>::RX;
  constexpr int U = WsPlanes<SHAPE, M, 0>::U;
  typedef TmaGeom<M, TX, TY, U, MODE == MODE_LAST, false, MODE == MODE_FIRST> G;
  auto k = ws_sweep_batch_kernel<M, P, MODE, TX, TY, R, RX, U>;
  static std::atomic<unsigned> attr_done{0};
  if (cudaError_t e = ensure_smem_attr(k, G::SMEM, attr_done)) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = (int)(a.total_items < sms ? a.total_items : sms);
  if (grid <= 0) return cudaSuccess;
  k<<<grid, WsWarps<TX, TY, R, VT<P>::OV, RX>::THREADS, G::SMEM, s>>>(a);
  return cudaGetLastError();
}

// Shapes 5 to 8 exist for some systems; what runs where is decided by ws_kernel_shape, which the
// launchers below rely on: shape 5 complex64 boxes, 6 to 8 terms 1 to 3 of complex64 boxes and order-4
// cells, 6 also of complex128.  Shapes 5 and 8 compute one complex64 value per thread vector, 6 and 7 two.
template <int SHAPE> struct C64Shape {
  static constexpr bool ONLY = SHAPE >= 5;
  static constexpr int P = SHAPE == 7 || SHAPE == 6 ? P_C64 : P_C64S;
  static constexpr bool CELL = SHAPE >= 6;     // has periodic-cell kernels (order 4)
  static constexpr bool LAST = SHAPE == 5;     // has last-term kernels
};

template <int SHAPE>
cudaError_t launch_ws_batch_shape(int M, int prec, int mode, const BatchSweepArgs &a, cudaStream_t s) {
#define TDKS_WSB_MODES(MM, PP)                                                    \
  switch (mode) {                                                                 \
    case MODE_FIRST: return launch_ws_batch_t<SHAPE, MM, PP, MODE_FIRST>(a, s);   \
    case MODE_MID: return launch_ws_batch_t<SHAPE, MM, PP, MODE_MID>(a, s);       \
    case MODE_LAST: return launch_ws_batch_t<SHAPE, MM, PP, MODE_LAST>(a, s);     \
  }                                                                               \
  return cudaErrorInvalidValue;
  if constexpr (C64Shape<SHAPE>::ONLY) {
    constexpr int P = C64Shape<SHAPE>::P;
    if constexpr (SHAPE == 6) {
      if (prec == P_C128 && M == 2 && mode == MODE_FIRST) return launch_ws_batch_t<SHAPE, 2, P_C128, MODE_FIRST>(a, s);
      if (prec == P_C128 && M == 2 && mode == MODE_MID) return launch_ws_batch_t<SHAPE, 2, P_C128, MODE_MID>(a, s);
      if (prec == P_C128 && M == 4 && mode == MODE_FIRST) return launch_ws_batch_t<SHAPE, 4, P_C128, MODE_FIRST>(a, s);
      if (prec == P_C128 && M == 4 && mode == MODE_MID) return launch_ws_batch_t<SHAPE, 4, P_C128, MODE_MID>(a, s);
    }
    if (prec != P_C64) return cudaErrorInvalidValue;
    if constexpr (C64Shape<SHAPE>::LAST) {
      if (M == 2 && mode == MODE_LAST) return launch_ws_batch_t<SHAPE, 2, P, MODE_LAST>(a, s);
      if (M == 4 && mode == MODE_LAST) return launch_ws_batch_t<SHAPE, 4, P, MODE_LAST>(a, s);
    }
    if (M == 2 && mode == MODE_FIRST) return launch_ws_batch_t<SHAPE, 2, P, MODE_FIRST>(a, s);
    if (M == 2 && mode == MODE_MID) return launch_ws_batch_t<SHAPE, 2, P, MODE_MID>(a, s);
    if (M == 4 && mode == MODE_FIRST) return launch_ws_batch_t<SHAPE, 4, P, MODE_FIRST>(a, s);
    if (M == 4 && mode == MODE_MID) return launch_ws_batch_t<SHAPE, 4, P, MODE_MID>(a, s);
  } else {
    if (prec == P_C64) {
      if constexpr (SHAPE != 1) {
        if (M == 2) { TDKS_WSB_MODES(2, P_C64) }
        if (M == 4) { TDKS_WSB_MODES(4, P_C64) }
      }
      return cudaErrorInvalidValue;
    }
    if (M == 2) { TDKS_WSB_MODES(2, P_C128) }
    if (M == 4) { TDKS_WSB_MODES(4, P_C128) }
  }
#undef TDKS_WSB_MODES
  return cudaErrorInvalidValue;
}

// One boundary kind of one shape: every mode, FD order and precision.
template <int SHAPE, int BLOCH>
static cudaError_t launch_ws_bc(int M, int prec, int mode, const SweepMaps &maps, const SweepParams &p, int grid,
                                cudaStream_t s) {
#define TDKS_WS_MODES(MM, PP)                                                                \
  switch (mode) {                                                                            \
    case MODE_FIRST: return launch_ws_t<SHAPE, MM, PP, MODE_FIRST, BLOCH>(maps, p, grid, s); \
    case MODE_MID: return launch_ws_t<SHAPE, MM, PP, MODE_MID, BLOCH>(maps, p, grid, s);     \
    case MODE_LAST: return launch_ws_t<SHAPE, MM, PP, MODE_LAST, BLOCH>(maps, p, grid, s);   \
  }                                                                                          \
  return cudaErrorInvalidValue;
  // (complex64: shape 1 not at all, shape 2 in cells the last term of order 4 only)
  if (prec == P_C64) {
    if constexpr (SHAPE == 2 && BLOCH) {
      if (M == 2 && mode == MODE_LAST) return launch_ws_t<SHAPE, 2, P_C64, MODE_LAST, BLOCH>(maps, p, grid, s);
    } else if constexpr (SHAPE != 1) {
      if (M == 2) { TDKS_WS_MODES(2, P_C64) }
      if (M == 4) { TDKS_WS_MODES(4, P_C64) }
    }
    return cudaErrorInvalidValue;
  }
  if (M == 2) { TDKS_WS_MODES(2, P_C128) }
  if (M == 4) { TDKS_WS_MODES(4, P_C128) }
#undef TDKS_WS_MODES
  return cudaErrorInvalidValue;
}

// Every mode, FD order, precision and boundary (finite box or periodic cell) of one shape
// (instantiated once per shape, in a translation unit of its own).
template <int SHAPE>
cudaError_t launch_ws_shape(int M, int prec, int mode, int bloch, const SweepMaps &maps, const SweepParams &p,
                            int grid, cudaStream_t s) {
  if constexpr (C64Shape<SHAPE>::ONLY) {
    if constexpr (SHAPE == 6) {
      if (prec == P_C128) {
        if (mode == MODE_LAST) return cudaErrorInvalidValue;
        const bool first = mode == MODE_FIRST;
        if (bloch && M == 2)
          return first ? launch_ws_t<SHAPE, 2, P_C128, MODE_FIRST, 1>(maps, p, grid, s)
                       : launch_ws_t<SHAPE, 2, P_C128, MODE_MID, 1>(maps, p, grid, s);
        if (bloch) return cudaErrorInvalidValue;
        if (M == 2)
          return first ? launch_ws_t<SHAPE, 2, P_C128, MODE_FIRST, 0>(maps, p, grid, s)
                       : launch_ws_t<SHAPE, 2, P_C128, MODE_MID, 0>(maps, p, grid, s);
        return first ? launch_ws_t<SHAPE, 4, P_C128, MODE_FIRST, 0>(maps, p, grid, s)
                     : launch_ws_t<SHAPE, 4, P_C128, MODE_MID, 0>(maps, p, grid, s);
      }
    }
    constexpr int P = C64Shape<SHAPE>::P;
    if (prec != P_C64) return cudaErrorInvalidValue;
#define TDKS_WS5_MODES(MM, BL)                                                                   \
  switch (mode) {                                                                                \
    case MODE_FIRST: return launch_ws_t<SHAPE, MM, P, MODE_FIRST, BL>(maps, p, grid, s);         \
    case MODE_MID: return launch_ws_t<SHAPE, MM, P, MODE_MID, BL>(maps, p, grid, s);             \
    case MODE_LAST:                                                                              \
      if constexpr (C64Shape<SHAPE>::LAST) return launch_ws_t<SHAPE, MM, P, MODE_LAST, BL>(maps, p, grid, s); \
  }                                                                                              \
  return cudaErrorInvalidValue;
    if constexpr (C64Shape<SHAPE>::CELL) {
      if (bloch && M == 2) { TDKS_WS5_MODES(2, 1) }
    }
    if (bloch) return cudaErrorInvalidValue;
    if (M == 2) { TDKS_WS5_MODES(2, 0) }
    if (M == 4) { TDKS_WS5_MODES(4, 0) }
#undef TDKS_WS5_MODES
    return cudaErrorInvalidValue;
  } else {
    return bloch ? launch_ws_bc<SHAPE, 1>(M, prec, mode, maps, p, grid, s)
                 : launch_ws_bc<SHAPE, 0>(M, prec, mode, maps, p, grid, s);
  }
}

}  // namespace tdks
