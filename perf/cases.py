"""What this library is timed on: calls a user makes through its public entry points, and the
values those calls return in 64 bits from plain torch.

A case is one system (or a batch of systems) and one kind of call:

* ``apply``: H applied once to a set of device vectors, as an eigensolver or a user's own
  integrator calls it (the smallest unit of work);
* ``steps``: a propagation of some configured steps of a molecule or a periodic cell, after
  which the program reads the records and the orbitals (into page-locked memory), and the
  photoelectron amplitudes or the heat current where it set them up;
* ``batch``: many uneven molecules advanced together.

Grids, orders, orbital counts, atoms, fields and step lengths are those of the named workloads
in ``inputs.py`` (tiny molecule, medium molecule, periodic cell, batched systems, the serving
trace's ranges), of ``bench.py``'s propagator comparison and of the tests' ragged grids.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1912_07921_gb300 import _lib
from paper_1912_07921_gb300 import inputs as I
from paper_1912_07921_gb300.system import Batch, System

R_C, R_CUT = 0.6, 2.0                  # projector width and support radius (bohr)
WELL_DEPTH, WELL_WIDTH = 2.0, 0.8      # local potential wells
AMP, OMEGA = {"length": 0.005, "velocity": 0.2}, {"length": 0.057, "velocity": 0.03}
PROPS = {"taylor4": 0, "cfm4": 1, "emr": 2}
XCS = {"lda": I.XC_LDA_X, "hartree": I.XC_LDA_X_HARTREE}
BATCH_EDGE, BATCH_ORB, BATCH_ATOMS = (32, 80), (4, 32), (0, 12)


def _case(name=None, **kw):
    """A case with every field present.  `ds` is the sub-step length."""
    c = dict(kind="steps", nx=24, ny=24, nz=24, h=0.25, order=8, bc="box", prec="c64", n_orb=8, n_k=1, n_atoms=4,
             projectors=True, xc="lda", field="length", prop="taylor4", ds=0.0125, substeps=1, steps=1, momenta=0,
             heat=False, tune=False, n_systems=1, layout_seed=0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: H once on the tiny molecule (an eigensolver's inner call on a toy system)
        _case("apply_tiny_c128", kind="apply", h=0.3, order=4, prec="c128", n_orb=4, n_atoms=2, projectors=False),
        # H once on a grid that fits no tile, with an orbital count that fills no whole batch
        _case("apply_ragged_c64", kind="apply", nx=53, ny=37, nz=45, n_orb=13, n_atoms=6),
        # H once on the medium molecule's grid: every orbital of a production system
        _case("apply_medium_c64", kind="apply", nx=96, ny=96, nz=96, n_orb=64, n_atoms=16),
        # the tiny molecule's propagation, ten steps: launches and host work per step
        _case("steps_tiny_c128", h=0.3, order=4, prec="c128", n_orb=4, n_atoms=2, projectors=False, ds=0.02, steps=10),
        # the flagship workload: the medium molecule in complex64, autotuned as the benchmark does
        _case("steps_medium_c64", nx=96, ny=96, nz=96, n_orb=64, n_atoms=16, substeps=4, steps=4, tune=True),
        # its complex128 path, with the orbitals one card of a state-parallel run would hold
        _case("steps_medium_c128", nx=96, ny=96, nz=96, n_orb=16, n_atoms=16, prec="c128", substeps=4, steps=1),
        # Bloch states of the periodic cell in the velocity gauge, eight of its k-points, autotuned
        _case("cell_c64", nx=64, ny=64, nz=64, h=10.2 / 64, order=4, bc="cell", n_orb=16, n_k=8, n_atoms=8,
              field="velocity", ds=0.04 / 6, substeps=6, steps=2, tune=True),
        # a small ragged cell in complex128 whose heat current is read after the step
        _case("cell_heat_c128", nx=30, ny=36, nz=32, h=0.25, order=4, bc="cell", prec="c128", n_orb=10, n_k=3,
              n_atoms=8, field="velocity", ds=0.0125, substeps=2, steps=1, heat=True),
        # uneven molecules advanced together (the many-systems workload), autotuned
        _case("batch_c64", kind="batch", order=4, ds=0.015, steps=10, n_systems=24, tune=True),
        # the order-four Magnus propagator on the molecule of the propagator comparison
        _case("cfm4_c128", nx=48, ny=48, nz=48, prec="c128", n_orb=16, n_atoms=6, prop="cfm4", substeps=4, steps=1),
        # exchange and Hartree potential in a ragged box, exponential midpoint rule
        _case("hartree_c64", nx=60, ny=64, nz=54, n_orb=24, n_atoms=6, xc="hartree", prop="emr", substeps=4, steps=1),
        # photoelectron amplitudes of a molecule (t-SURFF), a few hundred momenta
        _case("tsurff_c64", nx=64, ny=64, nz=64, n_orb=16, n_atoms=4, substeps=4, steps=2, momenta=400),
    ]


def _edges(rng, lo, hi):
    return {k: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for k in ("nx", "ny", "nz")}


def _orbitals(rng, hi):
    return int(round(math.exp(rng.uniform(math.log(4), math.log(hi)))))


def draw(rng):
    """One more case: a kind of call, then its sizes, spread over the logarithm of their range."""
    prec = rng.choice(["c64", "c64", "c128"])
    big, orb = (96, 64) if prec == "c64" else (72, 16)
    kind = rng.choice(["apply", "apply", "molecule", "molecule", "cell", "cell", "batch", "hartree", "tsurff"])
    order = rng.choice([4, 8])
    c = dict(prec=prec, order=order, layout_seed=rng.randrange(1000))
    if kind == "apply":
        cell = rng.random() < 0.4
        c.update(_edges(rng, 20, big if not cell else 64), kind="apply", n_orb=_orbitals(rng, orb), n_atoms=rng.randint(0, 12))
        if cell:
            c.update(order=4, bc="cell", n_k=rng.randint(1, 6), n_orb=_orbitals(rng, 16), n_atoms=8, field="velocity")
    elif kind == "molecule":
        c.update(_edges(rng, 20, big), n_orb=_orbitals(rng, orb), n_atoms=rng.randint(0, 16), substeps=rng.randint(1, 4),
                 steps=rng.randint(1, 2), prop=rng.choice(["taylor4", "taylor4", "cfm4", "emr"]), tune=rng.random() < 0.5)
    elif kind == "cell":
        c.update(_edges(rng, 20, 64), order=4, bc="cell", n_k=rng.randint(1, 8 if prec == "c64" else 3),
                 n_orb=_orbitals(rng, 16), n_atoms=8, field="velocity", substeps=rng.randint(1, 6),
                 heat=rng.random() < 0.3, tune=rng.random() < 0.5)
    elif kind == "batch":
        c.update(kind="batch", prec="c64", order=4, n_systems=rng.randint(4, 20), steps=rng.randint(1, 8), tune=True)
    elif kind == "hartree":
        even = {k: 2 * rng.randint(10, 32) for k in ("nx", "ny", "nz")}  # (cells: small prime factors only)
        if rng.random() < 0.4:
            c.update({k: rng.choice([24, 30, 32, 36, 40, 48, 50, 52, 56, 60, 64]) for k in even}, order=4, bc="cell",
                     n_k=rng.randint(1, 3), field="none", n_orb=_orbitals(rng, 12), n_atoms=8)
        else:
            c.update({k: v + rng.randint(0, 1) for k, v in even.items()}, n_orb=_orbitals(rng, 24), n_atoms=rng.randint(0, 6))
        c.update(xc="hartree", prop=rng.choice(["taylor4", "emr", "cfm4"]), substeps=rng.randint(1, 4))
    else:
        c.update(_edges(rng, 28, 64), n_orb=_orbitals(rng, 20), n_atoms=rng.randint(0, 4), substeps=rng.randint(1, 4),
                 steps=rng.randint(1, 2), momenta=rng.randint(40, 400))
    c["projectors"] = c.get("n_atoms", 0) > 0
    c["ds"] = 0.0125 if c.get("prop", "taylor4") == "taylor4" else 0.02
    c["ds"] = 0.0125 if order == 8 else c["ds"]
    return _case(**c)


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _members(case):
    """The systems of a case: itself, or the uneven molecules of a batch."""
    if case["kind"] != "batch":
        return [case]
    rng = I.SplitMix64(31 + case["layout_seed"])
    out = []
    for _ in range(case["n_systems"]):
        nx, ny, nz = (rng.randint(*BATCH_EDGE) for _ in range(3))
        n_orb, n_atoms = rng.randint(*BATCH_ORB), rng.randint(*BATCH_ATOMS)
        out.append(dict(case, nx=nx, ny=ny, nz=nz, n_orb=n_orb, n_atoms=n_atoms, projectors=n_atoms > 0))
    return out


def _axes(c, dev):
    n = (c["nx"], c["ny"], c["nz"])
    off = [(m - 1) / 2.0 if c["bc"] == "box" else 0.0 for m in n]
    return [(torch.arange(m, dtype=torch.float64, device=dev) - o) * c["h"] for m, o in zip(n, off)]


class _Inputs:
    """Atoms, wells, k-points, momenta (host) and orbitals (device, [k][z][y][x][orb])."""

    def __init__(self, c, seed, orbitals=True):
        dev = torch.device("cuda")
        rng = np.random.default_rng([seed, c["nx"], c["ny"], c["nz"], c["n_orb"]])
        n = np.array([c["nx"], c["ny"], c["nz"]])
        L = n * c["h"]
        cell = c["bc"] == "cell"
        if cell:  # diamond sites, the lattice shifted off the grid
            fcc = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
            frac = np.concatenate([fcc, fcc + 0.25])[: c["n_atoms"]] + rng.uniform(0.0, 0.1, 3)
            self.pos = frac * L
        else:     # anywhere in the inner half of the box
            half = (n - 1) * c["h"] / 2.0
            self.pos = rng.uniform(-0.5, 0.5, (c["n_atoms"], 3)) * half
        self.D = rng.uniform(-1.0, 1.0, (c["n_atoms"], 4))
        self.kpts = rng.uniform(-math.pi, math.pi, (c["n_k"], 3)) / L if cell else np.zeros((1, 3))
        self.kw = np.full(c["n_k"], 1.0 / c["n_k"])
        self.momenta = rng.normal(0.0, 0.6, (c["momenta"], 3))
        ax = _axes(c, dev)
        v = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=dev)
        for a in range(c["n_atoms"]):
            g = []
            for d in range(3):
                x = ax[d] - float(self.pos[a, d])
                x = x - L[d] * torch.round(x / L[d]) if cell else x
                g.append(torch.exp(-x ** 2 / (2.0 * WELL_WIDTH ** 2)))
            v -= WELL_DEPTH * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
        self.vloc = v
        if not orbitals:
            return
        # orthonormal wave packets: Gaussians of width 1 with random small momenta (periodic cells:
        # summed over the nearest images, times e^{ik.r})
        centre = rng.uniform(0.0, 1.0, (c["n_orb"], 3)) * L if cell else rng.uniform(-0.25, 0.25, (c["n_orb"], 3)) * (n - 1) * c["h"]
        mom = rng.normal(0.0, 0.7, (c["n_orb"], 3))
        mom = np.round(mom * L / (2 * math.pi)) * 2 * math.pi / L if cell else mom
        f = []
        for d in range(3):
            x = ax[d][:, None] - torch.tensor(centre[:, d], device=dev)[None, :]
            g = sum(torch.exp(-(x + s * float(L[d])) ** 2 / 2.0) for s in ((-1, 0, 1) if cell else (0,)))
            f.append(g * torch.exp(1j * ax[d][:, None] * torch.tensor(mom[:, d], device=dev)[None, :]))
        A = (f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :]).reshape(-1, c["n_orb"])
        w, V = torch.linalg.eigh((A.conj().T @ A) * c["h"] ** 3)
        A = A @ (V * torch.clamp(w, min=1e-8 * float(w[-1])).rsqrt()) @ V.conj().T
        psi = torch.empty((c["n_k"], A.shape[0], c["n_orb"]), dtype=torch.complex128, device=dev)
        for k in range(c["n_k"]):
            e = [torch.exp(1j * float(self.kpts[k, d]) * ax[d]) for d in range(3)]
            ph = (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]).reshape(-1, 1)
            psi[k] = A * ph if cell else A
        self.psi = psi.reshape(c["n_k"], c["nz"], c["ny"], c["nx"], c["n_orb"])


def _spec(c):
    gauge = {"none": I.GAUGE_NONE, "length": I.GAUGE_LENGTH, "velocity": I.GAUGE_VELOCITY}[c["field"]]
    return I.SystemSpec(nx=c["nx"], ny=c["ny"], nz=c["nz"], h=c["h"], fd_order=c["order"],
                        bc=I.BC_ZERO if c["bc"] == "box" else I.BC_BLOCH,
                        prec=I.PREC_C64 if c["prec"] == "c64" else I.PREC_C128, n_orb=c["n_orb"], n_k=c["n_k"],
                        n_atoms=c["n_atoms"], projectors=c["projectors"], r_c=R_C, r_cut=R_CUT, xc=XCS[c["xc"]],
                        gauge=gauge, amp=AMP.get(c["field"], 0.0), omega=OMEGA.get(c["field"], 0.0),
                        dt=c["ds"] * c["substeps"], substeps=c["substeps"])


def _momentum_box(c):
    """Grid planes of the t-SURFF surface: an eighth of the edge inside each face."""
    M = c["order"] // 2
    lo = [max(M, n // 8) for n in (c["nx"], c["ny"], c["nz"])]
    return [lo[0], c["nx"] - 1 - lo[0], lo[1], c["ny"] - 1 - lo[1], lo[2], c["nz"] - 1 - lo[2]]


def _system(c, seed, stream):
    inp = _Inputs(c, seed)
    host = torch.empty(inp.psi.shape, dtype=torch.complex128, pin_memory=True)
    host.copy_(inp.psi)
    s = System(_spec(c), I.Inputs(vloc=inp.vloc.cpu().numpy(), psi0=host.numpy(), pos=inp.pos, D=inp.D, kpts=inp.kpts,
                                  kw=inp.kw), stream=stream)
    return s, inp, host


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    parts = [_system(c, seed + i, stream) for i, c in enumerate(_members(case))]
    systems = [p[0] for p in parts]
    st = {"case": case, "systems": systems, "t": 0.0, "dt": case["ds"] * case["substeps"]}
    if case["kind"] == "apply":
        s, inp, _ = parts[0]
        bs, nb, eb, _ = s.layout()
        c = _members(case)[0]
        pad = torch.zeros((c["n_k"], c["nz"], c["ny"], c["nx"], nb * bs), dtype=torch.complex128, device="cuda")
        pad[..., : c["n_orb"]] = inp.psi
        x = pad.reshape(c["n_k"], c["nz"], c["ny"], c["nx"], nb, bs).permute(0, 4, 1, 2, 3, 5)
        st["x"] = x.to(torch.complex64 if eb == 8 else torch.complex128).contiguous()
        st["y"] = torch.empty_like(st["x"])
    else:
        # the page-locked buffer the orbitals are read into
        st["host"] = torch.empty(sum(p[2].numel() for p in parts), dtype=torch.complex128, pin_memory=True)
    if case["kind"] == "batch":
        for s in systems:
            s.set_clock(0.0, st["dt"], case["substeps"])
        st["batch"] = Batch(systems, stream=stream)
        if case["tune"]:
            st["batch"].autotune(3)
    else:
        s = systems[0]
        if case["prop"] != "taylor4":
            s.set_propagator(PROPS[case["prop"]])
        if case["tune"]:
            s.autotune(3)
        if case["momenta"]:
            s.set_tsurff(_momentum_box(case), parts[0][1].momenta)
    return st


def _read_orbitals(st):
    """Every system's orbitals, one after another, into the page-locked buffer."""
    at = st["host"].data_ptr()
    for s in st["systems"]:
        _lib.check(s.lib.tdks_get_orbitals(s.h, ctypes.c_void_p(at)))
        at += 16 * math.prod(s.shape)
    return st["host"]


def run(st):
    case, s = st["case"], st["systems"][0]
    if case["kind"] == "apply":
        s.apply_H(1.0, st["x"].data_ptr(), st["y"].data_ptr())
        return {"y": st["y"]}
    n = case["steps"]
    if case["kind"] == "batch":
        st["batch"].propagate(n)
        return {"records": np.stack([q.reductions(q.step_count() - n, n) for q in st["systems"]]), "psi": _read_orbitals(st)}
    s.propagate(st["t"], st["dt"], n, case["substeps"])
    st["t"] += n * st["dt"]
    out = {"records": s.reductions(s.step_count() - n, n), "psi": _read_orbitals(st)}
    if case["heat"]:
        out["heat"] = s.heat_current(st["t"])
    if case["momenta"]:
        out["b"] = s.tsurff()[0]
    return out


def work(case):
    """Bytes and operations of one pass.

    A sub-step is four applications of H whose inputs and outputs are whole arrays (each needs
    the projector products and the density of the whole one before it): the terms written once
    and read once each, the series added to the state in the last, 13 values of 8 bytes moved per
    orbital value in complex64 (its state is two such numbers) and 11 of 16 in complex128.  An
    application of H is 6 M + 1 products and as many sums on each part of the value.
    """
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _members(case):
        N, M = c["nx"] * c["ny"] * c["nz"], c["order"] // 2
        values, eb = float(N) * c["n_orb"] * c["n_k"], 8 if c["prec"] == "c64" else 16
        apply_flops = values * 4 * (6 * M + 1)
        if c["kind"] == "apply":
            total["bytes"] += 2 * values * eb + 8.0 * N
            total["flops"] += apply_flops
            continue
        exps = c["steps"] * c["substeps"] * {"taylor4": 1, "emr": 1, "cfm4": 2}[c["prop"]]
        total["bytes"] += exps * (values * (104 if eb == 8 else 176) + 16.0 * N) + 16 * values
        total["flops"] += exps * 4 * apply_flops
        if c["xc"] == "hartree":  # forward and inverse transforms of the padded density
            P = N * (8 if c["bc"] == "box" else 1)
            total["flops"] += c["steps"] * c["substeps"] * 2 * 2.5 * P * math.log2(P)
            total["bytes"] += c["steps"] * c["substeps"] * 16.0 * N
        if c["momenta"]:
            b = _momentum_box(c)
            ex, ey, ez = (b[2 * a + 1] - b[2 * a] + 1 for a in range(3))
            total["flops"] += (c["steps"] + 1) * 2.0 * (ex * ey + ey * ez + ex * ez) * c["n_orb"] * c["momenta"] * 12
    return total


# ---------------------------------------------------------------------------------------------
# The same calls in 64 bits: plain torch on [k][orb][z][y][x]
# ---------------------------------------------------------------------------------------------

def _weights(M):
    """Central weights of the first and second derivative of order 2M (closed form)."""
    g, c = [0.0], [0.0]
    for m in range(1, M + 1):
        r = (-1.0) ** (m + 1) * math.factorial(M) ** 2 / (math.factorial(M - m) * math.factorial(M + m))
        g.append(r / m)
        c.append(2.0 * r / m ** 2)
    c[0] = -2.0 * sum(c[1:])
    return g, c


class _Plain:
    """One system of a case: its Hamiltonian, propagators and observables."""

    def __init__(self, c, seed):
        self.c, self.h, self.M = c, c["h"], c["order"] // 2
        inp = _Inputs(c, seed)
        self.inp, self.cell = inp, c["bc"] == "cell"
        self.psi = inp.psi.permute(0, 4, 1, 2, 3).contiguous()
        self.N = c["nx"] * c["ny"] * c["nz"]
        self.L = [c["nx"] * self.h, c["ny"] * self.h, c["nz"] * self.h]
        self.k = inp.kpts
        self.w = [2.0 * float(x) for x in inp.kw]  # weight times occupation
        x, y, z = _axes(c, "cuda")
        self.r = [x[None, None, :], y[None, :, None], z[:, None, None]]
        self.g, self.lap = _weights(self.M)
        self.spheres = [self._sphere(a) for a in range(c["n_atoms"])] if c["projectors"] else []

    def _sphere(self, a):
        """Indices, offsets d, lattice translations T and beta of one atom's points."""
        n, R, ii = (self.c["nx"], self.c["ny"], self.c["nz"]), self.inp.pos[a], []
        for d in range(3):
            o = 0.0 if self.cell else (n[d] - 1) / 2.0
            lo, hi = math.floor((R[d] - R_CUT) / self.h + o) - 1, math.ceil((R[d] + R_CUT) / self.h + o) + 1
            lo, hi = (lo, hi) if self.cell else (max(lo, 0), min(hi, n[d] - 1))
            ii.append(torch.arange(lo, hi + 1, device="cuda"))
        ix, iy, iz = (t.reshape(-1) for t in torch.meshgrid(*ii, indexing="ij"))
        idx = [ix, iy, iz]
        d = [(idx[q].double() - (0.0 if self.cell else (n[q] - 1) / 2.0)) * self.h - float(R[q]) for q in range(3)]
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        keep = r2 <= R_CUT ** 2
        wrap = [torch.div(t, m, rounding_mode="floor") for t, m in zip(idx, n)]
        at = ((idx[2] - wrap[2] * n[2]) * n[1] + idx[1] - wrap[1] * n[1]) * n[0] + idx[0] - wrap[0] * n[0]
        g = torch.exp(-r2 / (2.0 * R_C ** 2))
        d = torch.stack(d)
        return at[keep], d[:, keep], torch.stack([wrap[q].double() * self.L[q] for q in range(3)])[:, keep], \
            torch.stack([g, d[0] * g, d[1] * g, d[2] * g])[:, keep]

    def field(self, t):
        """(E, A, recorded value): along z, no envelope."""
        f = AMP.get(self.c["field"], 0.0) * math.sin(OMEGA.get(self.c["field"], 0.0) * t)
        return (f, 0.0, f) if self.c["field"] == "length" else (0.0, f, f)

    def shift(self, u, axis, s):
        """u at offset s along an axis (x, y, z = 0, 1, 2): zero outside a box, Bloch images in a cell."""
        dim = u.dim() - 1 - axis
        n = u.shape[dim]
        if not self.cell:
            out = torch.zeros_like(u)
            if abs(s) < n:
                out.narrow(dim, max(0, -s), n - abs(s)).copy_(u.narrow(dim, max(0, s), n - abs(s)))
            return out
        i = torch.arange(n, device="cuda") + s
        w = torch.div(i, n, rounding_mode="floor")
        kk = torch.tensor(self.k[:, axis], device="cuda")
        ph = torch.exp(1j * self.L[axis] * kk[:, None] * w[None, :])
        sh = [len(self.k)] + [1] * (u.dim() - 1)
        sh[dim] = n
        return u.index_select(dim, i - w * n) * ph.reshape(sh)

    def grad(self, u, axis):
        return sum(self.g[m] / self.h * (self.shift(u, axis, m) - self.shift(u, axis, -m)) for m in range(1, self.M + 1))

    def laplacian(self, u):
        acc = (3.0 * self.lap[0] / self.h ** 2) * u
        for a in range(3):
            for m in range(1, self.M + 1):
                acc.add_(self.shift(u, a, m), alpha=self.lap[m] / self.h ** 2)
                acc.add_(self.shift(u, a, -m), alpha=self.lap[m] / self.h ** 2)
        return acc

    def density(self, u):
        return sum(w * (u[k].abs() ** 2).sum(0) for k, w in enumerate(self.w))

    def hxc(self, n):
        """(v_x + v_H, v_H) of a density."""
        v, vh = -(3.0 * n / math.pi) ** (1.0 / 3.0), None
        if self.c["xc"] == "hartree":
            sz = n.shape
            if self.cell:
                G = [2.0 * math.pi * torch.fft.fftfreq(m, d=self.h, dtype=torch.float64, device="cuda") for m in sz]
                G2 = G[0][:, None, None] ** 2 + G[1][None, :, None] ** 2 + G[2][None, None, :] ** 2
                G2[0, 0, 0] = 1.0
                f = torch.fft.fftn(n) * 4.0 * math.pi / G2
                f[0, 0, 0] = 0.0
                vh = torch.fft.ifftn(f).real
            else:
                o = [torch.cat([torch.arange(m, device="cuda"), torch.arange(-m, 0, device="cuda")]).double() for m in sz]
                d = (o[0][:, None, None] ** 2 + o[1][None, :, None] ** 2 + o[2][None, None, :] ** 2).sqrt()
                K = 1.0 / (self.h * d)
                K[0, 0, 0] = (3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi) / self.h
                s2 = [2 * m for m in sz]
                vh = self.h ** 3 * torch.fft.irfftn(torch.fft.rfftn(K) * torch.fft.rfftn(n, s=s2), s=s2)[: sz[0], : sz[1], : sz[2]]
            v = v + vh
        return v, vh

    def potential(self, vhxc, E, A):
        return self.inp.vloc + vhxc + (E * self.r[2] if not self.cell else 0.0) + 0.5 * A * A

    def phases(self, sp, k, A):
        _, d, T, _ = sp
        kk = torch.tensor(self.k[k], device="cuda")
        return torch.exp(1j * (kk @ T + A * d[2]))

    def apply(self, u, V, A):
        out = -0.5 * self.laplacian(u)
        out += V * u
        if A != 0.0:
            out += -1j * A * self.grad(u, 2)
        flat, of = u.reshape(u.shape[0], u.shape[1], -1), out.reshape(u.shape[0], u.shape[1], -1)
        for a, sp in enumerate(self.spheres):
            at, _, _, beta = sp
            D = torch.tensor(self.inp.D[a], device="cuda") * self.h ** 3
            for k in range(u.shape[0]):
                b = beta * self.phases(sp, k, A)
                q = (flat[k][:, at] @ b.T) * D
                of[k].index_add_(1, at, q @ b.conj())
        return out

    def exponential(self, u, V, A, tau):
        t, acc = u, u.clone()
        for j in range(1, 5):
            t = self.apply(t, V, A) * (-1j * tau / j)
            acc += t
        return acc

    def record(self, u, t, ds):
        n = self.density(u)
        (v, vh), (E, A, f) = self.hxc(n), self.field(t + 0.5 * ds)
        V, h3 = self.potential(v, E, A), self.h ** 3
        vx = v if vh is None else v - vh
        ex = 0.75 * float((n * vx).sum()) * h3
        hu = self.apply(u, V, A)
        e = sum(w * float((u[k].conj() * hu[k]).sum().real) for k, w in enumerate(self.w)) * h3
        e += -float((n * (vx if vh is None else vx + 0.5 * vh)).sum()) * h3 + ex
        nint = float(n.sum()) * h3
        if not self.cell:
            o = [float((n * self.r[a]).sum()) * h3 for a in range(3)]
        else:
            om = self.N * h3
            o = [sum(w * float((u[k].conj() * self.grad(u, a)[k]).sum().imag) for k, w in enumerate(self.w)) * h3
                 + (A * nint if a == 2 else 0.0) for a in range(3)]
            flat = u.reshape(u.shape[0], u.shape[1], -1)
            for ia, sp in enumerate(self.spheres):
                at, d, _, beta = sp
                D = torch.tensor(self.inp.D[ia], device="cuda")
                for k, w in enumerate(self.w):
                    b = beta * self.phases(sp, k, A)
                    p = flat[k][:, at] @ b.T * h3
                    for a in range(3):
                        q = flat[k][:, at] @ (b * d[a]).T * h3
                        o[a] += w * float((-2.0 * D * (p.conj() * q).imag).sum())
            o = [-x / om for x in o]
        return [t, nint / 2.0, e, ex, *o, f]

    def propagate(self):
        c, u, hist, recs = self.c, self.psi, [], []
        ds, r3 = c["ds"], math.sqrt(3.0)
        a1, a2, t1, t2 = (3 - 2 * r3) / 12, (3 + 2 * r3) / 12, 0.5 - r3 / 6, 0.5 + r3 / 6
        factors = {"cfm4": [(0.5, [(t1, 2 * a2), (t2, 2 * a1)]), (0.5, [(t1, 2 * a1), (t2, 2 * a2)])],
                   "emr": [(1.0, [(0.5, 1.0)])]}.get(c["prop"])
        if c["momenta"]:
            self.begin_flux()
        for st in range(c["steps"]):
            t = st * ds * c["substeps"]
            if c["momenta"]:
                self.add_flux(u, t, ds * c["substeps"] * (0.5 if st == 0 else 1.0))
            recs.append(self.record(u, t, ds))
            for j in range(c["substeps"]):
                tj = t + j * ds
                v = self.hxc(self.density(u))[0]
                if factors is None:
                    E, A, _ = self.field(tj + 0.5 * ds)
                    u = self.exponential(u, self.potential(v, E, A), A, ds)
                    continue
                hist = [v] + hist[:3]
                for frac, nodes in factors:
                    E = sum(w * self.field(tj + th * ds)[0] for th, w in nodes)
                    ve = sum(sum(w * math.prod((th + i) / (i - q) for i in range(len(hist)) if i != q) for th, w in nodes) * hist[q]
                             for q in range(len(hist)))
                    u = self.exponential(u, self.potential(ve, E, 0.0), 0.0, frac * ds)
        if c["momenta"]:
            self.add_flux(u, c["steps"] * ds * c["substeps"], 0.5 * ds * c["substeps"])
        self.u = u
        return np.array(recs)

    # t-SURFF: flux of the state through the box surface for every momentum
    def begin_flux(self):
        self.b, self.volkov, self.t_volkov = 0.0, np.zeros(3), 0.0  # a, alpha, beta along z

    def _advance(self, t):
        """a = -int E, alpha = int a, beta = int a^2 by the classical Runge-Kutta method, one step per call."""
        dt, t0, y = t - self.t_volkov, self.t_volkov, self.volkov
        f = lambda s, q: np.array([-self.field(s)[0], q[0], q[0] ** 2])  # noqa: E731
        if dt > 0.0:
            k1 = f(t0, y)
            k2 = f(t0 + dt / 2, y + dt / 2 * k1)
            k3 = f(t0 + dt / 2, y + dt / 2 * k2)
            k4 = f(t0 + dt, y + dt * k3)
            self.volkov, self.t_volkov = y + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4), t

    def add_flux(self, u, t, weight):
        self._advance(t)
        a, alpha, beta = self.volkov
        p = torch.tensor(self.inp.momenta, device="cuda")
        kp = p.clone()
        kp[:, 2] += a
        box, x, total = _momentum_box(self.c), [r.reshape(-1) for r in self.r], 0.0
        for ax in range(3):
            ua, va = [q for q in range(3) if q != ax]
            g = self.grad(u, ax)[0]
            for side in (0, 1):
                pl, sl, ws, ph = box[2 * ax + side], [None] * 3, {}, 1.0
                for q in (ua, va):
                    sl[q] = slice(box[2 * q], box[2 * q + 1] + 1)
                    ws[q] = torch.full((box[2 * q + 1] + 1 - box[2 * q],), self.h, dtype=torch.float64, device="cuda")
                    ws[q][0] *= 0.5
                    ws[q][-1] *= 0.5
                sl[ax] = slice(pl, pl + 1)
                cut = (slice(None), sl[2], sl[1], sl[0])
                phi, dphi = u[0][cut], g[cut]
                e = [torch.exp(-1j * kp[:, q, None] * x[q][sl[q]][None, :]) * (ws[q] if q != ax else 1.0) for q in range(3)]
                for_ = lambda f: torch.einsum("ozyx,pz,py,px->op", f, e[2], e[1], e[0])  # noqa: E731
                total = total + (1.0 if side else -1.0) * (kp[None, :, ax] * for_(phi) - 1j * for_(dphi))
        phase = 0.5 * ((p ** 2).sum(1) * t + 2.0 * p[:, 2] * alpha + beta)
        self.b = self.b + 0.5 * weight * (2.0 * math.pi) ** -1.5 * torch.exp(1j * phase)[None, :] * total

    def heat_current(self, t):
        """Cell average of the kinetic heat current, covariant differences composed."""
        A = self.field(t)[1]
        u = self.u
        D = lambda v, a: self.grad(v, a) + (1j * A * v if a == 2 else 0.0)  # noqa: E731
        lap = self.laplacian(u) + 2j * A * self.grad(u, 2) - A * A * u
        d2 = sum(D(D(u, a), a) for a in range(3))
        out = []
        for a in range(3):
            d = D(u, a)
            f = (d2.conj() * d).imag - (d.conj() * lap).imag
            out.append(sum(w * float(f[k].sum()) for k, w in enumerate(self.w)) / (4.0 * self.N))
        return np.array(out)

    def host_layout(self):
        return self.u.permute(0, 2, 3, 4, 1)


def exact(case, seed):
    parts = [_Plain(c, seed + i) for i, c in enumerate(_members(case))]
    if case["kind"] == "apply":
        q = parts[0]
        E, A, _ = q.field(1.0)
        y = q.apply(q.psi, q.potential(q.hxc(q.density(q.psi))[0], E, A), A)
        bs = 8 if case["prec"] == "c64" else 4
        nb = -(-case["n_orb"] // bs)
        pad = torch.zeros((case["n_k"], nb * bs, *y.shape[2:]), dtype=torch.complex128, device="cuda")
        pad[:, : case["n_orb"]] = y
        return {"y": pad.reshape(case["n_k"], nb, bs, *y.shape[2:]).permute(0, 1, 3, 4, 5, 2).contiguous()}
    recs = [q.propagate() for q in parts]
    out = {"records": np.stack(recs) if case["kind"] == "batch" else recs[0],
           "psi": torch.cat([q.host_layout().reshape(-1) for q in parts])}
    if case["heat"]:
        out["heat"] = parts[0].heat_current(case["steps"] * case["ds"] * case["substeps"])
    if case["momenta"]:
        out["b"] = parts[0].b.cpu().numpy()
    return out
