"""What is measured: the calls that a program using this library makes, over their real range.

Kinds of case (the `kind` entry):
  md           a trajectory: System.step, then the state read back, as a driver does that writes a
               frame every few steps.  512 atoms (the smallest periodic box of the tests) to the
               884,736-atom benchmark cube, cubes and uneven boxes, whole crystals and ragged ones
               (`drop` atoms removed), both precisions, and the three spin updates: "pc" (the
               predictor-corrector), "midpoint" (the self-consistent iteration, stopped by its
               tolerance) and "longitudinal" (variable moment lengths).
  film         the production protocol: a stripe with free edges and surfaces, random spins, a
               field that steps along x, and the film's texture read after every stretch of steps.
  batch        a temperature and field sweep: replicas of uneven size in one batched call.
  point        a single-point evaluation: a new configuration in, energy, forces, fields and virial
               out (an outer optimiser or sampler that owns the dynamics).
  descriptors  the descriptors and atomic energies of a configuration (fitting, similarity maps).
  plugin       the no-allocation entry point: device arrays of a small system in, descriptors and
               energies out (a host engine's plugin).

Trajectories go on from pass to pass, as a simulation does.  `exact` is a plain float64 torch
statement of the method: Chebyshev carrier, Legendre channels by Cartesian moments, network,
derivatives by autograd, and the integrator with its counter-based noise.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_14073_gb300 import nep_params, spinlat, workloads

SKIN = 1.0
GAMMA, LAMBDA = 0.01, 0.1          # the library's default dampings
DT = 1.0                           # fs
ALPHA, LANDAU = 0.1, ((-0.2, 0.08), (-0.2, 0.08))   # the benchmark's longitudinal settings
MID_CAP, MID_TOL = 8, 1e-6         # the benchmark's midpoint settings
TEXTURE_CELL = 4.7                 # A, the crystal's lattice constant


def listed():
    return [
        # a plugin's call: one cell block of a host engine, every step of that engine
        dict(name="plugin_1000", kind="plugin", nx=5, ny=5, nz=5, drop=0),
        # the smallest box, validation in FP64, where launches and latency are everything
        dict(name="md_512_fp64", kind="md", mode="pc", precision="fp64", nx=4, ny=4, nz=4, drop=0,
             spins="random", T=300.0, B=0.0, steps=25),
        # a small ragged sample in production precision
        dict(name="md_1725_mixed", kind="md", mode="pc", precision="mixed", nx=6, ny=6, nz=6, drop=3,
             spins="random", T=300.0, B=0.2, steps=25),
        # the smallest request of the serving mix
        dict(name="md_13824_mixed", kind="md", mode="pc", precision="mixed", nx=12, ny=12, nz=12, drop=0,
             spins="canted", T=150.0, B=0.1, steps=25),
        # an ordinary production box
        dict(name="md_110592_mixed", kind="md", mode="pc", precision="mixed", nx=24, ny=24, nz=24, drop=0,
             spins="canted", T=300.0, B=0.0, steps=20),
        # the benchmark's cube
        dict(name="md_884736_mixed", kind="md", mode="pc", precision="mixed", nx=48, ny=48, nz=48, drop=0,
             spins="canted", T=300.0, B=0.0, steps=20),
        # a reference trajectory in FP64
        dict(name="md_32768_fp64", kind="md", mode="pc", precision="fp64", nx=16, ny=16, nz=16, drop=0,
             spins="canted", T=300.0, B=0.0, steps=10),
        # the stripe protocol, with its texture diagnostics
        dict(name="film_49152_mixed", kind="film", precision="mixed", nx=64, ny=24, nz=4, drop=0, T=160.0,
             steps=20),
        # a sweep over temperatures and fields in one batch, 4,096 to 65,536 atoms each
        dict(name="batch_8_mixed", kind="batch", precision="mixed", replicas=8, least=4096, most=65536, steps=20),
        # the self-consistent spin update
        dict(name="midpoint_13824_mixed", kind="md", mode="midpoint", precision="mixed", nx=12, ny=12, nz=12,
             drop=0, spins="canted", T=300.0, B=0.0, steps=10),
        # an outer sampler's energy call on a ragged sample, FP64 with the virial
        dict(name="point_4093_fp64", kind="point", precision="fp64", nx=8, ny=8, nz=8, drop=3),
        # descriptors of one frame of a fitting set
        dict(name="descriptors_32768_mixed", kind="descriptors", precision="mixed", nx=16, ny=16, nz=16, drop=0),
    ]


def _box(rng, least, most):
    """Cells per side of a box of about `atoms` atoms, log-uniform in [least, most]; sides uneven."""
    atoms = math.exp(rng.uniform(math.log(least), math.log(most)))
    side = (atoms / 8.0) ** (1.0 / 3.0)
    nx = max(3, round(side * math.exp(rng.uniform(-0.3, 0.3))))
    ny = max(3, round(side * math.exp(rng.uniform(-0.3, 0.3))))
    nz = max(3, math.floor(atoms / (8.0 * nx * ny)))
    return dict(nx=nx, ny=ny, nz=nz, drop=rng.choice([0, 0, rng.randrange(1, 30)]))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "md", "film", "batch", "point", "point", "descriptors", "plugin"])
    if kind == "plugin":
        return dict(kind=kind, **_box(rng, 216, 2000))
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if kind == "film":
        return dict(kind=kind, precision=precision, nx=rng.randrange(16, 80 if precision == "mixed" else 32),
                    ny=rng.randrange(8, 32), nz=rng.randrange(2, 7), drop=rng.choice([0, rng.randrange(1, 30)]),
                    T=round(rng.uniform(50.0, 300.0), 1), steps=rng.randrange(5, 30 if precision == "mixed" else 10))
    if kind == "batch":
        top = 100000 if precision == "mixed" else 16384
        return dict(kind=kind, precision=precision, replicas=rng.randrange(2, 13), least=512,
                    most=rng.randrange(4096, top), steps=rng.randrange(5, 30 if precision == "mixed" else 10))
    if kind in ("point", "descriptors"):
        return dict(kind=kind, precision=precision, **_box(rng, 512, 250000 if precision == "mixed" else 60000))
    mode = rng.choice(["pc", "pc", "pc", "midpoint", "longitudinal"])
    top = {"pc": 400000, "longitudinal": 400000, "midpoint": 60000}[mode]
    if precision == "fp64":
        top = 40000 if mode != "midpoint" else 8000
    box = _box(rng, 512, top)
    n = 8 * box["nx"] * box["ny"] * box["nz"]
    work = {"mixed": 4.0e6, "fp64": 3.0e5}[precision] / (1 if mode != "midpoint" else 6)
    return dict(kind="md", mode=mode, precision=precision, spins=rng.choice(["random", "canted"]),
                T=round(rng.uniform(50.0, 320.0), 1), B=rng.choice([0.0, round(rng.uniform(0.0, 0.5), 3)]),
                steps=max(3, min(25, int(work / n))), **box)


# ------------------------------------------------------------------ inputs
def _inputs(nx, ny, nz, drop, spins, T, seed, periodic=(1, 1, 1), vacuum=8.0):
    """A jittered B20 crystal with Maxwell-Boltzmann velocities; free axes get a vacuum on both sides."""
    rng = np.random.Generator(np.random.PCG64([seed, nx, ny, nz]))
    pos, species, box = workloads.b20_lattice(nx, ny, nz)
    pos = pos + rng.normal(0.0, 0.02, size=pos.shape)
    for a in range(3):
        if not periodic[a]:
            pos[:, a] += vacuum
            box[a] += 2.0 * vacuum
    pos = workloads.wrap(pos, box, periodic)
    n = pos.shape[0]
    if spins == "random":
        s = workloads.random_unit_vectors(rng, n)
    else:   # ferromagnetic along z, canted 5 degrees
        phi, th = rng.uniform(0.0, 2.0 * math.pi, size=n), math.radians(5.0)
        s = np.stack([math.sin(th) * np.cos(phi), math.sin(th) * np.sin(phi), np.full(n, math.cos(th))], axis=1)
    vel = workloads.maxwell_boltzmann(rng, species, T)
    if drop:
        keep = np.ones(n, dtype=bool)
        keep[rng.choice(n, drop, replace=False)] = False
        pos, s, vel, species = pos[keep], s[keep], vel[keep], species[keep]
    return dict(positions=pos, spins=s, velocities=vel, species=species, box=box,
                periodic=np.asarray(periodic, dtype=np.int32))


def _stepped_field(inp):
    """B_z of 0, 0.05, 0.1 and 0.15 T in four equal segments along x."""
    k = np.minimum((inp["positions"][:, 0] / inp["box"][0] * 4.0).astype(int), 3)
    B = np.zeros_like(inp["positions"])
    B[:, 2] = 0.05 * k
    return B


def _replicas(case, seed):
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    shape = np.random.Generator(np.random.PCG64([case["replicas"], case["least"], case["most"]]))
    n = np.exp(shape.uniform(math.log(case["least"]), math.log(case["most"]), size=case["replicas"]))
    cells = np.maximum(np.rint(np.cbrt(n / 8.0)).astype(int), 3)
    steps = np.maximum(1, np.rint(case["steps"] * shape.uniform(0.5, 1.0, size=case["replicas"])).astype(int))
    steps[0] = case["steps"]
    T, Bz = rng.uniform(100.0, 300.0, size=case["replicas"]), rng.uniform(0.0, 0.5, size=case["replicas"])
    return [dict(inp=_inputs(int(c), int(c), int(c), 0, "canted", float(t), seed * 64 + k), steps=int(s), T=float(t),
                 B=(0.0, 0.0, float(b)), seed=(seed * 64 + k) & 0xFFFFFFFF)
            for k, (c, s, t, b) in enumerate(zip(cells, steps, T, Bz))]


def _prec(case):
    return spinlat.SL_PREC_MIXED if case["precision"] == "mixed" else spinlat.SL_PREC_FP64


def _system(inp, params, **kw):
    return spinlat.System(inp["positions"], inp["spins"], inp["box"], inp["periodic"], inp["species"], params,
                          inp["velocities"], skin=SKIN, gamma=GAMMA, lam=LAMBDA, **kw)


def _md_inputs(case, seed):
    return _inputs(case["nx"], case["ny"], case["nz"], case["drop"], case["spins"], case["T"], seed)


def _film_inputs(case, seed):
    return _inputs(case["nx"], case["ny"], case["nz"], case["drop"], "random", case["T"], seed, periodic=(1, 0, 0))


def _point_inputs(case, seed):
    return _inputs(case["nx"], case["ny"], case["nz"], case["drop"], "random", 300.0, seed)


def prepare(case, seed):
    params = nep_params.load()
    kind = case["kind"]
    st = dict(case=case)
    if kind == "md":
        kw = dict(midpoint_iters=MID_CAP, midpoint_tol=MID_TOL) if case["mode"] == "midpoint" else {}
        st["sys"] = _system(_md_inputs(case, seed), params, precision=_prec(case), seed=seed, **kw)
        if case["mode"] == "longitudinal":
            st["sys"].set_longitudinal(True, ALPHA, LANDAU)
    elif kind == "film":
        inp = _film_inputs(case, seed)
        st["sys"] = _system(inp, params, precision=_prec(case), seed=seed)
        st["sys"].set_atom_fields(_stepped_field(inp))
    elif kind == "batch":
        reps = _replicas(case, seed)
        st["systems"] = [_system(r["inp"], params, precision=_prec(case), seed=r["seed"]) for r in reps]
        st["batch"] = spinlat.Batch(st["systems"])
        st["args"] = ([r["steps"] for r in reps], DT, [r["T"] for r in reps], [r["B"] for r in reps])
    elif kind in ("point", "descriptors"):
        st["inp"] = _point_inputs(case, seed)
        st["sys"] = _system(st["inp"], params, precision=_prec(case), seed=seed)
    else:
        inp = _point_inputs(case, seed)
        n = inp["positions"].shape[0]
        pad = lambda a: torch.tensor(np.concatenate([a, np.zeros((n, 1))], axis=1), device="cuda")  # noqa: E731
        st.update(inp=inp, params=params, n=n, pos=pad(inp["positions"]), spin=pad(inp["spins"]),
                  species=torch.tensor(inp["species"], dtype=torch.int32, device="cuda"),
                  q=torch.zeros(n, 66, dtype=torch.float64, device="cuda"),
                  e=torch.zeros(n, dtype=torch.float64, device="cuda"))
    return st


_STATE = ("positions", "velocities", "spins", "forces", "fields")


def _state(system):
    s = system.get_state()
    return {k: s[k] for k in _STATE}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "md":
        state["sys"].step(case["steps"], DT, case["T"], (0.0, 0.0, case["B"]))
        return _state(state["sys"])
    if kind == "film":
        state["sys"].step(case["steps"], DT, case["T"])
        m, charge = state["sys"].texture(2, TEXTURE_CELL)
        return dict(_state(state["sys"]), m=m, charge=charge)
    if kind == "batch":
        state["batch"].step(*state["args"])
        return [_state(s) for s in state["systems"]]
    if kind == "point":
        inp = state["inp"]
        state["sys"].set_state(inp["positions"], inp["velocities"], inp["spins"])
        return state["sys"].energy_forces_fields()
    if kind == "descriptors":
        q, e = state["sys"].get_descriptors()
        return dict(q=q, e=e)
    inp = state["inp"]
    spinlat.sl_descriptors_energies_noalloc(
        state["pos"].data_ptr(), state["spin"].data_ptr(), state["species"].data_ptr(), state["n"], inp["box"],
        inp["periodic"], state["params"], state["q"].data_ptr(), state["e"].data_ptr(),
        torch.cuda.current_stream().cuda_stream)
    return dict(q=state["q"], e=state["e"])


# ------------------------------------------------------------------ work
# Counted operations of the method (a multiply-add is 2) at the crystal's neighbour numbers: per
# atom 69.7 neighbours inside 6 A and 20.7 inside 4 A.
N_R, N_A = 69.7, 20.7
_FORWARD = 880 + 680 + 166 * N_R + 664 * N_A
_NETWORK = 8166
_BACKWARD = 814 + 480 + 393 * N_R + 1668 * N_A + 6 * N_R


def _atoms(case):
    return 8 * case["nx"] * case["ny"] * case["nz"] - case["drop"]


def work(case):
    kind = case["kind"]
    step = _FORWARD + _NETWORK + _BACKWARD
    if kind == "md":
        evaluations = case["steps"] * (4 if case["mode"] == "midpoint" else 1)
        return dict(bytes=_atoms(case) * 24.0 * (2 * len(_STATE)), flops=_atoms(case) * step * evaluations)
    if kind == "film":
        return dict(bytes=_atoms(case) * 24.0 * (2 * len(_STATE) + 1), flops=_atoms(case) * step * case["steps"])
    if kind == "batch":
        reps = _replicas(case, 0)
        n = [r["inp"]["positions"].shape[0] for r in reps]
        return dict(bytes=sum(n) * 24.0 * (2 * len(_STATE)),
                    flops=sum(a * r["steps"] for a, r in zip(n, reps)) * step)
    n = _atoms(case)
    if kind == "point":
        return dict(bytes=n * 24.0 * 5, flops=n * step)
    return dict(bytes=n * (2 * 24 + 4 + 67 * 8.0), flops=n * (_FORWARD + _NETWORK / 2))


def tolerance(case):
    """About four times what a last-bit change of the positions makes of the outputs (measured over
    listed and drawn cases, on the first two passes).  Under this potential the dynamics is chaotic:
    such a change stays at rounding level for some 50 steps and then grows fast, so a pass takes
    fewer than 30 of them."""
    if case["kind"] == "plugin":
        return {"rel": 1e-13, "max": 1e-11}
    if case["precision"] == "fp64":
        return {"rel": 1e-12, "max": 2e-11}
    return {"rel": 1e-4, "max": 5e-3}


# ------------------------------------------------------------------ the method in float64
KB, HBAR, MUB, ACC = 8.617333262e-5, 0.6582119569, 5.7883818060e-5, 9.6485332e-3

# unique monomials x^a y^b z^c of degrees 0..4 with their multinomial weights l!/(a! b! c!):
# sum over monomials of weight * M_abc^2 is the squared norm of the full moment tensor
_MONO = [(a, b, d - a - b) for d in range(5) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]
_MONO_W = [math.factorial(sum(m)) / math.prod(math.factorial(k) for k in m) for m in _MONO]
_MONO_D = [sum(m) for m in _MONO]


class _Model:
    def __init__(self, dev):
        p = nep_params.load()
        t = lambda k: torch.tensor(np.asarray(p[k], dtype=np.float64), device=dev)  # noqa: E731
        self.c, self.scal = t("coeffs").reshape(2, 2, 6, 5, 9), t("q_scaler").reshape(66)
        self.w0, self.b0, self.w1, self.b1 = t("w0").reshape(30, 66), t("b0"), t("w1"), float(p["b1"])
        self.rc, self.ra = float(p["rc_rad"]), float(p["rc_ang"])
        self.mass, self.moment = t("mass_amu"), t("moment_muB")


def _basis(r, rc):
    fc = 0.5 * (1.0 + torch.cos(math.pi * r / rc))
    x = 2.0 * (r / rc - 1.0) ** 2 - 1.0
    T = [torch.ones_like(x), x]
    for _ in range(7):
        T.append(2.0 * x * T[-1] - T[-2])
    return 0.5 * (torch.stack(T, dim=1) + 1.0) * fc[:, None]


def _min_image(d, L, per):
    return d - per * L * torch.round(d / L)


class _Reference:
    """Energy, forces, fields, virial and descriptors of one system, and its trajectory."""

    def __init__(self, inp, dev="cuda"):
        self.dev = dev
        t = lambda a, k=torch.float64: torch.tensor(np.ascontiguousarray(a), dtype=k, device=dev)  # noqa: E731
        self.m = _Model(dev)
        self.L, self.per = t(inp["box"]), t(inp["periodic"])
        self.species = t(inp["species"], torch.int64)
        self.r, self.v, self.s = t(inp["positions"]), t(inp["velocities"]), t(inp["spins"])
        self.s = self.s / torch.linalg.norm(self.s, dim=1, keepdim=True)
        self.n = self.r.shape[0]
        self.moment = self.m.moment[self.species] * MUB
        self.landau = None
        self.ref = None

    def pairs(self, r):
        """Ordered pairs within the radial cutoff plus a margin, by centre; kept while no atom has
        moved far."""
        if self.ref is not None:
            moved = _min_image(r - self.ref, self.L, self.per)
            if float((moved * moved).sum(1).max()) < 0.45 ** 2:
                return
        cut = self.m.rc + 1.0
        L, per = self.L.tolist(), [bool(x) for x in self.per.tolist()]
        nc = [max(1, int(L[a] // cut)) for a in range(3)]
        found_i, found_j = [], []
        if any(per[a] and nc[a] < 3 for a in range(3)):
            rows = max(1, int(4e7 // self.n))
            for lo in range(0, self.n, rows):
                d = _min_image(r[None, :, :] - r[lo:lo + rows, None, :], self.L, self.per)
                i, j = torch.nonzero((d * d).sum(2) < cut * cut, as_tuple=True)
                found_i.append(i + lo)
                found_j.append(j)
        else:
            cell = [torch.clamp((r[:, a] / (L[a] / nc[a])).floor().long(), 0, nc[a] - 1) for a in range(3)]
            flat = (cell[2] * nc[1] + cell[1]) * nc[0] + cell[0]
            count = torch.bincount(flat, minlength=nc[0] * nc[1] * nc[2])
            occ = int(count.max())
            order = torch.argsort(flat)
            first = torch.cumsum(count, 0) - count
            table = torch.full((count.numel(), occ), -1, dtype=torch.int64, device=self.dev)
            table[flat[order], torch.arange(self.n, device=self.dev) - first[flat[order]]] = order
            ids = torch.arange(count.numel(), device=self.dev)
            cx, cy, cz = ids % nc[0], (ids // nc[0]) % nc[1], ids // (nc[0] * nc[1])
            around = []
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    for dx in (-1, 0, 1):
                        x, y, z, ok = cx + dx, cy + dy, cz + dz, torch.ones_like(ids, dtype=torch.bool)
                        for a, w in enumerate((x, y, z)):
                            if not per[a]:
                                ok &= (w >= 0) & (w < nc[a])
                        other = ((z % nc[2]) * nc[1] + y % nc[1]) * nc[0] + x % nc[0]
                        around.append(torch.where(ok[:, None], table[other], -1))
            around = torch.cat(around, dim=1)
            rows = max(1, int(2e7 // (occ * around.shape[1])))
            for lo in range(0, count.numel(), rows):
                i, j = table[lo:lo + rows], around[lo:lo + rows]
                d = _min_image(r[j.clamp(min=0)][:, None] - r[i.clamp(min=0)][:, :, None], self.L, self.per)
                near = ((d * d).sum(3) < cut * cut) & (i >= 0)[:, :, None] & (j >= 0)[:, None, :]
                c, a, b = torch.nonzero(near, as_tuple=True)
                found_i.append(i[c, a])
                found_j.append(j[c, b])
        i, j = torch.cat(found_i), torch.cat(found_j)
        keep = i != j
        i, j = i[keep], j[keep]
        order = torch.argsort(i)
        self.pi, self.pj = i[order], j[order]
        self.starts = torch.cumsum(torch.bincount(i, minlength=self.n), 0)
        self.ref = r.clone()

    def evaluate(self, r, s, B=None, grad=True, rows=6144):
        """dict(E, F, H, W, q, e); B [n][3]: the external field on every atom, or None."""
        m, n = self.m, self.n
        self.pairs(r)
        ends = self.starts.cpu()
        F, H, W = torch.zeros_like(r), torch.zeros_like(s), torch.zeros(3, 3, dtype=r.dtype, device=self.dev)
        qs, es, E = [], [], 0.0
        for lo in range(0, n, rows):
            hi = min(n, lo + rows)
            p0, p1 = (int(ends[lo - 1]) if lo else 0), int(ends[hi - 1])
            i, j = self.pi[p0:p1], self.pj[p0:p1]
            d = _min_image(r[j] - r[i], self.L, self.per)
            inside = (d * d).sum(1) < m.rc * m.rc
            i, j, d = i[inside], j[inside], d[inside]
            S = s.clone()
            if grad:
                d.requires_grad_(True)
                S.requires_grad_(True)
            q = self._descriptor(i - lo, i, j, d, S, lo, hi)
            e = torch.tanh((q * m.scal) @ m.w0.T - m.b0) @ m.w1 - m.b1
            total = e.sum()
            if self.landau is not None:
                m2 = (S[lo:hi] * S[lo:hi]).sum(1)
                ab = self.landau[self.species[lo:hi]]
                total = total + (ab[:, 0] * m2 + ab[:, 1] * m2 * m2).sum()
            if B is not None:
                total = total - (self.moment[lo:hi, None] * B[lo:hi] * S[lo:hi]).sum()
            if grad:
                gd, gs = torch.autograd.grad(total, (d, S))
                F.index_add_(0, i, gd)
                F.index_add_(0, j, -gd)
                H -= gs
                W -= d.detach().T @ gd
            E += float(total.detach())
            qs.append(q.detach())
            es.append(e.detach())
        return dict(E=E, F=F, H=H, W=W, q=torch.cat(qs), e=torch.cat(es))

    def _descriptor(self, row, i, j, d, S, lo, hi):
        m, rows = self.m, hi - lo
        ti, tj = self.species[i], self.species[j]
        r = torch.sqrt((d * d).sum(1))
        u = d / r[:, None]
        si, sj = S[i], S[j]
        sij, siu, sju = (si * sj).sum(1), (si * u).sum(1), (sj * u).sum(1)
        phi = [torch.ones_like(sij), sij, (torch.linalg.cross(si, sj) * u).sum(1), siu * sju, siu * siu]
        f = _basis(r, m.rc)
        ct = m.c[self.species[lo:hi]]                       # [rows][tj][group][n][k]
        out = []
        for g, w in zip((0, 2, 3, 4, 5), phi):
            sums = torch.zeros(rows * 2, 9, dtype=f.dtype, device=self.dev).index_add_(0, row * 2 + tj, f * w[:, None])
            out.append(torch.einsum("rtk,rtnk->rn", sums.reshape(rows, 2, 9), ct[:, :, g]))
        near = torch.nonzero(r < m.ra, as_tuple=True)[0]
        g = torch.einsum("pk,pnk->pn", _basis(r[near], m.ra), m.c[ti[near], tj[near], 1])
        x, y, z = u[near].unbind(1)
        power = lambda b: [torch.ones_like(b), b, b * b, b * b * b, b * b * b * b]  # noqa: E731
        X, Y, Z = power(x), power(y), power(z)
        mono = torch.stack([X[a] * Y[b] * Z[c] for a, b, c in _MONO], dim=1)
        channels = []
        for w in (g, g * sij[near][:, None]):
            mom = torch.zeros(rows, 5, len(_MONO), dtype=f.dtype, device=self.dev)
            mom = mom.index_add_(0, row[near], w[:, :, None] * mono[:, None, :])
            sq = mom * mom * torch.tensor(_MONO_W, dtype=f.dtype, device=self.dev)
            N = [sum(sq[:, :, k] for k in range(len(_MONO)) if _MONO_D[k] == l) for l in range(5)]
            channels.append(torch.stack([N[1], 1.5 * N[2] - 0.5 * N[0], 2.5 * N[3] - 1.5 * N[1],
                                         (35.0 * N[4] - 30.0 * N[2] + 3.0 * N[0]) / 8.0], dim=2).reshape(rows, 20))
        own = (S[lo:hi] * S[lo:hi]).sum(1, keepdim=True)
        return torch.cat([out[0], channels[0], own, out[1], out[2], out[3], out[4], channels[1]], dim=1)

    # -------------------------------------------------------------- dynamics
    def omega(self, s, h, lam):
        return (h + lam * torch.linalg.cross(s, h)) / ((1.0 + lam * lam) * HBAR)

    @staticmethod
    def rotate(s, w, dt):
        size = torch.linalg.norm(w, dim=1, keepdim=True)
        a = torch.where(size > 0, w / torch.where(size > 0, size, torch.ones_like(size)), torch.zeros_like(w))
        th = size * dt
        along = (a * s).sum(1, keepdim=True)
        return s * torch.cos(th) + torch.linalg.cross(a, s) * torch.sin(th) + a * along * (1.0 - torch.cos(th))

    def trajectory(self, steps, T, B, seed, bits, mode="pc", Bat=None):
        """`steps` steps from the start; bits: 53 or 24 random bits of each uniform."""
        m, n, dt, lng = self.m, self.n, DT, mode == "longitudinal"
        field = torch.tensor(B, dtype=torch.float64, device=self.dev).expand(n, 3)
        if Bat is not None:
            field = field + torch.tensor(Bat, dtype=torch.float64, device=self.dev)
        if lng:
            self.landau = torch.tensor(LANDAU, dtype=torch.float64, device=self.dev)
        mass = m.mass[self.species][:, None]
        c = math.exp(-GAMMA * dt)
        sig_v = torch.sqrt((1.0 - c * c) * KB * T * ACC / mass)
        lam = 0.0 if lng else LAMBDA
        sig_eta = 0.0 if lng else math.sqrt(2.0 * LAMBDA * KB * T * HBAR / dt)
        drift, sig = (ALPHA * dt / HBAR, math.sqrt(2.0 * ALPHA * KB * T * dt / HBAR)) if lng else (0.0, 0.0)
        r, v, s = self.r, self.v, self.s
        first = self.evaluate(r, s)             # a system starts without an external field
        F, H = first["F"], first["H"]
        wrap = lambda x: torch.where(self.per > 0, x - self.L * torch.floor(x / self.L), x)  # noqa: E731
        for step in range(steps):
            xi, ze = (torch.tensor(_normals(step, n, stream, seed, bits), device=self.dev) for stream in (1, 2))
            r0 = r
            v = v + 0.5 * dt * F * ACC / mass
            r = r + 0.5 * dt * v
            v = c * v + sig_v * xi
            r = r + 0.5 * dt * v
            mid = wrap(r0 + 0.5 * (r - r0))
            r = wrap(r)
            eta = sig_eta * ze
            w0 = self.omega(s, H + eta, lam)
            guess = self.rotate(s, w0, dt) + drift * H + sig * ze
            if mode == "midpoint":
                X = guess
                for it in range(MID_CAP):
                    M = s + X
                    M = M / torch.linalg.norm(M, dim=1, keepdim=True)
                    h = self.evaluate(mid, M, field)["H"]
                    G = self.rotate(s, self.omega(M, h + eta, lam), dt)
                    moved = float(torch.linalg.norm(G - X, dim=1).max())
                    X = G
                    if moved < MID_TOL:
                        break
                s = X / torch.linalg.norm(X, dim=1, keepdim=True)
                now = self.evaluate(r, s, field)
            else:
                now = self.evaluate(r, guess, field)
                w1 = self.omega(guess, now["H"] + eta, lam)
                s = self.rotate(s, 0.5 * (w0 + w1), dt) + drift * 0.5 * (H + now["H"]) + sig * ze
                if not lng:
                    s = s / torch.linalg.norm(s, dim=1, keepdim=True)
            F, H = now["F"], now["H"]
            v = v + 0.5 * dt * F * ACC / mass
        return dict(positions=r, velocities=v, spins=s, forces=F, fields=H)


def _mulhilo(a, b):
    """High and low 64 bits of the products of a constant and an array of 64-bit words."""
    low = np.uint64(0xFFFFFFFF)
    a0, a1, s = np.uint64(a & 0xFFFFFFFF), np.uint64(a >> 32), np.uint64(32)
    b0, b1 = b & low, b >> s
    p00, p01, p10, p11 = a0 * b0, a0 * b1, a1 * b0, a1 * b1
    mid = (p00 >> s) + (p01 & low) + (p10 & low)
    return p11 + (p01 >> s) + (p10 >> s) + (mid >> s), (mid << s) | (p00 & low)


def _normals(step, n, stream, seed, bits):
    """Three normals per atom: Philox4x64-10 at counter (step, atom, stream, 0), key (seed, 0),
    and Box-Muller on uniforms of `bits` bits."""
    with np.errstate(over="ignore"):
        c = [np.full(n, step, np.uint64), np.arange(n, dtype=np.uint64), np.full(n, stream, np.uint64),
             np.zeros(n, np.uint64)]
        k0, k1 = int(seed), 0
        for rnd in range(10):
            if rnd:
                k0, k1 = (k0 + 0x9E3779B97F4A7C15) % 2 ** 64, (k1 + 0xBB67AE8584CAA73B) % 2 ** 64
            hi0, lo0 = _mulhilo(0xD2E7470EE14C6C93, c[0])
            hi1, lo1 = _mulhilo(0xCA5A826395121157, c[2])
            c = [hi1 ^ c[1] ^ np.uint64(k0), lo1, hi0 ^ c[3] ^ np.uint64(k1), lo0]
    u = [(x >> np.uint64(64 - bits)).astype(np.float64) for x in c]
    scale = 2.0 ** -bits
    a, b = np.sqrt(-2.0 * np.log((u[0] + 1.0) * scale)), 2.0 * math.pi * u[1] * scale
    return np.stack([a * np.cos(b), a * np.sin(b),
                     np.sqrt(-2.0 * np.log((u[2] + 1.0) * scale)) * np.cos(2.0 * math.pi * u[3] * scale)], axis=1)


EXACT_ATOM_EVALUATIONS = 1.2e6     # about 20 seconds of `evaluate`


def _numpy(d, *keys):
    return {k: d[k].cpu().numpy() for k in keys}


def _texture(r, s, L, per, cell):
    """Normalised spin sums of the columns along z: [n_b][n_a][3]."""
    na, nb = (max(1, int(math.floor(float(L[a]) / cell))) for a in (0, 1))
    ia, ib = (torch.clamp((r[:, a] / (L[a] / k)).floor().long(), 0, k - 1) for a, k in ((0, na), (1, nb)))
    m = torch.zeros(nb * na, 3, dtype=s.dtype, device=s.device).index_add_(0, ib * na + ia, s)
    size = torch.linalg.norm(m, dim=1, keepdim=True)
    m = torch.where(size > 0, m / torch.where(size > 0, size, torch.ones_like(size)), torch.zeros_like(m))
    return m.reshape(nb, na, 3)


def _solid_angle(a, b, c):
    return 2.0 * torch.atan2((a * torch.linalg.cross(b, c)).sum(-1),
                             1.0 + (a * b).sum(-1) + (b * c).sum(-1) + (c * a).sum(-1))


def _charge(m):
    """Berg-Luescher charge of a map periodic along its second index only."""
    right = torch.roll(m, -1, dims=1)
    a, b, c, d = m[:-1], right[:-1], right[1:], m[1:]
    return float((_solid_angle(a, b, c) + _solid_angle(a, c, d)).sum()) / (4.0 * math.pi)


def exact(case, seed):
    kind = case["kind"]
    bits = 24 if case.get("precision") == "mixed" else 53
    if kind == "batch":
        reps = _replicas(case, seed)
        if sum(r["inp"]["positions"].shape[0] * (r["steps"] + 1) for r in reps) > EXACT_ATOM_EVALUATIONS:
            return None
        return [_numpy(_Reference(r["inp"]).trajectory(r["steps"], r["T"], r["B"], r["seed"], bits), *_STATE)
                for r in reps]
    if kind in ("md", "film"):
        per_step = 6 if case.get("mode") == "midpoint" else 1
        if _atoms(case) * (per_step * case["steps"] + 1) > EXACT_ATOM_EVALUATIONS:
            return None
        if kind == "md":
            ref = _Reference(_md_inputs(case, seed))
            got = ref.trajectory(case["steps"], case["T"], (0.0, 0.0, case["B"]), seed, bits, case["mode"])
            return _numpy(got, *_STATE)
        inp = _film_inputs(case, seed)
        ref = _Reference(inp)
        got = ref.trajectory(case["steps"], case["T"], (0.0, 0.0, 0.0), seed, bits, Bat=_stepped_field(inp))
        m = _texture(got["positions"], got["spins"], ref.L, ref.per, TEXTURE_CELL)
        return dict(_numpy(got, *_STATE), m=m.cpu().numpy(), charge=_charge(m))
    if _atoms(case) > EXACT_ATOM_EVALUATIONS:
        return None
    ref = _Reference(_point_inputs(case, seed))
    got = ref.evaluate(ref.r, ref.s, grad=kind == "point")
    if kind == "point":
        return dict(E=got["E"], **_numpy(got, "F", "H", "W"))
    return _numpy(got, "q", "e")
