"""The work a user of this library has it do, as timed cases: run segments of the stabilised PIC step
(import a state, advance it, read the result), the batched sweep, the adjoint and a checkpoint restart,
over the sizes, precisions, shapes, gathers and solvers of the repository's configurations and tests.

Every pass starts from the same imported state, so a pass can be repeated and its outputs compared:
``pic_set_state`` -> ``pic_step`` -> ``pic_get_state`` (and the energies, or the gradients). The beam
carries small smooth fields at the start, so that the fields a run ends with are set by its inputs
and not by the rounding of two nearly cancelling species currents.

``exact`` advances the same state in FP64 with plain torch operations: the filter and the correction
as transfer functions in Fourier space, everything else node by node in a window of the particle.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_1401_0838_gb300 as P
from paper_1401_0838_gb300.autograd import WPerp

FIELDS = ("ex", "ey", "ez", "bx", "by", "bz")
SCHEMES = ("galerkin", "uniform", "momentum")
STAGGER = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))  # (x, y, z) of Ex .. Bz


def _case(**kw):
    """A case with the paper's beam problem as its defaults (Sec. 3: gamma = 130, filter (1, 1, a = 3))."""
    c = dict(kind="run", ndim=2, nx=64, ny=1, nz=128, ppc=4, alpha=0.5, gamma=130.0, scheme="galerkin", order=1,
             fp64=False, nbin=1, ncomp=1, comp=3.0, rational=False, ck=False, sigma=0.0, load="beam", u_th=1e-4,
             steps=10, ids=False, every=0, runs=0, mix=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest run: 64 x 128 in FP64, 4 particles per cell and species, 200 steps, energies every
        # step; latency and launches decide it
        _case(name="small_2d_fp64", fp64=True, steps=200, ids=True),
        # the main workload: 512 x 1024, 16 per cell and species, FP32, Galerkin, the 3-pass filter
        _case(name="beam_2d_fp32", nx=512, nz=1024, ppc=16, nbin=2, comp=2.0, steps=24),
        # the same grid with the Uniform gather at c dt/dz = 0.3: cells hold uneven numbers of particles
        _case(name="uniform_2d_fp32", nx=512, nz=1024, ppc=16, alpha=0.3, scheme="uniform", nbin=2, comp=2.0, steps=24),
        # the FP64 comparison run of the same workload, c dt/dz = 0.7
        _case(name="beam_2d_fp64", nx=512, nz=1024, ppc=16, alpha=0.7, fp64=True, nbin=2, comp=2.0, steps=8),
        # the 3D beam with a transverse Gaussian profile, at its full size (134M particles)
        _case(name="beam_3d_fp32", ndim=3, nx=128, ny=128, nz=512, ppc=8, sigma=20.0, steps=4),
        # cubic shapes, the setting of the paper's Sec. 3, on the main workload's grid
        _case(name="cubic_2d_fp32", nx=512, nz=1024, ppc=16, order=3, nbin=2, comp=2.0, steps=10),
        # one run of the growth-rate variants: 128 x 128, cubic, Cole-Karkkainen solver, the exact
        # rational multiplier
        _case(name="variant_2d_fp32", nx=128, nz=128, order=3, alpha=0.9, ck=True, rational=True, steps=100),
        # momentum-conserving gather on a ragged grid, a thermal load with random cell counts, and the
        # charge diagnostic at the end
        _case(name="momentum_2d_fp32", nx=301, nz=517, ppc=8, scheme="momentum", load="plasma", u_th=0.05, steps=20,
              ids=True),
        # 3D with cubic shapes, a small odd box
        _case(name="cubic_3d_fp32", ndim=3, nx=44, ny=36, nz=70, ppc=8, order=3, steps=4, ids=True),
        # the parameter sweep: 32 uneven runs advanced together
        _case(name="sweep_2d_fp32", kind="batch", nx=256, nz=1024, ppc=16, steps=20, every=10, runs=32, mix=4),
        # gradient of the final transverse field energy: forward, checkpoints, backward
        _case(name="adjoint_2d_fp32", kind="adjoint", nx=256, nz=512, ppc=8, steps=20, every=10, ids=True),
        # restart: load a checkpoint of tracked particles, a few steps, energies, write the next one
        _case(name="restart_2d_fp32", kind="restart", nx=512, nz=1024, ppc=16, steps=2, ids=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("linear",) * 5 + ("high",) * 3 + ("3d",) * 2 + ("batch", "adjoint", "restart"))
    c = _case(gamma=rng.choice((3.0, 10.0, 50.0, 130.0)), alpha=rng.choice((0.1, 0.2, 0.3, 0.4, 0.5, 0.6, 0.7)),
              scheme=rng.choice(SCHEMES[:2]), load=rng.choice(("beam", "beam", "plasma")),
              nx=_log_int(rng, 33, 512), nz=_log_int(rng, 65, 1024), ppc=rng.choice((2, 4, 6, 8, 9, 12, 16)))
    if c["load"] == "plasma":
        c["u_th"] = 0.05
    if rng.random() < 0.5:
        c.update(nbin=2, comp=2.0)
    if kind == "batch":
        c.update(kind="batch", scheme="galerkin", gamma=130.0, alpha=0.5, load="beam", u_th=1e-4, nx=256, nz=1024, ppc=16,
                 steps=rng.choice((10, 20)), every=10, runs=rng.randint(8, 28), mix=rng.randint(10, 10000))
        return c
    if kind == "adjoint":
        c.update(kind="adjoint", nx=_log_int(rng, 33, 256), nz=_log_int(rng, 65, 512), ppc=rng.choice((4, 8)),
                 load="beam", u_th=1e-4, fp64=rng.random() < 0.3, steps=rng.randint(6, 16), every=rng.randint(2, 10), ids=True)
        return c
    if kind == "restart":
        c.update(kind="restart", fp64=rng.random() < 0.4, steps=rng.randint(1, 3), ids=True)
        return c
    if kind == "high":
        c.update(order=rng.choice((1, 3, 3)), scheme=rng.choice(SCHEMES), fp64=rng.random() < 0.25)
        if c["order"] == 1:
            c["scheme"] = "momentum"
        if rng.random() < 0.3:
            c.update(ck=True, alpha=rng.choice((0.5, 0.8, 0.9, 0.95)))
        c["rational"] = c["scheme"] == "galerkin" and rng.random() < 0.3
        c.update(steps=rng.randint(4, 12), ids=rng.random() < 0.5)
        return c
    if kind == "3d":
        c.update(ndim=3, nx=_log_int(rng, 18, 96), ny=_log_int(rng, 18, 96), nz=_log_int(rng, 34, 256),
                 alpha=rng.choice((0.2, 0.3, 0.5)), ppc=rng.choice((2, 4, 8)), sigma=rng.choice((0.0, 12.0)),
                 steps=rng.randint(2, 4), ids=rng.random() < 0.5)
        if rng.random() < 0.3:
            c.update(nx=_log_int(rng, 18, 40), ny=_log_int(rng, 18, 40), nz=_log_int(rng, 34, 64), order=3, sigma=0.0,
                     scheme=rng.choice(SCHEMES))
        elif rng.random() < 0.2:
            c["fp64"] = True
        return c
    c.update(fp64=rng.random() < 0.35, ids=rng.random() < 0.4, steps=rng.randint(6, 24))
    if rng.random() < 0.2:
        c.update(ck=True, alpha=rng.choice((0.5, 0.8, 0.9)))
    return c


# --------------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------------
def _cells(c):
    return c["nx"] * (c["ny"] if c["ndim"] == 3 else 1) * c["nz"]


def _lattice(c):
    """Lattice points per cell and direction, as even as the count allows."""
    n, ndim = c["ppc"], c["ndim"]
    if ndim == 2:
        a = max(d for d in range(1, math.isqrt(n) + 1) if n % d == 0)
        return a, 1, n // a
    return min(((a, b, n // (a * b)) for a in range(1, n + 1) if n % a == 0 for b in range(a, n // a + 1)
                if (n // a) % b == 0 and n // (a * b) >= b), key=lambda t: t[2] - t[0])


def _initial(c, seed):
    """Fields and particles of the run at its start, in the run's precision and layout (on the GPU)."""
    dev, real = "cuda", torch.float64 if c["fp64"] else torch.float32
    g = torch.Generator(device=dev).manual_seed(int(seed) % (1 << 62))
    nx, ny, nz = c["nx"], c["ny"] if c["ndim"] == 3 else 1, c["nz"]
    fields = {}
    for n in FIELDS:
        f = torch.randn(nz, ny, nx, generator=g, device=dev, dtype=torch.float32)
        for d in range(3):
            if f.shape[d] > 1:
                f = (torch.roll(f, 1, d) + f + torch.roll(f, -1, d)) / 3
        fields[n] = (0.02 * f).to(real).contiguous()
    m = _cells(c) * c["ppc"]  # particles per species
    cell = torch.arange(_cells(c), device=dev, dtype=torch.int32).repeat_interleave(c["ppc"])
    off = []
    if c["load"] == "beam":  # a jittered lattice; the positron of a point sits on its electron
        lat = _lattice(c)
        q = torch.arange(c["ppc"], device=dev)
        place = (q % lat[0], (q // lat[0]) % lat[1], q // (lat[0] * lat[1]))
        for d in range(3):
            jit = 0.1 * (2 * torch.rand(m, generator=g, device=dev, dtype=torch.float32) - 1)
            o = ((place[d].float() + 0.5) / lat[d]).repeat(_cells(c)) + jit
            off.append(o.clamp_(0.0, 0.999).to(real).repeat(2))
        cell = cell.repeat(2)
    else:  # thermal plasma: both species uniform in the box, so cells hold random numbers
        cell = torch.randint(0, _cells(c), (2 * m,), generator=g, device=dev, dtype=torch.int32)
        cell = torch.cat([cell[:m].sort().values, cell[m:].sort().values])
        off = [torch.rand(2 * m, generator=g, device=dev, dtype=torch.float32).clamp_(0.0, 0.999).to(real) for _ in range(3)]
    part = {"cell": cell.contiguous(),
            "species": torch.arange(2, device=dev, dtype=torch.int32).repeat_interleave(m),
            "ox": off[0], "oy": off[1] if c["ndim"] == 3 else None, "oz": off[2]}
    for n in ("dux", "duy", "duz"):
        part[n] = (c["u_th"] * torch.randn(2 * m, generator=g, device=dev, dtype=torch.float32)).to(real)
    part["w"] = None
    if c["sigma"] > 0:  # transverse Gaussian profile about the box axis
        x = cell % nx + off[0] - 0.5 * nx
        y = (cell // nx) % ny + off[1] - 0.5 * ny
        part["w"] = (_weight(c) * torch.exp(-(x * x + y * y) / (2 * c["sigma"] ** 2))).to(real)
    part["id"] = torch.arange(2 * m, device=dev, dtype=torch.int32) if c["ids"] else None
    return fields, part


def _weight(c):
    return 0.3868 ** 2 / (2 * c["ppc"])


def _config(c, seed, diag):
    return P.pic_config_default(
        ndim=c["ndim"], nx=c["nx"], ny=c["ny"], nz=c["nz"], dt=c["alpha"], gamma=c["gamma"],
        scheme=SCHEMES.index(c["scheme"]), shape_order=c["order"], precision=P.PIC_FP64 if c["fp64"] else P.PIC_FP32,
        ppc_per_species=c["ppc"], u_th=c["u_th"], sigma_perp=c["sigma"], filter_nbin=c["nbin"], filter_ncomp=c["ncomp"],
        filter_comp_alpha=c["comp"], seed=seed % 1000 + 1, init_beam=0, track_ids=int(c["ids"]), diag_every=diag,
        correction_mode=P.PIC_CORR_RATIONAL if c["rational"] else P.PIC_CORR_SPLIT,
        field_solver=P.PIC_CK if c["ck"] else P.PIC_YEE)


def _sweep(c):
    """The runs of a batch: a mix of grids, particles per cell, Courant numbers and energies."""
    r = np.random.default_rng(c["mix"])
    runs = []
    for _ in range(c["runs"]):
        runs.append(_case(nx=int(r.choice([64, 128, 256])), nz=int(r.choice([128, 256, 512, 1024])),
                          ppc=int(r.choice([4, 8, 16])), alpha=float(r.choice([0.1, 0.2, 0.3, 0.4, 0.5, 0.6, 0.7])),
                          gamma=float(r.choice([10.0, 50.0, 130.0])), nbin=c["nbin"], comp=c["comp"], steps=c["steps"]))
    return runs


class _State:
    """What the program holds: the handle (or batch), its stream, the initial state and the arrays it reads back into."""

    def __init__(self, case):
        self.case, self.h, self.b, self.runs = case, None, None, []
        self.stream = torch.cuda.Stream()

    def __del__(self):
        if self.b is not None:
            P.pic_batch_destroy(self.b)
        elif self.h is not None:
            P.pic_destroy(self.h)


def _arrays(c, fields, part, particles):
    """Arrays to read a run's state back into."""
    out = {"fields": {n: torch.empty_like(f) for n, f in fields.items()}, "part": None}
    if particles:
        out["part"] = {n: torch.empty_like(a) for n, a in part.items() if a is not None}
    return out


def prepare(case, seed):
    c = dict(case)
    s = _State(c)
    if c["kind"] == "batch":
        cases = _sweep(c)
        s.b = P.pic_batch_create([_config(k, seed + i, c["every"]) for i, k in enumerate(cases)])
        P.pic_batch_set_stream(s.b, s.stream.cuda_stream)
        for i, k in enumerate(cases):
            P.pic_batch_set_correction_stencil(s.b, i, *P.pic_compute_correction_coeffs(P.PIC_GALERKIN, k["alpha"]))
            fields, part = _initial(k, seed + 7919 * i)
            out = _arrays(k, fields, part, False)
            s.runs.append((P.pic_batch_run(s.b, i), P.make_state(P.PIC_DEVICE, fields, part), out, (fields, part)))
    else:
        s.h = P.pic_create(_config(c, seed, 0 if c["kind"] == "adjoint" else 1))
        P.pic_set_stream(s.h, s.stream.cuda_stream)
        psi = P.pic_compute_correction_coeffs(SCHEMES.index(c["scheme"]), c["alpha"])
        fields, part = _initial(c, seed)
        if c["kind"] == "adjoint":
            s.psi = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in psi]
            s.fields = [fields[n].requires_grad_(True) for n in FIELDS]
            s.part = part
            s.start = P.make_state(P.PIC_DEVICE, None, {k: v for k, v in part.items() if k != "id"})
        else:
            P.pic_set_correction_stencil(s.h, *psi)
            s.keep = (fields, part)
            s.start = P.make_state(P.PIC_DEVICE, fields, part)
            s.out = _arrays(c, fields, part, c["ids"])
    torch.cuda.synchronize()
    return s


def _energies(h, real):
    e = [[q["w_e"], q["w_b"], q["w_perp"], q["k"]] for q in h]
    return torch.tensor(e, dtype=real)


def _read(h, c, out, start):
    """The run's fields and, where they are tracked, its particles in id order: the displacement since the
    start (in cells) and the momenta."""
    st = P.make_state(P.PIC_DEVICE, out["fields"], out["part"])
    P.pic_get_state(h, st)
    got = dict(out["fields"])
    if out["part"] is not None:
        a, i = out["part"], out["part"]["id"].long()
        n = (c["nx"], c["ny"], c["nz"])
        strides = (1, c["nx"], c["nx"] * c["ny"])
        moves = []
        for d, name in ((0, "ox"), (1, "oy"), (2, "oz")):
            if name not in a:
                continue
            cells = (a["cell"] // strides[d]) % n[d] - (start["cell"][i] // strides[d]) % n[d]
            move = cells + (a[name] - start[name][i])
            move = move - n[d] * torch.round(move / n[d])
            moves.append(torch.empty_like(move).index_copy_(0, i, move))
        got["move"] = torch.stack(moves)
        got["du"] = torch.stack([torch.empty_like(a[name]).index_copy_(0, i, a[name]) for name in ("dux", "duy", "duz")])
    return got


def run(state):
    c = state.case
    real = torch.float64 if c["fp64"] else torch.float32
    with torch.cuda.stream(state.stream):
        if c["kind"] == "batch":
            for h, start, _, _ in state.runs:
                P.pic_set_state(h, start)
            P.pic_batch_step(state.b, c["steps"])
            got = {n: [] for n in FIELDS}
            hist = []
            for i, (h, _, out, keep) in enumerate(state.runs):
                for n, f in _read(h, c, out, keep[1]).items():
                    got[n].append(f.reshape(-1))
                hist.append(_energies(P.pic_batch_energy_history(state.b, i, c["steps"] // c["every"]), real))
            return {**{n: torch.cat(v) for n, v in got.items()}, "energies": torch.cat(hist)}
        P.pic_set_state(state.h, state.start)
        if c["kind"] == "adjoint":
            for t in state.psi + state.fields:
                t.grad = None
            w = WPerp.apply(state.h, c["steps"], c["every"], *state.psi, *state.fields)
            w.backward()
            return {"w_perp": w.detach().to(real), "psi_e": state.psi[0].grad.to(real), "psi_b": state.psi[1].grad.to(real),
                    **{n: f.grad for n, f in zip(FIELDS, state.fields)}}
        P.pic_step(state.h, c["steps"])
        if c["kind"] == "restart":
            e = _energies([P.pic_energy(state.h)], real)
        else:
            e = _energies(P.pic_energy_history(state.h, c["steps"]), real)
        got = {**_read(state.h, c, state.out, state.keep[1]), "energies": e}
        if c["load"] == "plasma":
            r = P.pic_charge_residual(state.h)
            got["residual"] = torch.tensor([r["max"], r["rms"], r["rho_max"]], dtype=real)
        return got


def work(case):
    """Per step: every particle's offsets, momenta (and weight) read and written once, E and B read and written
    once; the arithmetic of gather, push, move and deposit (window sizes of the shape order), the stencils and the
    field update. The adjoint: the forward run, its recomputation and the transposed passes (twice the forward's)."""
    if case["kind"] == "batch":
        parts = [work(k) for k in _sweep(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    c = case
    n, cells, es = 2 * _cells(c) * c["ppc"], _cells(c), 8 if c["fp64"] else 4
    arrays = (3 if c["ndim"] == 3 else 2) + 3 + (1 if c["sigma"] > 0 else 0)
    nodes = (c["order"] + 1) ** c["ndim"]
    per_particle = 12 * nodes + 90 + 6 * (c["order"] + 2) * nodes
    per_cell = 6 * 2 * 9 + 9 * 2 * 5 * c["ndim"] + 60
    steps = c["steps"] * (4 if c["kind"] == "adjoint" else 1)
    return {"bytes": steps * 2.0 * es * (n * arrays + 6 * cells), "flops": steps * (float(n) * per_particle + cells * per_cell)}


# --------------------------------------------------------------------------------------------------
# The same passes in FP64
# --------------------------------------------------------------------------------------------------
def _coefficients(scheme, alpha):
    """The (4, 4) rational interpolant of the field multiplier on xi = sin^2(k dz / 2) = j / 8 (Sec. 2)."""
    xi = np.arange(9) / 8.0
    s = np.arcsin(np.sqrt(xi))
    s[0] = 1.0
    base = 0.5 * np.sin(2 * alpha * s) / alpha / np.sin(s)
    m = base * {"galerkin": s / np.sin(s), "uniform": 1.0, "momentum": np.cos(s)}[scheme]
    m[0] = 1.0
    if np.all(np.abs(m - 1) < 1e-12):
        return np.eye(5)[0], np.eye(5)[0]
    a = np.concatenate([xi[:, None] ** np.arange(5), -m[:, None] * xi[:, None] ** np.arange(1, 5)], axis=1)
    x = np.linalg.solve(a, m)
    return x[:5], np.concatenate([[1.0], x[5:]])


def _transfers(c, psi_e, psi_b):
    """Fourier transfer functions of the transverse E copies, of the other copies and of the current."""
    axes = [torch.arange(n, device="cuda", dtype=torch.float64) * (2 * math.pi / n) for n in (c["nz"], c["ny"], c["nx"])]
    filt = torch.ones((), device="cuda", dtype=torch.float64)
    for d, k in enumerate(axes):
        if d == 1 and c["ndim"] == 2:
            continue
        cos = torch.cos(k)
        t = (0.5 + 0.5 * cos) ** c["nbin"] * (c["comp"] - (c["comp"] - 1) * cos) ** c["ncomp"]
        filt = filt * t.reshape([-1 if q == d else 1 for q in range(3)])
    xi = (torch.sin(axes[0] / 2) ** 2).reshape(-1, 1, 1)
    pe, pb = (sum(v[n] * xi ** n for n in range(5)) for v in (psi_e, psi_b))
    if c["rational"]:
        return pe / pb * filt, filt, filt
    return pe * filt, pb * filt, filt


def _apply(t, f):
    return torch.fft.ifftn(torch.fft.fftn(f) * t).real


def _spline(n, t):
    a = t.abs()
    if n == 0:
        return ((t >= -0.5) & (t < 0.5)).to(t.dtype)
    if n == 1:
        return (1 - a).clamp(min=0)
    if n == 2:
        return torch.where(a <= 0.5, 0.75 - a * a, 0.5 * (1.5 - a).clamp(min=0) ** 2)
    return torch.where(a <= 1, 2 / 3 - a * a + 0.5 * a ** 3, (2 - a).clamp(min=0) ** 3 / 6)


def _wrap(i, n):
    return torch.remainder(i, n)


def _gather(c, G, cell, off):
    """The six components at the particles (cell and off: lists per direction)."""
    dims = (0, 2) if c["ndim"] == 2 else (0, 1, 2)
    n = (c["nx"], c["ny"], c["nz"])
    made = {}

    def line(d, st, order):
        if (d, st, order) not in made:
            xs = off[d] - 0.5 * st
            fl = torch.floor(xs if order % 2 else xs + 0.5).detach()
            first = fl - (order // 2)
            made[d, st, order] = [(_wrap(cell[d] + first.long() + q, n[d]), _spline(order, xs - (first + q)) if order else None)
                                  for q in range(order + 1)]
        return made[d, st, order]

    out = []
    for q in range(6):
        flat = G[q].reshape(-1)
        lines = []
        for d in dims:
            st = 0 if c["scheme"] == "momentum" else STAGGER[q][d]
            lines.append(line(d, st, c["order"] - st if c["scheme"] == "galerkin" else c["order"]))
        acc = 0
        for kz, wz in lines[-1]:
            for ky, wy in (lines[1] if c["ndim"] == 3 else ((None, None),)):
                row = kz * c["ny"] + ky if ky is not None else kz
                for kx, wx in lines[0]:
                    v = flat[row * c["nx"] + kx]
                    for w in (wx, wy, wz):
                        v = v * w if w is not None else v
                    acc = acc + v
        out.append(acc)
    return out


def _deposit(c, J, cell, off, move, vy, qw):
    """Esirkepov's current, added to the flat arrays J."""
    lo, nw = (-1, 4) if c["order"] == 1 else (-2, 6)
    n = (c["nx"], c["ny"], c["nz"])
    dims = (0, 2) if c["ndim"] == 2 else (0, 1, 2)
    idx, ds, mid, run_ = {}, {}, {}, {}
    for d in dims:
        idx[d] = [_wrap(cell[d] + lo + a, n[d]) for a in range(nw)]
        s0 = [_spline(c["order"], lo + a - off[d]) for a in range(nw)]
        ds[d] = [_spline(c["order"], lo + a - off[d] - move[d]) - s0[a] for a in range(nw)]
        mid[d] = [s0[a] + 0.5 * ds[d][a] for a in range(nw)]
        acc, run_[d] = 0, []
        for a in range(nw - 1):
            acc = acc + ds[d][a]
            run_[d].append(-qw / c["alpha"] * acc)  # dx = dy = dz = 1

    def at(ix, iy, iz):
        return (iz * c["ny"] + iy) * c["nx"] + ix if iy is not None else iz * c["nx"] + ix

    def cross(d, e, a, b):
        return mid[d][a] * mid[e][b] + ds[d][a] * ds[e][b] / 12

    if c["ndim"] == 2:
        for b in range(nw):
            for a in range(nw - 1):
                J[0].index_add_(0, at(idx[0][a], None, idx[2][b]), run_[0][a] * mid[2][b])
                J[2].index_add_(0, at(idx[0][b], None, idx[2][a]), run_[2][a] * mid[0][b])
            for a in range(nw):
                J[1].index_add_(0, at(idx[0][a], None, idx[2][b]), qw * vy * cross(0, 2, a, b))
        return
    for d in dims:
        e, f = [k for k in dims if k != d]
        for b in range(nw):
            for g in range(nw):
                t = cross(e, f, b, g)
                for a in range(nw - 1):
                    k = {d: idx[d][a], e: idx[e][b], f: idx[f][g]}
                    J[d].index_add_(0, at(k[0], k[1], k[2]), run_[d][a] * t)


def _push(c, G, J, p):
    """One chunk of particles: gather, Boris, move, deposit. p: (cell, off, u, q, w); returns the same, moved."""
    cell, off, u, q, w = p
    F = _gather(c, G, cell, off)
    h = 0.5 * c["alpha"] * q
    m = [u[a] + h * F[a] for a in range(3)]
    gam = torch.sqrt(1 + m[0] ** 2 + m[1] ** 2 + m[2] ** 2)
    t = [h * F[3 + a] / gam for a in range(3)]
    s = 2 / (1 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
    cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
    r = cross(m, t)
    r = cross([m[a] + r[a] for a in range(3)], [s * t[a] for a in range(3)])
    u = [m[a] + r[a] + h * F[a] for a in range(3)]
    gam = torch.sqrt(1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    v = [x / gam for x in u]
    move = [c["alpha"] * x for x in v]
    _deposit(c, J, cell, off, move, v[1], q * w)
    n = (c["nx"], c["ny"], c["nz"])
    to, new = list(cell), list(off)
    for d in (0, 2) if c["ndim"] == 2 else (0, 1, 2):
        x = off[d] + move[d]
        fl = torch.floor(x).detach()
        to[d], new[d] = _wrap(cell[d] + fl.long(), n[d]), x - fl
    return to, new, u, q, w


def _advance(c, F, parts, tr):
    """One step of fields F (list of six) and particle chunks."""
    G = [_apply(tr[0] if q < 2 else tr[1], F[q]) for q in range(6)]
    if c["scheme"] == "momentum":
        for q in range(6):
            for d, axis in enumerate((2, 1, 0)):
                if STAGGER[q][d]:
                    G[q] = 0.5 * (G[q] + torch.roll(G[q], 1, axis))
    J = [torch.zeros(F[0].numel(), device="cuda", dtype=torch.float64) for _ in range(3)]
    parts = [_push(c, G, J, p) for p in parts]
    J = [_apply(tr[2], j.reshape(F[0].shape)) for j in J]
    up = lambda f, ax: torch.roll(f, -1, ax) - f  # noqa: E731
    dn = lambda f, ax: f - torch.roll(f, 1, ax)  # noqa: E731
    mean = lambda f, ax: 0.75 * f + 0.125 * (torch.roll(f, 1, ax) + torch.roll(f, -1, ax))  # noqa: E731
    ux = (lambda f: mean(up(f, 2), 0)) if c["ck"] else (lambda f: up(f, 2))  # Cole-Karkkainen: beta = 1/8
    uz = (lambda f: mean(up(f, 0), 2)) if c["ck"] else (lambda f: up(f, 0))
    uy = lambda f: up(f, 1)  # noqa: E731

    def half(e, b):
        h = 0.5 * c["alpha"]
        return [b[0] - h * (uy(e[2]) - uz(e[1])), b[1] - h * (uz(e[0]) - ux(e[2])), b[2] - h * (ux(e[1]) - uy(e[0]))]

    e, b = F[:3], half(F[:3], F[3:])
    curl = (dn(b[2], 1) - dn(b[1], 0), dn(b[0], 0) - dn(b[2], 2), dn(b[1], 2) - dn(b[0], 1))
    e = [e[a] + c["alpha"] * (curl[a] - J[a]) for a in range(3)]
    return e + half(e, b), parts


def _chunks(c, part, size):
    u0 = math.sqrt(c["gamma"] ** 2 - 1)
    out = []
    for lo in range(0, part["cell"].numel(), size):
        cut = {n: a[lo:lo + size] for n, a in part.items() if a is not None}
        cl = cut["cell"].long()
        cell = [cl % c["nx"], (cl // c["nx"]) % c["ny"], cl // (c["nx"] * c["ny"])]
        off = [cut["ox"].double(), cut["oy"].double() if c["ndim"] == 3 else None, cut["oz"].double()]
        u = [cut["dux"].double(), cut["duy"].double(), u0 + cut["duz"].double()]
        w = cut["w"].double() if "w" in cut else torch.full_like(u[0], _weight(c))
        out.append((cell, off, u, cut["species"].double() * 2 - 1, w))
    return out


def _sums(F, parts):
    e, b = sum((f * f).sum() for f in F[:3]), sum((f * f).sum() for f in F[3:])
    perp = sum((F[q] * F[q]).sum() for q in (0, 1, 3, 4))
    k = 0
    for _, _, u, _, w in parts:
        u2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        k = k + (w * u2 / (torch.sqrt(1 + u2) + 1)).sum()
    return torch.stack([0.5 * e, 0.5 * b, 0.5 * perp, k])


def _residual(c, F, parts, tr):
    """max and RMS of div E - F rho over the nodes, and max |F rho|."""
    rho = torch.zeros(F[0].numel(), device="cuda", dtype=torch.float64)
    lo, nn = (0, 2) if c["order"] == 1 else (-1, 4)
    n = (c["nx"], c["ny"], c["nz"])
    for cell, off, _, q, w in parts:
        nodes = {d: [(_wrap(cell[d] + lo + a, n[d]), _spline(c["order"], lo + a - off[d])) for a in range(nn)]
                 for d in ((0, 2) if c["ndim"] == 2 else (0, 1, 2))}
        for kz, wz in nodes[2]:
            for ky, wy in nodes.get(1, ((0, 1.0),)):
                for kx, wx in nodes[0]:
                    rho.index_add_(0, (kz * c["ny"] + ky) * c["nx"] + kx, q * w * wx * wy * wz)
    rho = _apply(tr[2], rho.reshape(F[0].shape))
    res = sum(F[a] - torch.roll(F[a], 1, 2 - a) for a in range(3) if c["ndim"] == 3 or a != 1) - rho
    return torch.stack([res.abs().max(), res.square().mean().sqrt(), rho.abs().max()])


def _exact_run(c, seed):
    fields, part = _initial(c, seed)
    F = [fields[n].double() for n in FIELDS]
    psi = _coefficients(c["scheme"], c["alpha"])
    tr = _transfers(c, *psi)
    parts = _chunks(c, part, 1 << 22)
    energies = []
    for _ in range(c["steps"]):
        F, parts = _advance(c, F, parts, tr)
        energies.append(_sums(F, parts))
    got = dict(zip(FIELDS, F))
    if c["kind"] == "restart":
        energies = energies[-1:]
    return got, energies, parts, tr, part


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        got, hist = {n: [] for n in FIELDS}, []
        with torch.no_grad():
            for i, k in enumerate(_sweep(c)):
                f, e, _, _, _ = _exact_run(k, seed + 7919 * i)
                for n in FIELDS:
                    got[n].append(f[n].reshape(-1))
                hist += e[c["every"] - 1::c["every"]]
        return {**{n: torch.cat(v) for n, v in got.items()}, "energies": torch.stack(hist)}
    n = 2 * _cells(c) * c["ppc"]
    window = (c["order"] + 3) ** c["ndim"] * c["ndim"]
    if n * c["steps"] * window > 2.5e10:
        return None
    if c["kind"] == "adjoint":
        fields, part = _initial(c, seed)
        psi = [torch.tensor(v, device="cuda", dtype=torch.float64, requires_grad=True)
               for v in _coefficients(c["scheme"], c["alpha"])]
        F0 = [fields[k].double().requires_grad_(True) for k in FIELDS]
        F, parts = F0, _chunks(c, part, n)
        for _ in range(c["steps"]):
            F, parts = checkpoint(lambda f, p, a, b: _advance(c, f, p, _transfers(c, a, b)), F, parts, *psi, use_reentrant=False)
        w = 0.5 * sum((F[q] * F[q]).sum() for q in (0, 1, 3, 4))
        w.backward()
        return {"w_perp": w.detach(), "psi_e": psi[0].grad, "psi_b": psi[1].grad, **{k: f.grad for k, f in zip(FIELDS, F0)}}
    with torch.no_grad():
        got, energies, parts, tr, part = _exact_run(c, seed)
        got["energies"] = torch.stack(energies)
        if c["ids"]:
            start = _chunks(c, part, 1 << 22)
            m = (c["nx"], c["ny"], c["nz"])
            moves = []
            for d in (0, 2) if c["ndim"] == 2 else (0, 1, 2):
                move = torch.cat([(p[0][d] - q[0][d]) + (p[1][d] - q[1][d]) for p, q in zip(parts, start)])
                moves.append(move - m[d] * torch.round(move / m[d]))
            got["move"] = torch.stack(moves)
            u = [torch.cat([p[2][a] for p in parts]) for a in range(3)]
            got["du"] = torch.stack([u[0], u[1], u[2] - math.sqrt(c["gamma"] ** 2 - 1)])
        if c["load"] == "plasma":
            got["residual"] = _residual(c, [got[k] for k in FIELDS], parts, tr)
        return got
