"""Timed cases: the calls that users of this framework make, over the sizes they make them at.

A case is one pass of a user's program through the public entry points (`binding.py`, the C ABI's names, and
`adjoint.py`).  Most passes are a run that restarts from a state kept on the device: one copy puts fields and
particles back into the caller's buffers, then the run's steps follow.  So every pass does the same work, whatever
ran before it.  The particles of a state are grouped by tiles as they were a few steps earlier, the order in which a
sort finds them.

Outputs are the caller's own buffers.  The library reorders particles when it sorts, in no specified order inside a
bin, so the particle arrays are returned where no sort runs in the pass (`restart_2d`) and the field planes, on which
every particle's push and deposit act, in all runs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1906_06306_gb300 import binding as B

C = 0.45  # Courant number of every set-up of the repository
DEV = "cuda:0"


# ------------------------------------------------------------------------------------------------ the cases

def listed():
    step = dict(kind="step", order=2, pusher="boris", passes=0, setup="turbulence", tuning="default")
    return [
        # the 1D Weibel box of the benchmark: 65,536 particles, so that launches and latency are what counts
        dict(step, name="weibel_1d", setup="weibel", dim=1, nx=512, ny=1, nz=1, ppc=64, steps=20),
        # a run that is watched as it goes: one pic_step(1) per pass, the state moving on from pass to pass
        dict(kind="live", name="live_2d", setup="turbulence", dim=2, nx=130, ny=94, nz=1, ppc=8, order=2,
             pusher="boris", passes=1, tuning="default"),
        # a 2D Weibel box with odd sides, as the ensemble draws them, stepped alone
        dict(step, name="weibel_2d_odd", setup="weibel", dim=2, nx=133, ny=133, nz=1, ppc=40, steps=20),
        # the headline: decaying turbulence on 1024^2 with 33.5 M particles, at the tuning that autotune settles on
        dict(step, name="turbulence_2d", dim=2, nx=1024, ny=1024, nz=1, ppc=16, steps=10, tuning="16x8h4"),
        # the solvers of the paper's shock run (FDTD4, Higuera-Cary, 8 filter passes) on a 2D box
        dict(step, name="fdtd4_hc_2d", setup="flow", dim=2, nx=768, ny=384, nz=1, ppc=16, steps=10, order=4,
             pusher="higuera_cary", passes=8),
        # the 3D shock benchmark's plasma in a periodic box: 134 M cold streaming particles, 4 filter passes
        dict(step, name="shock_3d", setup="flow", dim=3, nx=512, ny=128, nz=128, ppc=8, steps=3, passes=4),
        # the same flow running into the conducting wall, on a ragged box; the upstream has ended (no injection)
        dict(step, name="wall_3d", setup="wall", dim=3, nx=121, ny=43, nz=38, ppc=8, steps=3, passes=4),
        # one step from a checkpoint whose tile grouping was kept (what the adjoint's reverse sweep does to
        # recompute a segment): no sort, so the particles come back in their own slots
        dict(kind="restart", name="restart_2d", setup="turbulence", dim=2, nx=256, ny=256, nz=1, ppc=16, order=2,
             pusher="boris", passes=0, tuning="default"),
        # smoothing of a current by itself, on the planes of the 3D benchmark
        dict(kind="filter", name="filter_3d", dim=3, nx=1024, ny=128, nz=128, passes=4, static=False),
        # the diagnostics of the headline box: energies and the Gauss residual, read by the host
        dict(kind="energies", name="energies_2d", setup="turbulence", dim=2, nx=1024, ny=1024, nz=1, ppc=16,
             passes=0),
        # gradient of the magnetic energy after 20 steps, by the discrete adjoint (forward and reverse)
        dict(kind="adjoint", name="adjoint_2d", nx=128, ny=128, ppc=32, modes=4, steps=20, every=20),
        # an ensemble of uneven 1D and 2D Weibel boxes stepped as one batch
        dict(kind="batch", name="batch_weibel", boxes=24, n1_max=4096, n2_max=256, ppc_max=64, steps=10),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sides(dim, cells):
        """Sides of a box of about `cells` cells, no more than 4 apart in ratio."""
        if dim == 1:
            return cells, 1, 1
        r = [math.exp(rng.uniform(-0.7, 0.7)) for _ in range(dim)]
        s = (cells / math.prod(r)) ** (1.0 / dim)
        n = [max(8, int(round(s * x))) for x in r]
        return tuple(n + [1] * (3 - dim))

    kind = rng.choice(["step"] * 6 + ["live", "restart", "filter", "energies", "adjoint", "batch"])
    if kind == "batch":
        return dict(kind=kind, boxes=rng.randint(8, 32), n1_max=log(512, 4096), n2_max=log(64, 256),
                    ppc_max=log(24, 64), steps=rng.choice([10, 20]))
    if kind == "adjoint":
        n = log(24, 128)
        return dict(kind=kind, nx=n, ny=max(8, n + rng.randint(-7, 0)), ppc=2 * log(2, 16), modes=rng.randint(2, 4),
                    steps=rng.randint(8, 20), every=rng.choice([5, 10, 20]))
    dim = rng.choice([1, 2, 2, 3, 3])
    if kind == "filter":
        static = rng.random() < 0.3
        nx, ny, nz = sides(dim, log(2000, 1_000_000 if static else 12_000_000))
        return dict(kind=kind, dim=dim, nx=nx, ny=min(ny, 65535), nz=nz, passes=rng.choice([1, 2, 4, 8]),
                    static=static)
    ppc = 2 * log(2, {1: 64, 2: 20, 3: 4}[dim])
    most = {1: 4096, 2: 500_000, 3: 4_000_000}[dim]
    nx, ny, nz = sides(dim, log({1: 128, 2: 1500, 3: 4000}[dim], most if kind in ("step", "energies") else most // 8))
    passes = rng.choice([0, 0, 1, 4])
    if kind == "energies":
        return dict(kind=kind, setup="turbulence", dim=dim, nx=nx, ny=ny, nz=nz, ppc=ppc, passes=passes)
    order = rng.choice([2, 2, 4]) if dim < 3 else 2
    case = dict(kind=kind, setup=rng.choice(["weibel", "turbulence", "flow"]), dim=dim, nx=nx, ny=ny, nz=nz, ppc=ppc,
                order=order, pusher=rng.choice(["boris", "boris", "higuera_cary"]), passes=passes,
                tuning="16x8h4" if dim == 2 and rng.random() < 0.5 else "default")
    if kind == "step":
        if dim > 1 and nx >= 24 and rng.random() < 0.2:
            case["setup"] = "wall"
        case["steps"] = rng.choice([3, 6]) if dim == 3 else rng.choice([10, 20]) if nx * ny * ppc < 4e6 else 10
    return case


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _thermal(g, n, theta):
    """Isotropic Maxwell-Juettner four-velocities [3, n]: |u| by inverting the tabulated distribution of
    u^2 exp(-(gamma - 1) / theta)."""
    p = np.linspace(0.0, math.sqrt((1.0 + 40.0 * theta) ** 2 - 1.0), 1 << 14)
    f = p * p * np.exp(-(np.sqrt(1.0 + p * p) - 1.0) / theta)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (f[1:] + f[:-1]))])
    inv = np.interp(np.linspace(0.0, 1.0, 1 << 16), cdf / cdf[-1], p)
    table = torch.tensor(inv, dtype=torch.float32, device=DEV)
    t = torch.rand(n, generator=g, device=DEV) * (len(inv) - 1)
    k = t.to(torch.int64).clamp_(max=len(inv) - 2)
    mag = torch.lerp(table[k], table[k + 1], t - k)
    ct = 2.0 * torch.rand(n, generator=g, device=DEV) - 1.0
    phi = 2.0 * math.pi * torch.rand(n, generator=g, device=DEV)
    st = torch.sqrt((1.0 - ct * ct).clamp_(min=0.0))
    return torch.stack([mag * st * torch.cos(phi), mag * st * torch.sin(phi), mag * ct])


SETUPS = {  # temperature, skin depth in cells, bulk Lorentz factor, its axis, steps since the last sort
    "turbulence": dict(theta=0.3, r_p=4.0, gamma=1.0, axis=0, age=10),  # at rest in a guide field, sigma = 10
    "weibel": dict(theta=0.01, r_p=10.0, gamma=3.0, axis=1, age=10),  # counter-streaming beams
    "flow": dict(theta=1e-4, r_p=10.0, gamma=10.0, axis=0, age=3),  # cold flow toward -x
    "wall": dict(theta=1e-4, r_p=10.0, gamma=10.0, axis=0, age=3),  # the same, onto the conducting wall
}
WALL = 2  # node plane of the conducting wall


def _charge(setup, ppc):
    s = SETUPS[setup]
    th = s["theta"]
    mean = s["gamma"] if s["gamma"] > 1.0 else 1.0 + 1.5 * th + 15.0 / 8.0 * th * th
    return float(np.float32((C / s["r_p"]) ** 2 * mean / (2.0 * ppc))), mean


def _plasma(g, case):
    """An electron-positron plasma of about ppc particles per cell per species: species dicts with q, m, cell int32[n],
    off float32[D, n], u float32[3, n] (pairs start co-located), and the field planes float32[9, nz, ny, nx]."""
    setup, dim, ppc = case["setup"], case["dim"], case["ppc"]
    s, N = SETUPS[setup], (case["nx"], case["ny"], case["nz"])
    q, mean = _charge(setup, ppc)
    lo, hi = (WALL, N[0] - 3) if setup == "wall" else (0, N[0])
    n = (hi - lo) * N[1] * N[2] * ppc
    ijk = [torch.randint(lo if d == 0 else 0, hi if d == 0 else N[d], (n,), generator=g, device=DEV,
                         dtype=torch.int32) for d in range(dim)]
    off = torch.rand((dim, n), generator=g, device=DEV)
    tile = {1: (64,), 2: (16, 16), 3: (8, 8, 4)}[dim]
    species = []
    for sign in (-1.0, 1.0):
        u = _thermal(g, n, s["theta"])
        if s["gamma"] > 1.0:
            beta = math.sqrt(1.0 - 1.0 / s["gamma"] ** 2)
            b = torch.full((n,), -beta, device=DEV)
            if setup == "weibel":  # half of each species each way
                b = torch.where(torch.rand(n, generator=g, device=DEV) < 0.5, beta, -beta)
            ax = 0 if setup == "weibel" and dim > 1 else s["axis"]
            gam = torch.sqrt(1.0 + (u * u).sum(0))
            u[ax] = s["gamma"] * (u[ax] + b * gam)
        # the order of an array that was sorted by tile `age` steps ago
        gam = torch.sqrt(1.0 + (u * u).sum(0))
        key = torch.zeros(n, dtype=torch.int32, device=DEV)
        for d in reversed(range(dim)):
            past = torch.floor(ijk[d] + off[d] - s["age"] * C * u[d] / gam).to(torch.int32) % N[d]
            key = key * ((N[d] + tile[d] - 1) // tile[d]) + past // tile[d]
        o = torch.argsort(key, stable=True)
        cell = torch.zeros(n, dtype=torch.int32, device=DEV)
        for d in reversed(range(dim)):
            cell = cell * N[d] + ijk[d]
        species.append(dict(q=sign * q, m=q, cell=cell[o], off=off[:, o], u=u[:, o]))
        del u, gam, key, o, cell
    return species, _fields(g, case, q, mean)


def _fields(g, case, q=0.0, mean=1.0):
    """Smooth field planes: a guide field along z for the turbulence, and a few low modes."""
    N, dim = (case["nx"], case["ny"], case["nz"]), case["dim"]
    F = torch.zeros((9, N[2], N[1], N[0]), device=DEV)
    b0 = math.sqrt(10.0 * case.get("ppc", 1) * q * C * C * mean * 2.0)
    b0 *= 1.0 if case.get("setup") == "turbulence" else 0.1
    x = [torch.arange(N[d], device=DEV, dtype=torch.float32) * (2.0 * math.pi / N[d]) for d in range(3)]
    r = torch.rand((6, 3, 5), generator=g, device=DEV).cpu().numpy()
    for c in range(6):
        amp = b0 * (0.1 if c < 3 else 0.4)
        for a, p, *m in r[c]:
            k = [1 + int(3 * v) if d < dim else 0 for d, v in enumerate(m)]
            F[c] += amp * float(a) * torch.cos(k[0] * x[0][None, None, :] + k[1] * x[1][None, :, None] +
                                               k[2] * x[2][:, None, None] + 6.3 * float(p))
    if case.get("setup") == "turbulence":
        F[5] += b0
    return F


class Box:
    """A run as a user's program holds it: the caller's buffers, in one allocation, and the library's context."""

    def __init__(self, case, species, fields, flat=None):
        self.dim, self.plane = case["dim"], fields[0].numel()
        caps = [(s["cell"].numel() + 3) // 4 * 4 for s in species]
        self.words = (9 * self.plane + 3) // 4 * 4 + sum(c * (4 + self.dim) for c in caps)
        self.flat = torch.zeros(self.words, device=DEV) if flat is None else flat
        self.fields = self.flat[:9 * self.plane].view(fields.shape)
        self.fields.copy_(fields)
        self.species, at = [], (9 * self.plane + 3) // 4 * 4
        for s, cap in zip(species, caps):
            n, D = s["cell"].numel(), self.dim
            d = dict(q=s["q"], m=s["m"], n=n, cap=cap, cell=self.flat[at:at + cap].view(torch.int32),
                     off=self.flat[at + cap:at + cap * (1 + D)].view(D, cap),
                     u=self.flat[at + cap * (1 + D):at + cap * (4 + D)].view(3, cap))
            for k in ("cell", "off", "u"):
                d[k][..., :n].copy_(s[k])
            self.species.append(d)
            at += cap * (4 + D)
        self.given = self.flat.clone()  # in the order the program made them in: the library sorts its buffers now
        self.stream = torch.cuda.current_stream()
        sps = [B.pic_species(d["q"], d["m"], d["n"], d["cell"].data_ptr(), d["off"].data_ptr(), d["u"].data_ptr(),
                             d["cap"]) for d in self.species]
        self.ctx = B.pic_init(B.pic_grid(case["dim"], case["nx"], case["ny"], case["nz"]), sps, C, 1.0,
                              self.fields.data_ptr(), self.stream.cuda_stream)
        t = B.pic_tuning()
        t.filter_passes = case.get("passes", 0)
        if case.get("tuning") == "16x8h4":
            t.tile[0], t.tile[1], t.halo = 16, 8, 4
        B.pic_set_tuning(self.ctx, t)
        if case.get("order", 2) == 4:
            B.pic_set_field_solver(self.ctx, 4)
        if case.get("pusher") == "higuera_cary":
            B.pic_set_pusher(self.ctx, B.PIC_PUSHER_HIGUERA_CARY)
        if case.get("setup") == "wall":
            sh = B.pic_shock()  # the injector stands still: the upstream has ended
            sh.wall, sh.lt, sh.x0, sh.x_max, sh.v_inj, sh.v_up = WALL, 4, case["nx"] - 3.0, case["nx"] - 3.0, 0.0, 0.0
            B.pic_set_shock(self.ctx, sh)
            self.given[:9 * self.plane] = self.flat[:9 * self.plane]  # with the wall's boundary values

    def out(self):
        return {"E": self.fields[0:3], "B": self.fields[3:6], "J": self.fields[6:9]}

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            torch.cuda.synchronize()
            B.pic_destroy(self.ctx)
            self.ctx = None


def _ensemble(case, seed):
    """Boxes of the batch, as case dicts: half 1D, half 2D, sizes uniform in their logarithm."""
    r = np.random.RandomState(int(seed) % (1 << 31))
    sizes = np.random.RandomState(case["boxes"] * 1009 + case["n1_max"] + 7 * case["n2_max"])  # not the seed's
    boxes = []
    for b in range(case["boxes"]):
        dim = 1 + b % 2
        lo, hi = (128, case["n1_max"]) if dim == 1 else (32, case["n2_max"])
        n = int(round(math.exp(sizes.uniform(math.log(lo), math.log(hi)))))
        ppc = 2 * int(round(math.exp(sizes.uniform(math.log(8), math.log(case["ppc_max"] / 2)))))
        boxes.append((dict(dim=dim, nx=n, ny=n if dim == 2 else 1, nz=1, ppc=ppc, setup="weibel", passes=0, order=2,
                           pusher="boris"), int(r.randint(1 << 30))))
    return boxes


def _adjoint_inputs(case, seed):
    """The differentiable box: species, base fields (guide field), mode fields [M, 3, 1, ny, nx] (lattice curls of a
    vector potential) and their amplitudes."""
    g = _gen(seed)
    box = dict(dim=2, nx=case["nx"], ny=case["ny"], nz=1, ppc=case["ppc"], setup="turbulence")
    species, F = _plasma(g, box)
    q, mean = _charge("turbulence", case["ppc"])
    b0 = math.sqrt(case["ppc"] * q * C * C * mean * 2.0)
    F.zero_()
    F[5] = b0
    nx, ny, M = case["nx"], case["ny"], case["modes"]
    ph = torch.rand((M, M, 2), generator=g, device=DEV, dtype=torch.float64) * (2.0 * math.pi)
    i = torch.arange(nx, device=DEV, dtype=torch.float64) * (2.0 * math.pi / nx)
    j = torch.arange(ny, device=DEV, dtype=torch.float64) * (2.0 * math.pi / ny)
    modes = torch.zeros((M * M, 3, 1, ny, nx), device=DEV)
    for a in range(M):
        for b in range(M):
            K = math.hypot(a + 1, b + 1)
            az = nx / (2.0 * math.pi * K) * torch.outer(torch.sin((b + 1) * j + ph[a, b, 1]),
                                                        torch.sin((a + 1) * i + ph[a, b, 0]))
            modes[a * M + b, 0, 0] = az.roll(-1, 0) - az
            modes[a * M + b, 1, 0] = -(az.roll(-1, 1) - az)
    amps = 0.1 * b0 / M * torch.randn(M * M, generator=g, device=DEV)
    return species, F, modes, amps


def prepare(case, seed):
    kind = case["kind"]
    if kind == "filter":
        g = _gen(seed)
        N = (case["nx"], case["ny"], case["nz"])
        F = torch.zeros((9, N[2], N[1], N[0]), device=DEV)
        F[6:] = torch.randn((3, N[2], N[1], N[0]), generator=g, device=DEV)
        if case["static"]:
            return dict(kind=kind, static=True, J=F[6:].clone(), passes=case["passes"], grid=B.pic_grid(case["dim"], *N),
                        stream=torch.cuda.current_stream())
        none = dict(q=1.0, m=1.0, cell=torch.zeros(0, dtype=torch.int32, device=DEV),
                    off=torch.zeros((case["dim"], 0), device=DEV), u=torch.zeros((3, 0), device=DEV))
        return dict(kind=kind, static=False, box=Box(dict(case, passes=0), [none], F), passes=case["passes"])
    if kind == "batch":
        cases = _ensemble(case, seed)
        made = [_plasma(_gen(s), c) for c, s in cases]
        words = [(9 * f[0].numel() + 3) // 4 * 4 + sum((s["cell"].numel() + 3) // 4 * 4 * (4 + c["dim"]) for s in sp)
                 for (c, _), (sp, f) in zip(cases, made)]
        flat, at, boxes = torch.zeros(sum(words), device=DEV), 0, []
        given = torch.empty_like(flat)
        for (c, _), (sp, f), w in zip(cases, made, words):
            boxes.append(Box(c, sp, f, flat[at:at + w]))
            given[at:at + w] = boxes[-1].given
            boxes[-1].given = None
            at += w
        st = dict(kind=kind, boxes=boxes, flat=flat, given=given, steps=case["steps"])
        st["batch"] = Handle(B.pic_batch_create([b.ctx for b in boxes]), boxes)
        return st
    if kind == "adjoint":
        from paper_1906_06306_gb300 import Simulation
        from paper_1906_06306_gb300.adjoint import MagneticEnergyProblem

        species, F, modes, amps = _adjoint_inputs(case, seed)
        host = [dict(q=s["q"], m=s["m"], **{k: s[k].cpu().numpy() for k in ("cell", "off", "u")}) for s in species]
        sim = Simulation(2, case["nx"], case["ny"], 1, C, F.cpu().numpy(), host, device=DEV)
        for d, s in zip(sim.species, species):  # the slots in the program's own order
            for k in ("cell", "off", "u"):
                d[k][..., :d["n"]].copy_(s[k])
        problem = MagneticEnergyProblem(sim, modes.cpu().numpy(), case["steps"], checkpoint_every=case["every"])
        return dict(kind=kind, problem=problem, amps=amps, u0=problem.u0())
    g = _gen(seed)
    box = Box(case, *_plasma(g, case))
    st = dict(kind=kind, box=box)
    if kind == "step":
        st["steps"] = case["steps"]
        # a run that is under way, at the start of a sort cycle
        B.pic_step(box.ctx, B.pic_get_tuning(box.ctx).sort_every)
    if kind == "restart":  # the grouping that the checkpoint keeps, inside a bin in the program's order
        box.flat.copy_(box.given)
        bins = B.pic_sort_bins(box.ctx)
        perm = [torch.empty(d["n"], dtype=torch.int32, device=DEV) for d in box.species]
        start = [torch.empty(bins + 1, dtype=torch.int32, device=DEV) for _ in box.species]
        B.pic_sort_record(box.ctx, [p.data_ptr() for p in perm], [t.data_ptr() for t in start])
        box.flat.copy_(box.given)
        for d, p, t in zip(box.species, perm, start):
            n = d["n"]
            at = torch.searchsorted(t[1:].contiguous(), torch.arange(n, device=DEV, dtype=torch.int32), right=True)
            o = p[torch.argsort(at * n + p)].to(torch.int64)
            for k in ("cell", "off", "u"):
                d[k][..., :n] = d[k][..., :n][..., o]
        box.given = box.flat.clone()
        st["start"] = start
    if kind in ("live", "energies"):  # these don't restart
        box.flat.copy_(box.given)
        box.given = None
        B.pic_sort(box.ctx)
    return st


class Handle:
    def __init__(self, h, boxes):
        self.h, self.boxes = h, boxes

    def __del__(self):
        torch.cuda.synchronize()
        B.pic_batch_destroy(self.h)


def run(st):
    kind = st["kind"]
    if kind == "step":
        box = st["box"]
        box.flat.copy_(box.given)
        B.pic_step(box.ctx, st["steps"])
        return box.out()
    if kind == "live":
        B.pic_step(st["box"].ctx, 1)
        return st["box"].out()
    if kind == "restart":
        box = st["box"]
        box.flat.copy_(box.given)
        B.pic_sort_assume(box.ctx, [t.data_ptr() for t in st["start"]])
        B.pic_step(box.ctx, 1)
        return dict(box.out(), particles=[{k: d[k][..., :d["n"]] for k in ("cell", "off", "u")} for d in box.species])
    if kind == "filter":
        if st["static"]:
            B.pic_filter_current_static(st["grid"], st["J"].data_ptr(), st["passes"], st["stream"].cuda_stream)
            return st["J"]
        B.pic_filter_current(st["box"].ctx, st["passes"])
        return st["box"].fields[6:9]
    if kind == "energies":
        return B.pic_energies(st["box"].ctx, 2)
    if kind == "adjoint":
        loss = st["problem"].run(st["amps"], st["u0"])
        g_amps, g_u0 = st["problem"].gradient()
        return {"loss": np.float32(loss), "amps": g_amps, "u0": g_u0}
    st["flat"].copy_(st["given"])
    B.pic_batch_step(st["batch"].h, st["steps"], st["boxes"][0].stream.cuda_stream)
    return [b.fields for b in st["boxes"]]


def work(case):
    """Per step: every particle record read and written (4 + 4 D + 12 bytes each way) and the nine planes read and
    written; the filter's and the diagnostics' own reads and writes.  Operations: about 250 a particle in 2D."""
    kind = case["kind"]

    def step(c):
        cells, D = c["nx"] * c["ny"] * c["nz"], c["dim"]
        n = 2 * cells * c["ppc"]
        return n * 2 * (16 + 4 * D) + cells * 72, n * (120 + 65 * D) + cells * (40 + 15 * c.get("passes", 0))

    if kind == "filter":
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 24 * cells, "flops": 15 * case["dim"] * case["passes"] * cells}
    if kind == "energies":
        cells = case["nx"] * case["ny"] * case["nz"]
        n = 2 * cells * case["ppc"]
        return {"bytes": n * (16 + 4 * case["dim"]) + 24 * cells, "flops": n * (20 + 4 * 2 ** case["dim"])}
    if kind == "batch":
        w = [step(c) for c, _ in _ensemble(case, 0)]
        return {"bytes": case["steps"] * sum(b for b, _ in w), "flops": case["steps"] * sum(f for _, f in w)}
    if kind == "adjoint":
        b, f = step(dict(case, nz=1, dim=2))
        # forward as above; reverse: the forward record read, the five gradient rows read and written
        n = 2 * case["nx"] * case["ny"] * case["ppc"]
        return {"bytes": case["steps"] * (b + n * (24 + 40) + case["nx"] * case["ny"] * 96), "flops": case["steps"] * 4 * f}
    b, f = step(case)
    return {"bytes": case.get("steps", 1) * b, "flops": case.get("steps", 1) * f}


# ------------------------------------------------------------------------------------------------ the same in 64 bits

STAG = (1, 2, 4, 6, 5, 3)  # bit d: the component sits half a cell up axis d
CHUNK = 1 << 22  # particles at a time


class Exact:
    """The step in plain torch, float64: fields [6 or 9 planes], particles as integer cells and offsets."""

    def __init__(self, case, species, fields):
        self.D, self.N = case["dim"], (case["nx"], case["ny"], case["nz"])
        self.c = float(np.float32(C))
        self.order, self.hc, self.passes = case.get("order", 2), case.get("pusher") == "higuera_cary", case.get("passes", 0)
        self.wall = WALL if case.get("setup") == "wall" else 0
        self.i_zero = self.N[0] - 1 if self.wall else 0
        F = fields.double()
        self.E, self.B, self.J = [F[k] for k in range(3)], [F[k] for k in range(3, 6)], [F[k] for k in range(6, 9)]
        self.sp = []
        for s in species:
            r, ijk = s["cell"].long(), []
            for d in range(self.D):
                ijk.append(r % self.N[d])
                r = torch.div(r, self.N[d], rounding_mode="floor")
            self.sp.append(dict(q=float(np.float32(s["q"])), m=float(np.float32(s["m"])), ijk=ijk,
                                off=[s["off"][d].double() for d in range(self.D)], u=[s["u"][a].double() for a in range(3)]))
        if self.wall:
            self.bc()

    def diff(self, A, d, up):
        """Staggered difference along axis d, at the points half a cell up (or down)."""
        if d >= self.D:
            return torch.zeros_like(A)
        ax, s = 2 - d, (-1 if up else 1)
        if self.order == 2:
            return A.roll(s, ax) - A if up else A - A.roll(s, ax)
        if up:
            return 9.0 / 8.0 * (A.roll(-1, ax) - A) - (A.roll(-2, ax) - A.roll(1, ax)) / 24.0
        return 9.0 / 8.0 * (A - A.roll(1, ax)) - (A.roll(-1, ax) - A.roll(2, ax)) / 24.0

    def curl(self, A, up):
        f = lambda a, d: self.diff(A[a], d, up)  # noqa: E731
        return [f(2, 1) - f(1, 2), f(0, 2) - f(2, 0), f(1, 0) - f(0, 1)]

    def b_half(self):
        r = self.curl(self.E, True)
        self.B = [b - 0.5 * self.c * x for b, x in zip(self.B, r)]
        self.bc()

    def e_update(self):
        r = self.curl(self.B, False)
        self.E = [e + self.c * x - j for e, x, j in zip(self.E, r, self.J)]
        self.bc()

    def bc(self):
        """The conductor's images about x = wall and the zero region past the injector."""
        if not self.wall:
            return
        w = self.wall
        i = torch.arange(w, device=DEV)
        planes = self.E + self.B
        for k, A in enumerate(planes):
            A = planes[k] = A.clone()
            integer = k in (1, 2, 3)  # integer-x points: Ey, Ez, Bx, odd about the wall
            A[..., :w] = -A[..., 2 * w - i] if integer else A[..., 2 * w - 1 - i]
            if k in (1, 2):
                A[..., w] = 0.0
            A[..., self.i_zero:] = 0.0
        self.E, self.B = planes[:3], planes[3:]

    def smooth(self, A):
        for d in range(self.D):
            A = 0.25 * A.roll(1, 2 - d) + 0.5 * A + 0.25 * A.roll(-1, 2 - d)
        return A

    def flat(self, at):
        r = torch.zeros_like(at[0])
        for d in reversed(range(self.D)):
            r = r * self.N[d] + at[d] % self.N[d]
        return r

    def gather(self, A, stag, ijk, off):
        base, w = [], []
        for d in range(self.D):
            if stag >> d & 1:
                up = (off[d] >= 0.5)
                base.append(ijk[d] - 1 + up.long())
                w.append(torch.where(up, off[d] - 0.5, off[d] + 0.5))
            else:
                base.append(ijk[d])
                w.append(off[d])
        v, A = 0.0, A.reshape(-1)
        for k in range(1 << self.D):
            t, at = 1.0, []
            for d in range(self.D):
                up = k >> d & 1
                t = t * (w[d] if up else 1.0 - w[d])
                at.append(base[d] + up)
            v = v + t * A[self.flat(at)]
        return v

    def push(self, u, e, b, qm):
        c, h = self.c, 0.5 * qm
        cross = lambda p, r: [p[1] * r[2] - p[2] * r[1], p[2] * r[0] - p[0] * r[2], p[0] * r[1] - p[1] * r[0]]  # noqa: E731
        dot = lambda p, r: p[0] * r[0] + p[1] * r[1] + p[2] * r[2]  # noqa: E731
        u1 = [c * u[a] + h * e[a] for a in range(3)]
        g2 = 1.0 + dot(u1, u1) / (c * c)
        tau = [h / c * x for x in b]
        if self.hc:
            us, tt = dot(u1, tau) / c, dot(tau, tau)
            s = g2 - tt
            r = torch.sqrt(s * s + 4.0 * (tt + us * us))
            gp = torch.sqrt(torch.where(s >= 0, 0.5 * (s + r), 2.0 * (tt + us * us) / (r - s).clamp(min=1e-300)))
            t = [x / gp for x in tau]
            f, ut = 1.0 / (1.0 + dot(t, t)), dot(u1, t)
            x = cross(u1, t)
            m = [f * (u1[a] + ut * t[a] + x[a]) for a in range(3)]
            x = cross(m, t)
            return [(m[a] + x[a] + h * e[a]) / c for a in range(3)]
        t = [x / torch.sqrt(g2) for x in tau]
        f, x = 2.0 / (1.0 + dot(t, t)), cross(u1, t)
        x = cross([f * (u1[a] + x[a]) for a in range(3)], t)
        return [(u1[a] + x[a] + h * e[a]) / c for a in range(3)]

    def segment(self, J, ijk, Dl, W, q):
        """The ZigZag current of one segment in the cell ijk: displacement Dl, weights W from its lower corner."""
        D = self.D
        for a in range(3):
            t = [d for d in range(D) if d != a]
            for k in range(1 << len(t)):
                w, at = 1.0, list(ijk)
                for p, d in enumerate(t):
                    up = k >> p & 1
                    w = w * (W[d] if up else 1.0 - W[d])
                    at[d] = at[d] + up
                if D == 3:  # the product's average along the straight segment
                    w = w + (1.0 if k in (0, 3) else -1.0) * Dl[t[0]] * Dl[t[1]] / 12.0
                J[a] = J[a].index_add(0, self.flat(at), q * Dl[a] * w)

    def zigzag(self, J, ijk, o1, dc, o2, dn, q):
        D = self.D
        D1, D2, W1, W2 = [], [], [], []
        for d in range(3):
            if d >= D:
                D1.append(0.5 * dn[d])
                D2.append(0.5 * dn[d])
                continue
            k = dc[d].double()
            x1, x2 = o1[d], k + o2[d]
            xr = torch.minimum(k.clamp(max=0.0) + 1.0, torch.maximum(k.clamp(min=0.0), 0.5 * (x1 + x2)))
            D1.append(xr - x1)
            D2.append(x2 - xr)
            W1.append(0.5 * (x1 + xr))
            W2.append(0.5 * (x2 + xr) - k)
        self.segment(J, ijk, D1, W1, q)
        self.segment(J, [ijk[d] + dc[d] for d in range(D)], D2, W2, q)

    def particles(self, J, s, ijk, off, u):
        D, c = self.D, self.c
        e = [self.gather(self.E[a], STAG[a], ijk, off) for a in range(3)]
        b = [self.gather(self.B[a], STAG[3 + a], ijk, off) for a in range(3)]
        u = self.push(u, e, b, s["q"] / s["m"])
        gam = torch.sqrt(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
        dn = [c * x / gam for x in u]
        o2 = [off[d] + dn[d] for d in range(D)]
        dc = [torch.floor(x.detach()).long() for x in o2]
        o2 = [x - k for x, k in zip(o2, dc)]
        if not self.wall:
            self.zigzag(J, ijk, off, dc, o2, dn, s["q"])
            return [(ijk[d] + dc[d]) % self.N[d] for d in range(D)], o2, u
        # reflection at x = wall: straight to the plane, then the mirror image of the rest
        hit = ijk[0] + dc[0] < self.wall
        m = ~hit
        pick = lambda v, k: [x[k] for x in v]  # noqa: E731
        self.zigzag(J, pick(ijk, m), pick(off, m), pick(dc, m), pick(o2, m), pick(dn, m), s["q"])
        i, a, k, z, w = (pick(v, hit) for v in (ijk, off, dc, o2, dn))
        f = a[0] / (a[0] + 1.0 - z[0])
        mid = [torch.zeros_like(a[0])] + [a[d] + f * (k[d] + z[d] - a[d]) for d in range(1, D)]
        km = [torch.zeros_like(k[0])] + [torch.minimum(torch.maximum(torch.floor(mid[d]).long(), k[d].clamp(max=0)),
                                                       k[d].clamp(min=0)) for d in range(1, D)]
        zm = [mid[d] - km[d] for d in range(D)]
        self.zigzag(J, i, a, km, zm, [f * x for x in w], s["q"])
        end = [1.0 - z[0]] + [z[d] for d in range(1, D)]
        ke = [torch.zeros_like(k[0])] + [k[d] - km[d] for d in range(1, D)]
        self.zigzag(J, [i[d] + km[d] for d in range(D)], zm, ke, end, [(1.0 - f) * x for x in w], s["q"])
        new = [(ijk[d] + dc[d]) % self.N[d] for d in range(D)]
        new[0] = torch.where(hit, ijk[0], new[0])
        o2[0] = torch.where(hit, 1.0 - o2[0], o2[0])
        u[0] = torch.where(hit, -u[0], u[0])
        return new, o2, u

    def step(self, n=1):
        for _ in range(n):
            self.b_half()
            J = [torch.zeros_like(self.E[0]).reshape(-1) for _ in range(3)]
            for s in self.sp:
                total = s["u"][0].numel()
                if total <= CHUNK:
                    s["ijk"], s["off"], s["u"] = self.particles(J, s, s["ijk"], s["off"], s["u"])
                    continue
                for lo in range(0, total, CHUNK):
                    r = slice(lo, lo + CHUNK)
                    got = self.particles(J, s, *([v[r] for v in s[k]] for k in ("ijk", "off", "u")))
                    for k, v in zip(("ijk", "off", "u"), got):
                        for x, y in zip(s[k], v):
                            x[r] = y
            self.J = [x.view(self.E[0].shape) for x in J]
            self.b_half()
            for _ in range(self.passes):
                self.J = [self.smooth(x) for x in self.J]
            self.e_update()

    def out(self):
        return {"E": torch.stack(self.E), "B": torch.stack(self.B), "J": torch.stack(self.J)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "filter":
        N = (case["nx"], case["ny"], case["nz"])
        x = Exact(dict(case, setup="none"), [], torch.zeros((9, N[2], N[1], N[0]), device=DEV))
        g = _gen(seed)
        J = torch.randn((3, N[2], N[1], N[0]), generator=g, device=DEV).double()
        r = []
        for A in J:
            for _ in range(case["passes"]):
                A = x.smooth(A)
            r.append(A)
        return torch.stack(r)
    if kind == "batch":
        r = []
        for c, s in _ensemble(case, seed):
            x = Exact(c, *_plasma(_gen(s), c))
            x.step(case["steps"])
            o = x.out()
            r.append(torch.cat([o["E"], o["B"], o["J"]]))
        return r
    if kind == "adjoint":
        species, F, modes, amps = _adjoint_inputs(case, seed)
        a = amps.double().requires_grad_(True)
        u0 = torch.cat([s["u"] for s in species], 1).double().requires_grad_(True)
        x = Exact(dict(case, dim=2, nz=1), species, F)
        x.B = [b + (a[:, None, None, None] * modes[:, k].double()).sum(0) for k, b in enumerate(x.B)]
        at = 0
        for s in x.sp:
            n = s["u"][0].numel()
            s["u"] = [u0[k, at:at + n] for k in range(3)]
            at += n
        x.step(case["steps"])
        loss = 0.5 * sum((b * b).sum() for b in x.B)
        loss.backward()
        return {"loss": loss.detach(), "amps": a.grad, "u0": u0.grad}
    species, F = _plasma(_gen(seed), case)
    if kind == "energies":
        x = Exact(case, species, F)
        r = [0.5 * sum(float((f * f).sum()) for f in A) for A in (x.E, x.B)]
        rho = torch.zeros(F[0].numel(), dtype=torch.float64, device=DEV)
        for s in x.sp:
            u2 = s["u"][0] ** 2 + s["u"][1] ** 2 + s["u"][2] ** 2
            r.append(s["m"] * x.c ** 2 * float((u2 / (torch.sqrt(1.0 + u2) + 1.0)).sum()))
            for k in range(1 << x.D):
                w, at = s["q"], []
                for d in range(x.D):
                    up = k >> d & 1
                    w = w * (s["off"][d] if up else 1.0 - s["off"][d])
                    at.append(s["ijk"][d] + up)
                rho.index_add_(0, x.flat(at), w)
        rho = rho.view(F[0].shape)
        for _ in range(x.passes):
            rho = x.smooth(rho)
        x.order = 2
        res = sum(x.diff(x.E[d], d, False) for d in range(x.D)) - rho
        return r + [float(res.abs().max()), float(torch.sqrt((res * res).mean()))]
    if kind == "restart":
        # each particle's slot in a grouped array depends on the library's bins: the fields alone
        x = Exact(case, species, F)
        x.step(1)
        return dict(x.out(), particles=[{"cell": None, "off": None, "u": None} for _ in species])
    x = Exact(case, species, F)
    x.step(case.get("steps", 1))
    return x.out()
