"""pic_energies against the same sums in extended precision: kinetic terms from
double-float arithmetic, charge from fixed-point cell moments per tile."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

SHAPES = {1: (70, 1, 1), 2: (37, 50, 1), 3: (19, 10, 9)}


def _sim(dim, shape, ppc, seed, **kw):
    from paper_1906_06306_gb300 import Simulation

    pl = workloads.uniform_plasma(dim, *shape, 0.45, ppc, 0.01, 0.5, seed=seed)
    rs = np.random.default_rng(seed)
    pl.fields[:6] = rs.normal(size=pl.fields[:6].shape) * 10.0 ** rs.integers(-6, 3, size=pl.fields[:6].shape)
    return pl, Simulation.from_plasma(pl, **kw)


def _reference(dim, shape, c, fields, species):
    """(energies, charge scale) in numpy's extended precision."""
    L = np.longdouble
    F = fields.astype(L)
    out = [0.5 * (F[:3] ** 2).sum(), 0.5 * (F[3:6] ** 2).sum()]
    n = np.array(shape)
    rho = np.zeros(shape[::-1], dtype=L)
    top = np.zeros(shape[::-1], dtype=L)
    for s in species:
        u2 = (s["u"].astype(L) ** 2).sum(0)
        out.append(L(np.float32(s["m"])) * L(np.float32(c)) ** 2 * (u2 / (np.sqrt(1 + u2) + 1)).sum())
        cell = s["cell"].astype(np.int64)
        ijk = [cell % n[0], cell // n[0] % n[1], cell // (n[0] * n[1])]
        for corner in range(1 << dim):
            w, at = L(1.0), []
            for d in range(3):
                up = d < dim and corner >> d & 1
                if d < dim:
                    o = s["off"][d].astype(L)
                    w = w * (o if up else 1 - o)
                at.append((ijk[d] + up) % n[d])
            np.add.at(rho, tuple(at[::-1]), L(np.float32(s["q"])) * w)
            np.add.at(top, tuple(at[::-1]), abs(L(np.float32(s["q"]))) * w)
    div = sum(F[d] - np.roll(F[d], 1, axis=2 - d) for d in range(dim))
    res = div - rho
    return out + [abs(res).max(), np.sqrt((res * res).mean())], float(top.max())


def _check(sim, pl, species):
    F = sim.fields.cpu().numpy()
    ref, top = _reference(sim.dim, (sim.nx, sim.ny, sim.nz), sim.c, F, species)
    got = sim.energies()
    ns = len(species)
    # field and kinetic terms: below 2^-44 of each term, plus an FP64 sum in
    # some order (at most 40 roundings deep: blocks of sums)
    for a, b in zip(got[:2 + ns], ref[:2 + ns]):
        assert abs(a - float(b)) <= (2.0 ** -44 + 40 * 2.0 ** -53) * abs(float(b))
    # the residual: each particle's weights below 2^-46, and FP64 sums of the
    # divergence's six terms and the charges
    scale = top + 6 * float(np.abs(F[:3]).max())
    for a, b in zip(got[2 + ns:], ref[2 + ns:]):
        assert abs(a - float(b)) <= 2.0 ** -46 * scale


@pytest.mark.parametrize("dim,ppc", [(1, 3), (1, 400), (2, 1), (2, 40), (3, 3)])
def test_energies_match_extended_precision(dim, ppc):
    pl, sim = _sim(dim, SHAPES[dim], ppc, seed=70 + dim)
    _check(sim, pl, sim.download()[1])
    sim.close()


def test_more_particles_of_a_tile_than_a_fold_takes():
    # one tile of 8 x 8 cells with 70,000 particles of a species, most of them in one cell
    pl, sim = _sim(2, (8, 8, 1), 1100, seed=75)
    for d in sim.species:
        d["cell"][: d["n"] - 300] = 27
    sim.sort()
    _check(sim, pl, sim.download()[1])
    sim.close()


@pytest.mark.parametrize("dim", [1, 2])
def test_extreme_offsets_speeds_and_particles_outside_their_window(dim):
    import torch

    pl, sim = _sim(dim, SHAPES[dim], 12, seed=80 + dim, tuning=dict(tile=[8, 8][:dim] + [1] * (2 - dim)))
    offs = [0.0, 1.0 - 2.0 ** -24, 2.0 ** -24, 2.0 ** -26, 2.0 ** -48, 2.0 ** -60, 1e-40, 0.5, -0.0]
    us = [0.0, 1e-30, 2.0 ** -41, 2.0 ** -39, 1.0, 1e6, 2.0 ** 59, 2.0 ** 61, 1e25]
    for d in sim.species:
        k = torch.arange(d["n"], device=sim.device)
        for a in range(dim):
            d["off"][a, :d["n"]] = torch.tensor(offs, device=sim.device)[(k // 9 ** a) % 9]
        # most particles away from the tile that their slot is in
        d["cell"][:d["n"]] = torch.roll(d["cell"][:d["n"]], d["n"] // 3)
    _check(sim, pl, sim.download()[1])
    for u in us:  # one magnitude at a time: larger ones would hide the rest
        for d in sim.species:
            d["u"].fill_(u)
            d["u"][1] *= -0.3
        _check(sim, pl, sim.download()[1])
    sim.close()


def test_injected_particles_after_the_last_sort_count():
    from paper_1906_06306_gb300 import Simulation

    pl = workloads.shock_tube(dim=2, nx=48, ny=8, nz=1, ppc=3, gamma_flow=3.0, theta=0.05, r_p=3.0,
                              wall=3, x_inj=20, x_max=40.0, lt=8, seed=93)
    cap = [s.n + workloads.injected_count(pl, 6) for s in pl.species]
    sim = Simulation.from_plasma(pl, capacity=cap, tuning=dict(sort_every=1000))
    sim.set_shock_from_plasma(pl)
    sim.step(5)
    assert sim.counts()[0] > pl.species[0].n
    got = sim.energies()
    ref, _ = _reference(2, (48, 8, 1), sim.c, sim.fields.cpu().numpy(), sim.download()[1])
    for a, b in zip(got[:4], ref[:4]):
        assert abs(a - float(b)) <= (2.0 ** -44 + 40 * 2.0 ** -53) * abs(float(b))
    sim.close()
