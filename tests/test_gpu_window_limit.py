"""The largest tile windows that pic_set_tuning accepts (200 KB of shared memory
with a stray queue of 512 entries), and both lengths of that queue when full."""
import numpy as np
import pytest

import workloads
from gpu_helpers import compare_fields, compare_particles, oracle_from_sim, step_floor, term_floor

pytestmark = pytest.mark.gpu

# (dim, box, largest accepted tile, halo, the next larger one): 14 words a window cell in
# 1D, 12 in 2D, and 512 words, in 51,200
WINDOWS = [(1, (4000, 1, 1), (3613, 1, 1), 3, (3614, 1, 1)),
           (2, (90, 100, 1), (55, 57, 1), 4, (56, 57, 1))]


@pytest.mark.parametrize("dim,n,tile,halo,larger", WINDOWS)
def test_largest_window_is_accepted_and_steps(dim, n, tile, halo, larger):
    import oracle
    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    pl = workloads.uniform_plasma(dim, *n, 0.45, 6, 0.01, 0.5, seed=11)
    sim = Simulation.from_plasma(pl)
    with pytest.raises(B.PicError):
        sim.set_tuning(tile=larger, halo=halo)
    sim.set_tuning(tile=tile, halo=halo, sort_every=1000)
    sim.sort()
    g, F, osp, _ = oracle_from_sim(sim)
    floor = step_floor(g, osp, 2)
    sim.step(2)
    sim.check()
    oracle.step(g, F, osp, nsteps=2)
    compare_fields(sim.download()[0], F, floor=floor)
    sim.close()


# 512 entries: with 1024, three blocks instead of four would fit an SM (a window of 33 x 34 cells)
@pytest.mark.parametrize("n,tile,halo", [((160, 160, 1), (16, 16, 1), 3), ((90, 93, 1), (30, 31, 1), 1)])
def test_more_strays_than_the_queue_holds(n, tile, halo):
    import torch

    import oracle
    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    # some 900 particles of a species to a block or more, nearly all of them outside its window
    pl = workloads.uniform_plasma(2, *n, 0.45, 64, 1e-4, 0.3, seed=12)
    sim = Simulation.from_plasma(pl, tuning=dict(tile=tile, halo=halo, sort_every=1000))
    sim.sort()
    for d in sim.species:
        d["cell"][:d["n"]] = torch.roll(d["cell"][:d["n"]], d["n"] // 2)
    g, F, osp, _ = oracle_from_sim(sim)
    B.pic_stats(sim.ctx)
    terms = []
    sim.step(1)
    oracle.step(g, F, osp, terms=terms)
    assert B.pic_stats(sim.ctx) > 0.8 * sum(s.n for s in osp)
    sim.check()
    Fg, spg = sim.download()
    compare_fields(Fg, F, floor=term_floor(g, terms))
    compare_particles(g, spg, osp)
    sim.close()
