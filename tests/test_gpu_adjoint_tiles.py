"""The adjoint's tile pass at the edges of its window's geometry, against the
global-memory pass on the same particles (which other tests hold against the
oracle; both take a particle's branches, the relay point and the half cell,
from the same float32 values, so no particle on a branch point separates
them): sums added to the lattice by aligned quads or, where
the rows or the caller's planes do not allow it, word by word; boxes shorter
than a window; several blocks to a tile; gradients of very different size
(the fixed-point quantum follows them)."""
import numpy as np
import pytest

import workloads

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu

CASES = [
    # dim, (nz, ny, nx), tile, halo, words before A's first plane, scale
    (1, (1, 1, 24), 8, 1, 0, 1.0),
    (2, (1, 12, 16), 4, 1, 0, 1.0),       # quads
    (2, (1, 12, 16), 4, 1, 1, 1.0),       # A not 16-byte aligned: words
    (2, (1, 12, 18), 4, 2, 0, 1.0),       # rows not whole quads: words
    (2, (1, 8, 8), 8, 2, 0, 1.0),         # window wider than the box, quads
    (2, (1, 7, 9), 8, 2, 0, 1.0),         # the same, words
    (2, (1, 12, 16), 8, 1, 0, 2.0 ** -66),
    (2, (1, 12, 16), 8, 1, 0, 2.0 ** 66),
    (3, (6, 7, 8), 4, 1, 0, 1.0),         # quads
    (3, (6, 6, 7), 4, 1, 0, 1.0),         # words
    (3, (4, 4, 4), 4, 1, 0, 1.0),         # window wider than the box
]


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


@pytest.mark.parametrize("dim,shape,tile,halo,lead,scale", CASES)
def test_tile_pass_matches_the_global_pass(dim, shape, tile, halo, lead, scale):
    # float32 chain and sums, terms rounded to 2^-22 of their batch's largest:
    # a few 1e-6 of the largest gradient, the bound 2e-5 of the other adjoint tests
    import torch

    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    nz, ny, nx = shape
    rs = np.random.default_rng(900 + 7 * nx + ny + lead)
    pl = workloads.uniform_plasma(dim, nx, ny, nz, 0.45, 60 if dim < 3 else 12, 0.02, 0.2, 900 + nx)
    pl.fields[:6] = random_fields(shape, rs)[:6]
    sim = Simulation.from_plasma(pl, tuning=dict(sort_every=1 << 30, filter_passes=0,
                                                 tile=[tile] * 3, halo=halo))
    nb, counts = B.pic_sort_bins(sim.ctx), sim.counts()
    perm = [torch.empty(n, dtype=torch.int32, device=sim.device) for n in counts]
    tst = [torch.empty(nb + 1, dtype=torch.int32, device=sim.device) for _ in counts]
    B.pic_sort_record(sim.ctx, [p.data_ptr() for p in perm], [t.data_ptr() for t in tst])
    sim.step(2)
    A = torch.from_numpy((scale * rs.normal(size=(9,) + shape)).astype(np.float32)).cuda()
    A[6:9] = 0.0
    rows = []
    for k in (dim, 3):
        for d in sim.species:
            r = torch.zeros((k, d["cap"]), dtype=torch.float32)
            r[:, : d["n"]] = torch.from_numpy((scale * rs.normal(size=(k, d["n"]))).astype(np.float32))
            rows.append(r.cuda())

    def reverse(tiled):
        At = torch.zeros(lead + A.numel(), device=sim.device)[lead:].view(A.shape)
        At.copy_(A)
        out = [r.clone() for r in rows]
        ns = len(sim.species)
        asp = [B.pic_adjoint_species(d["cell"].data_ptr(), d["off"].data_ptr(), d["u"].data_ptr(),
                                     x.data_ptr(), u.data_ptr(), t.data_ptr() if tiled else None)
               for d, x, u, t in zip(sim.species, out[:ns], out[ns:], tst)]
        B.pic_adjoint_step(sim.ctx, sim.fields.clone().data_ptr(), asp, At.data_ptr())
        sim.check()
        assert float(At[6:9].abs().max()) == 0.0
        return [At[:6]] + out

    for got, want in zip(reverse(True), reverse(False)):
        assert _rel(got.cpu(), want.cpu()) < 2e-5
    sim.close()
