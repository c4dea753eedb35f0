"""The charge behind pic_energies' Gauss residual where many particles share one
cell: the tile kernel's batches, and the sums that their words must hold."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

Q = np.float32(0.01)


def _box(dim, cell, off, tile=8):
    """One species at rest in a box of 64 tiles without fields: the residual is the charge."""
    from paper_1906_06306_gb300 import Simulation

    n = (512, 1, 1) if dim == 1 else (64, 64, 1)
    sp = dict(q=Q, m=1.0, cell=cell, off=off, u=np.zeros((3, cell.size), dtype=np.float32))
    sim = Simulation(dim, *n, 0.45, np.zeros((9,) + n[::-1], dtype=np.float32), [sp],
                     tuning=dict(tile=[tile] * dim + [1] * (3 - dim)))
    sim.sort()
    return sim


def _node_charges(off):
    """Charge of the corner nodes of the one cell that holds every particle, extended precision."""
    L = np.longdouble
    w = off.astype(L)
    out = []
    for corner in range(1 << w.shape[0]):
        t = L(1.0)
        for d in range(w.shape[0]):
            t = t * (w[d] if corner >> d & 1 else 1 - w[d])
        out.append(L(Q) * (t * np.ones(off.shape[1], dtype=L)).sum())
    return np.array(out)


@pytest.mark.parametrize("offset", [0.0, 2.0 ** -50, 0.25, 1.0 - 2.0 ** -24])
@pytest.mark.parametrize("n", [32_768, 70_000])
@pytest.mark.parametrize("dim", [1, 2])
def test_full_batches_in_one_cell(dim, n, offset):
    # a share of 32,768 particles or more, far above the mean of the tiles, from one block
    off = np.full((dim, n), offset, dtype=np.float32)
    cell = np.full(n, 300 if dim == 1 else 30 + 64 * 21, dtype=np.int32)
    sim = _box(dim, cell, off)
    ref = _node_charges(off)
    # E at the cell's low corner carries the sign: div E = +q n there, residual = q n - rho
    sim.fields[0].view(-1)[int(cell[0])] = float(ref[0])
    lo = float(np.float32(float(ref[0])))
    nodes = {0: lo - float(ref[0])}
    for k in range(1, 1 << dim):
        nodes[k] = -float(ref[k])
    nodes[1] -= lo  # the x neighbour's divergence takes E off again
    got = sim.energies()
    want = max(abs(v) for v in nodes.values())
    # each particle's weights within 2^-46 of their exact values, FP64 sums
    assert abs(got[3] - want) <= 2.0 ** -46 * float(Q) * n
    sim.close()


def _tiny(off):
    """Particles whose offsets the fixed-point sums do not hold whole: FP64 weights of four roundings."""
    return int(((off > 0) & (off < 2.0 ** -8)).any(0).sum())


def _check_whole(sim, off, cell):
    ref = _node_charges(off)
    got = sim.energies()
    # no fields: one rounding of a batch's sum, one of its product with q and one of its
    # addition to the node (4 batches at most here); four roundings of each queued
    # particle's weight and one of its addition
    batches = 4
    tol = 2.0 ** -53 * (3 * batches + 5 * _tiny(off)) * float(ref.max())
    assert abs(got[3] - float(ref.max())) <= tol


OFFSETS = [0.0, 2.0 ** -149, 2.0 ** -60, 2.0 ** -30, 2.0 ** -8 - 2.0 ** -32, 2.0 ** -8, 2.0 ** -8 + 2.0 ** -31,
           0.5, 1.0 - 2.0 ** -24]


@pytest.mark.parametrize("dim", [1, 2])
def test_one_particle_has_all_its_bits(dim):
    rs = np.random.default_rng(40 + dim)
    k = np.arange(len(OFFSETS) ** dim)
    edge = np.array([[OFFSETS[i // len(OFFSETS) ** d % len(OFFSETS)] for i in k] for d in range(dim)])
    draws = np.minimum(rs.random((dim, 60)).astype(np.float32) * 2.0 ** -rs.integers(0, 12, (dim, 60)),
                       1 - 2.0 ** -24)
    cell = np.array([300 if dim == 1 else 30 + 64 * 21], dtype=np.int32)
    sim = _box(dim, cell, np.zeros((dim, 1), dtype=np.float32))
    for o in np.concatenate([edge, draws], axis=1).astype(np.float32).T:
        sim.species[0]["off"][:, :1] = sim.torch.from_numpy(o.reshape(dim, 1)).to(sim.device)
        _check_whole(sim, o.reshape(dim, 1), cell)
    sim.close()


@pytest.mark.parametrize("n", [1, 255, 1025, 16_384, 40_000])
@pytest.mark.parametrize("dim", [1, 2])
def test_many_particles_of_a_cell_have_all_their_bits(dim, n):
    rs = np.random.default_rng(dim * n)
    off = np.minimum(rs.random((dim, n)).astype(np.float32), np.float32(1 - 2.0 ** -24))
    off[:, n // 2:] *= np.float32(2.0 ** -7)  # most of the second half goes through the queue
    cell = np.full(n, 300 if dim == 1 else 30 + 64 * 21, dtype=np.int32)
    sim = _box(dim, cell, off)
    _check_whole(sim, off, cell)
    sim.close()
