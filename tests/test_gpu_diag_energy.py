"""The energies of pic_energies to FP64's rounding: terms and partial sums of
three floats, against extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


def _box(dim, n, fields, u, m=1.0):
    from paper_1906_06306_gb300 import Simulation

    k = u.shape[1]
    sp = dict(q=0.01, m=m, cell=np.arange(k, dtype=np.int32) % int(np.prod(n)),
              off=np.full((dim, k), 0.5, dtype=np.float32), u=u.astype(np.float32))
    return Simulation(dim, *n, 0.45, fields, [sp])


def test_one_point_of_the_fields_has_fp64_accuracy():
    rs = np.random.default_rng(50)
    sim = _box(1, (64, 1, 1), np.zeros((9, 1, 1, 64), dtype=np.float32), np.zeros((3, 1)))
    for k in range(240):
        # components of one size, and of sizes far apart
        v = (rs.normal(size=6) * 2.0 ** (rs.integers(-38, 50) - rs.integers(0, 14 if k % 2 else 1, 6))).astype(np.float32)
        sim.fields[:6, 0, 0, 40] = sim.torch.from_numpy(v).to(sim.device)
        got = sim.energies()
        for h in range(2):
            ref = 0.5 * (v[3 * h:3 * h + 3].astype(L) ** 2).sum()
            # the three parts of the sum to a double: two roundings
            assert abs(got[h] - ref) <= 3 * 2.0 ** -53 * ref
    sim.close()


@pytest.mark.parametrize("dim,n", [(1, (70, 1, 1)), (2, (37, 50, 1)), (3, (19, 10, 9)), (2, (600, 700, 1))])
def test_fields_of_a_box_sum_to_fp64_accuracy(dim, n):
    rs = np.random.default_rng(60 + dim)
    F = np.zeros((9,) + n[::-1], dtype=np.float32)
    F[:6] = rs.normal(size=F[:6].shape) * 2.0 ** rs.integers(-45, 20, size=F[:6].shape)  # some below 2^-40
    sim = _box(dim, n, F, np.zeros((3, 1)))
    got = sim.energies()
    for h in range(2):
        ref = 0.5 * (F[3 * h:3 * h + 3].astype(L) ** 2).sum()
        # a thread's terms (at most 4 of the boxes' here), ten levels of a block's sum,
        # and the blocks' additions (at most 608), each a rounding of 2^-53
        assert abs(got[h] - ref) <= (4 + 10 + 608 ** 0.5 * 4) * 2.0 ** -53 * ref
    sim.close()


def _gamma_minus_1(u):
    u2 = (u.astype(L) ** 2).sum(0)
    return u2 / (np.sqrt(1 + u2) + 1)


def test_one_particle_has_fp64_accuracy():
    rs = np.random.default_rng(51)
    sim = _box(1, (64, 1, 1), np.zeros((9, 1, 1, 64), dtype=np.float32), np.zeros((3, 1)), m=1.7)
    mc2 = L(np.float32(1.7)) * L(np.float32(0.45)) ** 2
    for k in range(300):
        # from below 2^-40 to above 2^60, most of them near 1
        size = rs.integers(-44, 64) if k % 3 == 0 else rs.integers(-8, 8)
        u = (rs.normal(size=3) * 2.0 ** (size - rs.integers(0, 14 if k % 2 else 1, 3))).astype(np.float32)
        sim.species[0]["u"][:, :1] = sim.torch.from_numpy(u.reshape(3, 1)).to(sim.device)
        ref = mc2 * _gamma_minus_1(u.reshape(3, 1))[0]
        # FP64 form: u^2 3 roundings (half of their relative error at most 3), root, sum,
        # quotient; the three parts of the sum 2; m c^2 and its product 2
        assert abs(sim.energies()[2] - ref) <= 10 * 2.0 ** -53 * ref
    sim.close()


@pytest.mark.parametrize("n", [2, 7, 4097, 700_001])
def test_kinetic_energy_sums_to_fp64_accuracy(n):
    rs = np.random.default_rng(n)
    u = rs.normal(size=(3, n)) * 2.0 ** rs.integers(-42, 3, size=n)
    sim = _box(2, (64, 64, 1), np.zeros((9, 1, 64, 64), dtype=np.float32), u)
    ref = L(np.float32(0.45)) ** 2 * _gamma_minus_1(u.astype(np.float32)).sum()
    # as above, a thread's FP64 additions (2), a block's ten levels, the blocks' additions
    assert abs(sim.energies()[2] - ref) <= (10 + 2 + 10 + 4 * 608 ** 0.5) * 2.0 ** -53 * ref
    sim.close()
