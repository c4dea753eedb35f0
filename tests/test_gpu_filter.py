"""The fused Binomial2 passes at the edges of their columns (120 x points a
warp, 28 rows a 3D column) and of their splits into launches, against the
oracle's filter."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# (dim, (nx, ny, nz), passes): one quad, below and past a warp's 120 and 128
# points, rows of a multiple of 4 and not, columns of 28 rows and one more,
# fewer planes or rows than the halo; passes over every launch split
CASES = ([(1, (n, 1, 1), p) for n, p in [(4, 9), (119, 4), (120, 3), (124, 8), (481, 5), (1000, 1)]] +
         [(2, (n, m, 1), p) for n, m, p in [(120, 9, 4), (121, 40, 3), (244, 2, 8), (8, 300, 7), (3, 5, 9),
                                            (128, 17, 1), (360, 64, 2)]] +
         [(3, s, p) for s, p in [((120, 28, 9), 4), ((124, 29, 3), 3), ((121, 57, 2), 5), ((8, 1, 40), 4),
                                 ((256, 33, 5), 9), ((5, 3, 1), 6), ((240, 28, 31), 2)]])


@pytest.mark.parametrize("dim,shape,passes", CASES)
def test_fused_passes_match_oracle(dim, shape, passes):
    import torch

    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    nx, ny, nz = shape
    rs = np.random.default_rng(nx + 1000 * ny + nz)
    F32 = np.zeros((9, nz, ny, nx), np.float32)
    F32[6:] = rs.normal(size=(3, nz, ny, nx))
    empty = [dict(q=-1.0, m=1.0, cell=np.zeros(0, np.int32), off=np.zeros((dim, 0), np.float32),
                  u=np.zeros((3, 0), np.float32))]
    sim = Simulation(dim, nx, ny, nz, 0.45, F32, empty)
    sim.filter_current(passes)
    F = F32.astype(np.float64)
    oracle.filter_binomial(oracle.Grid(dim, nx, ny, nz, 0.45), F, passes)
    got = sim.download()[0][6:]
    # two roundings of at most 2^-24 of the largest value per sub-pass; the
    # filter's weights are positive and sum to 1, so errors do not grow
    assert np.abs(got - F[6:]).max() <= 2 * dim * passes * 2.0 ** -24 * np.abs(F32[6:]).max()
    J = torch.from_numpy(F32[6:].copy()).cuda()
    stream = torch.cuda.current_stream()
    B.pic_filter_current_static(B.pic_grid(dim, nx, ny, nz), J.data_ptr(), passes, stream.cuda_stream)
    assert np.array_equal(J.cpu().numpy(), got)
    sim.close()
