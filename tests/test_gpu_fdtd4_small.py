"""FDTD4's field updates on boxes of one to five points an axis, where the wide
stencil wraps onto itself, against the oracle."""
import numpy as np
import pytest

import oracle

from gpu_helpers import compare_fields, random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,shape", [(1, (1, 1, 1)), (1, (2, 1, 1)), (1, (3, 1, 1)), (2, (2, 3, 1)),
                                       (2, (1, 4, 1)), (2, (5, 1, 1)), (3, (2, 1, 3)), (3, (4, 2, 2))])
def test_updates_match_oracle(dim, shape):
    from paper_1906_06306_gb300 import PIC_FIELD_B_HALF, PIC_FIELD_E, Simulation

    nx, ny, nz = shape
    rs = np.random.default_rng(nx + 10 * ny + 100 * nz)
    F32 = random_fields((nz, ny, nx), rs)
    F32[6:9] = (0.01 * rs.normal(size=(3, nz, ny, nx))).astype(np.float32)
    empty = [dict(q=-1.0, m=1.0, cell=np.zeros(0, np.int32), off=np.zeros((dim, 0), np.float32),
                  u=np.zeros((3, 0), np.float32))]
    sim = Simulation(dim, nx, ny, nz, 0.45, F32, empty)
    sim.set_field_solver(4)
    g = oracle.Grid(dim, nx, ny, nz, 0.45)
    F = F32.astype(np.float64)
    oracle.set_field_order(4)
    try:
        # a dozen float32 operations per value, as in the test at ordinary sizes
        sim.field_update(PIC_FIELD_B_HALF)
        oracle.push_half_b(g, F)
        compare_fields(sim.download()[0], F, tol=1e-6)
        sim.field_update(PIC_FIELD_E)
        oracle.push_e(g, F)
        oracle.add_cur(g, F)
        compare_fields(sim.download()[0], F, tol=1e-6)
    finally:
        oracle.set_field_order(2)
    sim.close()
