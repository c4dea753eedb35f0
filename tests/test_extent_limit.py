"""Lattices so long that coordinates past their end would not fit in an int are
refused on the host, before any CUDA work (so this runs without a GPU)."""
import pytest


@pytest.mark.parametrize("dim,nx", [(1, 2 ** 31 - 1), (1, 2 ** 31 - 1024), (2, 2 ** 31 - 4), (3, 2 ** 31 - 900)])
def test_extents_next_to_2_31_are_refused(dim, nx):
    from paper_1906_06306_gb300 import build

    build.build()
    from paper_1906_06306_gb300 import binding as B

    grid = B.pic_grid(dim, nx, 1, 1)
    sp = [B.pic_species(-1.0, 1.0, 4, 0x1000, 0x1000, 0x1000, 0)]
    with pytest.raises(B.PicError, match="PIC_ERR_ARG.*int32"):
        B.pic_init(grid, sp, 0.45, 1.0, 0x1000, 0)
