"""The tile sort at the sizes where its scatter changes form (2^17 and 2^19
particles of a species), with ragged last chunks, many bins to a chunk and one
bin for all: the recorded permutation rebuilds the sorted records bit for bit
and every cell's particles are in one bin."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(dim, shape, n, cells, seed, tile=None):
    import torch

    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    rs = np.random.default_rng(seed)
    sp = [dict(q=1.0, m=1.0, cell=cells(rs, k).astype(np.int32), off=rs.random((dim, k), dtype=np.float32),
               u=rs.normal(size=(3, k)).astype(np.float32)) for k in (n, 3)]
    sim = Simulation(dim, *shape, 0.45, np.zeros((9,) + shape[::-1], np.float32), sp,
                     tuning=dict(tile=tile) if tile else None)
    d = sim.species[0]
    for k in ("cell", "off", "u"):  # the caller's order, not the set-up sort's
        d[k][..., :n] = torch.from_numpy(sp[0][k]).to(sim.device)
    nb = B.pic_sort_bins(sim.ctx)
    perm = [torch.full((s["n"],), -1, dtype=torch.int32, device=sim.device) for s in sim.species]
    start = [torch.full((nb + 1,), -1, dtype=torch.int32, device=sim.device) for _ in sim.species]
    B.pic_sort_record(sim.ctx, [p.data_ptr() for p in perm], [t.data_ptr() for t in start])
    p, t = perm[0].cpu().numpy(), start[0].cpu().numpy()
    assert np.array_equal(np.sort(p), np.arange(n))
    got = sim.download()[1][0]
    for k in ("cell", "off", "u"):
        assert np.array_equal(got[k].view(np.int32), sp[0][k][..., p].view(np.int32))
    assert t[0] == 0 and t[-1] == n and (np.diff(t) >= 0).all()
    bin_of = np.repeat(np.arange(nb), np.diff(t))
    lo, hi = np.full(shape[0] * shape[1] * shape[2], nb), np.full(shape[0] * shape[1] * shape[2], -1)
    np.minimum.at(lo, got["cell"], bin_of)
    np.maximum.at(hi, got["cell"], bin_of)
    used = hi >= 0
    assert np.array_equal(lo[used], hi[used])
    sim.check()
    sim.close()


@pytest.mark.parametrize("n", [255, (1 << 17) - 1, 1 << 17, (1 << 17) + 1023, (1 << 19) - 1, (1 << 19) + 2047])
@pytest.mark.parametrize("dim,shape", [(1, (1000, 1, 1)), (2, (203, 97, 1)), (3, (41, 33, 30))])
def test_sizes_where_the_scatter_changes(dim, shape, n):
    cells = shape[0] * shape[1] * shape[2]
    # nearly sorted: the order that a run finds some steps after a sort
    _run(dim, shape, n, lambda rs, k: np.clip(np.sort(rs.integers(0, cells, k)) + rs.integers(-9, 10, k), 0,
                                               cells - 1), seed=n % 1000 + dim)


@pytest.mark.parametrize("order", ["random over many bins", "one cell"])
def test_chunks_with_more_bins_than_the_table_and_with_one(order):
    shape = (256, 256, 1)
    many = lambda rs, k: rs.integers(0, 65536, k)  # noqa: E731  2x2 tiles: 16,384 bins
    one = lambda rs, k: np.full(k, 12345)  # noqa: E731
    _run(2, shape, 600_000, many if order.startswith("random") else one, seed=3,
         tile=[2, 2] if order.startswith("random") else None)


@pytest.mark.parametrize("tile", [[16, 16], [2, 2]])  # 2^13 bins: one launch; 2^16: a copy and a check each
def test_adopted_bucket_starts_are_checked(tile):
    import torch

    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    rs = np.random.default_rng(5)
    n = 5000
    sp = [dict(q=q, m=1e-3, cell=rs.integers(0, 512 * 512, k).astype(np.int32),
               off=rs.random((2, k), dtype=np.float32), u=np.zeros((3, k), np.float32))
          for q, k in ((1e-3, n), (-1e-3, 0), (-1e-3, n - 1))]
    sim = Simulation(2, 512, 512, 1, 0.45, np.zeros((9, 1, 512, 512), np.float32), sp,
                     tuning=dict(tile=tile, sort_every=1000))
    nb = B.pic_sort_bins(sim.ctx)
    perm = [torch.empty(max(s["n"], 1), dtype=torch.int32, device=sim.device) for s in sim.species]
    start = [torch.empty(nb + 1, dtype=torch.int32, device=sim.device) for _ in sim.species]
    B.pic_sort_record(sim.ctx, [p.data_ptr() for p in perm], [t.data_ptr() for t in start])
    B.pic_stats(sim.ctx)
    B.pic_sort_assume(sim.ctx, [t.data_ptr() for t in start])
    sim.step(2)
    sim.check()
    assert B.pic_stats(sim.ctx) == 0  # everyone in the window of its tile
    bad = start[2].clone()
    bad[nb // 2] = n + 7
    B.pic_sort_assume(sim.ctx, [start[0].data_ptr(), start[1].data_ptr(), bad.data_ptr()])
    with pytest.raises(B.PicError) as e:
        sim.check()
    assert e.value.status == B.PIC_ERR_STATE
    sim.close()


@pytest.mark.parametrize("counts", [(70_000, 0, 5), (3, 140_000, 1025), (600_000, 2049, 131_072, 0)])
@pytest.mark.parametrize("dim,shape,tile", [(1, (4000, 1, 1), None), (2, (203, 97, 1), None),
                                            (2, (256, 256, 1), [2, 2]), (3, (41, 33, 30), None)])
def test_species_of_different_size_in_one_sort(dim, shape, tile, counts):
    """Every species of a sort, whose launches they share (the largest one's
    size sets them): records bit for bit and the starts the bins' counts."""
    import torch

    from paper_1906_06306_gb300 import Simulation
    from paper_1906_06306_gb300 import binding as B

    rs = np.random.default_rng(sum(counts) + dim)
    cells = shape[0] * shape[1] * shape[2]
    sp = [dict(q=1.0, m=1.0, cell=rs.integers(0, cells, n).astype(np.int32),
               off=rs.random((dim, n), dtype=np.float32), u=rs.normal(size=(3, n)).astype(np.float32)) for n in counts]
    sim = Simulation(dim, *shape, 0.45, np.zeros((9,) + shape[::-1], np.float32), sp,
                     tuning=dict(tile=tile) if tile else None)
    for d, s in zip(sim.species, sp):
        for k in ("cell", "off", "u"):
            d[k][..., : d["n"]] = torch.from_numpy(s[k]).to(sim.device)
    nb = B.pic_sort_bins(sim.ctx)
    perm = [torch.full((max(n, 1),), -1, dtype=torch.int32, device=sim.device) for n in counts]
    start = [torch.full((nb + 1,), -1, dtype=torch.int32, device=sim.device) for _ in counts]
    B.pic_sort_record(sim.ctx, [p.data_ptr() for p in perm], [t.data_ptr() for t in start])
    sim.check()
    for got, s, p, t, n in zip(sim.download()[1], sp, perm, start, counts):
        if n == 0:
            continue
        p, t = p.cpu().numpy(), t.cpu().numpy()
        assert np.array_equal(np.sort(p), np.arange(n))
        for k in ("cell", "off", "u"):
            assert np.array_equal(got[k].view(np.int32), s[k][..., p].view(np.int32))
        assert t[0] == 0 and t[-1] == n and (np.diff(t) >= 0).all()
        bin_of = np.repeat(np.arange(nb), np.diff(t))
        order = np.argsort(got["cell"], kind="stable")
        c, b = got["cell"][order], bin_of[order]
        assert (b[1:] == b[:-1])[c[1:] == c[:-1]].all()
    sim.close()
