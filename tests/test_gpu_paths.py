"""Branches of the kernels that ordinary instances seldom take, against the
CPU oracle (bit-exact; needs a GB300): very long edges, mass ties, sizes at
the edges of tables and tiles."""
import numpy as np
import pytest

import oracle
from paper_2203_02228_gb300 import Batch, Colony, device_selftest, inputs

pytestmark = pytest.mark.gpu


def assert_run_equals_oracle(xy, k, ants, iters, **kw):
    g = Colony(xy, k, keep_ant_tours=1, **kw)
    kw.pop("seg_cap", None)
    o = oracle.Colony(xy, k, threads=8, **kw)
    gt, gl = g.initial()
    ot, ol = o.initial()
    assert gl == ol
    np.testing.assert_array_equal(gt, ot)
    for _ in range(iters):
        g.iterate(ants, 1)
        o.iterate(ants, 1)
        np.testing.assert_array_equal(g.ant_tours()[0], o.ant_tours()[0])
    np.testing.assert_array_equal(g.ant_tours()[1], o.ant_tours()[1])
    np.testing.assert_array_equal(g.best()[0], o.best()[0])
    assert np.array_equal(g.tau().view(np.uint32), o.tau().view(np.uint32))


@pytest.mark.parametrize("seg_cap", [-1, 0], ids=["tables", "arrays"])
@pytest.mark.parametrize("n,k", [(12, 5), (61, 16), (250, 24)])
def test_costs_beyond_the_estimate(n, k, seg_cap):
    """Coordinates over the whole [0, 2^24): most costs are 2^21 or more and
    take the exact integer steps."""
    assert_run_equals_oracle(inputs.uniform(n, seed=n, side=(1 << 24) - 1), k, 6, 6, seg_cap=seg_cap)


@pytest.mark.parametrize("seg_cap", [-1, 0], ids=["tables", "arrays"])
@pytest.mark.parametrize("rows,cols,k", [(9, 11, 8), (17, 19, 16), (13, 24, 27)])
def test_equal_gains_take_the_first_in_scan_order(rows, cols, k, seg_cap):
    assert_run_equals_oracle(inputs.lattice(rows, cols), k, 8, 8, seg_cap=seg_cap)


def test_euc2d_at_the_limit_of_the_estimate():
    """dx^2 + dy^2 on both sides of 2^42, and costs next to a half-integer
    just below 2^21, where the estimate is least certain."""
    rng = np.random.default_rng(5)
    ang = rng.uniform(0, np.pi / 2, 20000)
    r = (1 << 21) + rng.uniform(-3, 3, 20000)
    ring = np.stack([np.rint(r * np.cos(ang)), np.rint(r * np.sin(ang))], 1).astype(np.int64)
    # (k, isqrt(k) + t): dx^2 + dy^2 next to k^2 + k
    kk = rng.integers((1 << 20), (1 << 21), 20000)
    half = np.stack([kk, np.floor(np.sqrt(kk.astype(np.float64))).astype(np.int64) + rng.integers(-1, 2, 20000)], 1)
    d = np.concatenate([ring, half])
    inp = np.zeros((len(d), 4), np.int32)
    inp[:, 2:] = d
    inp[1::2] = inp[1::2][:, [2, 3, 0, 1]]
    out = np.zeros(len(d), np.int32)
    device_selftest(1, inp, out, len(d))
    want = [oracle.euc2d(np.array([[a, b], [c, e]], np.int32), 0, 1) for a, b, c, e in inp]
    np.testing.assert_array_equal(out, np.array(want, np.int32))


@pytest.mark.parametrize("seg_cap", [8, 33, 64, 256, -1])
@pytest.mark.parametrize("n", [31, 65, 1023, 2500])
def test_segment_table_capacities(n, seg_cap):
    """Tables that fill up in construction, in the search, or never: an ant
    that outgrows its table is redone on arrays with the same result."""
    xy = inputs.stippled(n, seed=n, blobs=6, ridges=1, side=50_000) if n > 1000 else inputs.uniform(n, seed=n)
    assert_run_equals_oracle(xy, 16, 12, 5, seg_cap=seg_cap, min_new_edges=24)


def _list_points(kind):
    rng = np.random.default_rng(17)
    if kind == "heap":       # one grid cell holds far more than a warp's buffer
        a = rng.integers(0, 60, size=(1500, 2))
        return np.concatenate([a, rng.integers(0, 1_000_000, size=(300, 2))])
    if kind == "same":       # most points coincide
        return np.concatenate([np.full((900, 2), 777), rng.integers(0, 5_000, size=(40, 2))])
    if kind == "outlier":    # one point far from the rest
        return np.concatenate([rng.integers(0, 2_000, size=(700, 2)), [[(1 << 24) - 1, (1 << 24) - 1]]])
    if kind == "line":
        return np.stack([np.arange(900) * 13, np.zeros(900)], 1)
    return rng.integers(0, 100_000, size=(int(kind), 2))


@pytest.mark.parametrize("kind", ["heap", "same", "outlier", "line", "4", "81", "82", "161", "162", "385"])
@pytest.mark.parametrize("k,bl", [(16, 64), (32, 128), (2, 0)])
def test_lists_of_uneven_points(kind, k, bl):
    xy = np.ascontiguousarray(_list_points(kind), dtype=np.int32)
    n = len(xy)
    g = Colony(xy, k, bl_size=bl)
    cand, backup, eta = g.lists()
    x = xy.astype(np.int64)
    d2 = (x[:, None, 0] - x[None, :, 0]) ** 2 + (x[:, None, 1] - x[None, :, 1]) ** 2
    d2[np.arange(n), np.arange(n)] = np.iinfo(np.int64).max
    order = np.argsort(d2, axis=1, kind="stable")  # ties by node id
    ke = min(k, n - 1)
    ble = min(bl, n - 1 - ke)
    np.testing.assert_array_equal(cand, order[:, :ke])
    np.testing.assert_array_equal(backup, order[:, ke:ke + ble])
    near = np.take_along_axis(d2, order[:, :ke], 1)
    d = np.floor(np.sqrt(near.astype(np.float64)) + 0.5)
    want = np.where(d > 0, np.float32(1) / np.maximum(d, 1).astype(np.float32), np.float32(1)).astype(np.float32)
    np.testing.assert_array_equal(eta, want)


@pytest.mark.parametrize("n,k", [(4095, 16), (4096, 16), (4097, 20), (8193, 16)])
def test_prefix_sums_at_tile_edges(n, k):
    """Tour lengths come from the prefix sums of the source edges, a block per
    4,096 of them."""
    assert_run_equals_oracle(inputs.uniform(n, seed=n), k, 6, 2)


@pytest.mark.parametrize("n", [8100, 8192, 8300, 40_000])
def test_lists_over_several_tiles_of_cells(n):
    """More than 4,096 grid cells: the cell starts come from several blocks."""
    xy = inputs.uniform(n, seed=n)
    g = Colony(xy, 4, bl_size=2)
    cand, backup, _ = g.lists()
    x = xy.astype(np.int64)
    for u in np.random.default_rng(n).integers(0, n, 300):
        d2 = ((x - x[u]) ** 2).sum(1)
        d2[u] = np.iinfo(np.int64).max
        near = np.argpartition(d2, 12)[:12]
        near = near[np.lexsort((near, d2[near]))][:6]
        np.testing.assert_array_equal(np.concatenate([cand[u], backup[u]]), near)


def check_short_lists(lists, n, k, bl, kind):
    """lists(xy, k, bl) of n points against full distance rows, for 200 of them."""
    rng = np.random.default_rng(n + k)
    xy = rng.integers(0, 1_000_000, size=(n, 2))
    if kind == "heap":   # many coincide, and a cell holds hundreds
        xy[: n // 8] = 500_000 + rng.integers(0, 25, size=(n // 8, 2))
    elif kind == "far":  # a few points with nothing near them
        xy[:5] = (1 << 24) - 1 - rng.integers(0, 1_000_000, size=(5, 2))
    xy = np.ascontiguousarray(xy, np.int32)
    cand, backup, eta = lists(xy, k, bl)
    x = xy.astype(np.int64)
    for u in np.concatenate([np.arange(8), rng.integers(0, n, 192)]):
        d2 = ((x - x[u]) ** 2).sum(1)
        d2[u] = np.iinfo(np.int64).max
        near = np.flatnonzero(d2 <= np.partition(d2, k + bl - 1)[k + bl - 1])  # with all ties
        near = near[np.lexsort((near, d2[near]))][: k + bl]
        np.testing.assert_array_equal(np.concatenate([cand[u], backup[u]]), near)
        d = np.floor(np.sqrt(d2[near[:k]].astype(np.float64)) + 0.5)
        np.testing.assert_array_equal(eta[u], (np.float32(1) / np.maximum(d, 1).astype(np.float32)).astype(np.float32))


@pytest.mark.parametrize("kind", ["uniform", "heap", "far"])
@pytest.mark.parametrize("n,k,bl", [(32_767, 4, 2), (32_768, 4, 2), (49_151, 7, 5), (49_152, 7, 5), (49_152, 2, 0),
                                    (60_000, 8, 5)])
def test_short_lists_of_many_nodes(n, k, bl, kind):
    """Both sides of the rule that takes a thread per node instead of a warp."""
    check_short_lists(lambda xy, k, bl: Colony(xy, k, bl_size=bl).lists(), n, k, bl, kind)


def sm_count():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("seg_cap", [-1, 28], ids=["tables", "full_tables"])
@pytest.mark.parametrize("k", [16, 24])
@pytest.mark.parametrize("more", [0, 1])
def test_both_register_variants(k, more, seg_cap):
    """At most two ant blocks per SM run one variant of the per-ant kernel,
    more run the other; with small tables some searches go on on arrays."""
    assert_run_equals_oracle(inputs.uniform(700, seed=k), k, 2 * sm_count() + more, 2, seg_cap=seg_cap)


def test_wide_batch_with_many_ants_on_tables():
    """More than two ant blocks per SM with lists wider than 16, in a batch."""
    xs = [inputs.uniform(n, seed=n) for n in (700, 260, 90, 410, 33)]
    ants = 2 * sm_count() // len(xs) + 1
    b = Batch(xs, 32, seeds=[3, 4, 5, 6, 7], plan=0)
    b.iterate(ants, 3)
    assert set(b.plan().tolist()) == {0}
    tours, lens = b.tours()
    for i, xy in enumerate(xs):
        o = oracle.Colony(xy, 32, seed=3 + i, threads=8)
        o.iterate(ants, 3)
        assert lens[i] == o.best()[1]
        np.testing.assert_array_equal(tours[i], o.best()[0])
        assert np.array_equal(b.tau(i).view(np.uint32), o.tau().view(np.uint32))


@pytest.mark.parametrize("k,new_edges", [(16, 350), (16, 900), (20, 350), (16, 600), (20, 600), (16, 1500)])
def test_batch_tables_full(k, new_edges):
    """A batch whose tables (1,024 segments and more) do not fill up, do in the
    search or in construction: the ants go on, or are built again, on arrays."""
    xs = [inputs.uniform(2500, seed=91), inputs.uniform(1800, seed=92), inputs.uniform(60, seed=93)]
    b = Batch(xs, k, seeds=[5, 6, 7], min_new_edges=new_edges, plan=0)
    b.iterate(24, 3)
    tours, lens = b.tours()
    for i, xy in enumerate(xs):
        o = oracle.Colony(xy, k, seed=5 + i, min_new_edges=new_edges, threads=8)
        o.iterate(24, 3)
        assert lens[i] == o.best()[1]
        np.testing.assert_array_equal(tours[i], o.best()[0])
        assert np.array_equal(b.tau(i).view(np.uint32), o.tau().view(np.uint32))
    if new_edges >= 900:
        assert b.stats(0).redone_ants > 0
