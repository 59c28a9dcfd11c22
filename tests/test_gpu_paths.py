"""Branches of the kernels that ordinary instances seldom take, against the
CPU oracle (bit-exact; needs a GB300): very long edges, mass ties, sizes at
the edges of tables and tiles."""
import numpy as np
import pytest

import oracle
from paper_2203_02228_gb300 import Colony, device_selftest, inputs

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
