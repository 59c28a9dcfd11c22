"""The kernels' own code on the CPU (tests/emu), with the order of a block's
threads shuffled and shared memory watched: results against plain numpy or the
oracle, and no access that CUDA would not order."""
import os
import subprocess
import sys

import pytest

EMU = os.path.join(os.path.dirname(os.path.abspath(__file__)), "emu")


@pytest.fixture(scope="module")
def emulated():
    """Runs Python code against the emulated library in a process of its own."""
    out = subprocess.run([sys.executable, "-c", "import build; print(build.build())"], cwd=EMU, capture_output=True,
                         text=True)
    assert out.returncode == 0, out.stderr
    lib = out.stdout.strip()

    def run(code, seed=1):
        r = subprocess.run([sys.executable, os.path.join(EMU, "run.py")], input=code, capture_output=True, text=True,
                           env=dict(os.environ, FACO_EMU=lib, EMU_SEED=str(seed)), timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr

    return run


LISTS = """
import ctypes
import numpy as np
from paper_2203_02228_gb300 import load

rng = np.random.default_rng(3)
kind = "{kind}"
if kind == "heap":       # a cell with more points than a warp's buffer
    xy = np.concatenate([rng.integers(0, 60, size=(500, 2)), rng.integers(0, 1_000_000, size=(60, 2))])
elif kind == "same":     # no distance cuts the buffer down
    xy = np.concatenate([np.full((420, 2), 777), rng.integers(0, 5_000, size=(30, 2))])
elif kind == "outlier":  # a block of cells with enough points, none of them close enough
    xy = np.concatenate([rng.integers(0, 2_000, size=(250, 2)), [[(1 << 24) - 1, (1 << 24) - 1]]])
else:
    xy = rng.integers(0, 100_000, size=(300, 2))
xy = np.ascontiguousarray(xy, np.int32)
n, k, bl = len(xy), 16, 64
cand, backup = np.zeros((n, k), np.int32), np.zeros((n, bl), np.int32)
eta = np.zeros((n, k), np.float32)
p = lambda a: ctypes.c_void_p(a.ctypes.data)
assert load().faco_lists_noalloc(p(xy), n, k, bl, p(cand), p(backup), p(eta), None) == 0
x = xy.astype(np.int64)
d2 = ((x[:, None] - x[None]) ** 2).sum(2)
d2[np.arange(n), np.arange(n)] = np.iinfo(np.int64).max
order = np.argsort(d2, axis=1, kind="stable")  # ties by node id
np.testing.assert_array_equal(np.concatenate([cand, backup], 1), order[:, :k + bl])
"""


@pytest.mark.parametrize("kind", ["heap", "same", "outlier", "even"])
def test_lists(emulated, kind):
    emulated(LISTS.format(kind=kind))


SETUP = """
import numpy as np
import oracle
from paper_2203_02228_gb300 import Colony, inputs

xy = inputs.uniform({n}, seed={n})
g, o = Colony(xy, {k}, init_3opt={three_opt}), oracle.Colony(xy, {k}, threads=2, init_3opt={three_opt})
np.testing.assert_array_equal(g.initial()[0], o.initial()[0])
assert g.initial()[1] == o.initial()[1]
"""


@pytest.mark.parametrize("n,k,three_opt", [(7, 3, 0), (90, 16, 0), (260, 16, 0), (120, 24, 1)])
def test_initial_search(emulated, n, k, three_opt):
    """Fewer and more nodes than the window, than the nodes read ahead, and
    than the ring they are kept in."""
    emulated(SETUP.format(n=n, k=k, three_opt=three_opt))


FULL_TABLES = """
import numpy as np
import oracle
from paper_2203_02228_gb300 import Colony, inputs

xy = inputs.uniform({n}, seed={n})
kw = dict({kw})
kept, plain = Colony(xy, {k}, seg_cap={cap}, keep_ant_tours=1, **kw), Colony(xy, {k}, seg_cap={cap}, **kw)
o = oracle.Colony(xy, {k}, threads=4, **kw)
last = np.zeros((6, 24), np.int64)
for _ in range(3):
    for c in (kept, plain, o):
        c.iterate(6, 1)
    np.testing.assert_array_equal(kept.ant_tours()[0], o.ant_tours()[0])
    np.testing.assert_array_equal(plain.source()[0], o.source()[0])
    st = kept.ant_stats()
    full = st[:, 10] > last[:, 10]
    assert (st[full, 15] != last[full, 15]).all()  # a block's evaluation time: not left to the one-warp kernel
    last = st
assert last[:, 10].any()
"""


@pytest.mark.parametrize("n,k,cap,kw", [(250, 16, 24, ""), (400, 24, 40, "min_new_edges=12"),
                                        (300, 16, 32, "verify_pass=0")])
def test_search_goes_on_when_its_table_is_full(emulated, n, k, cap, kw):
    """Tables that hold every tour as constructed and fill up in the search."""
    emulated(FULL_TABLES.format(n=n, k=k, cap=cap, kw=kw), seed=n)


SHORT_LISTS = """
import numpy as np
from tests.test_gpu_paths import check_short_lists
import ctypes
from paper_2203_02228_gb300 import load

def lists(xy, k, bl):
    n = len(xy)
    cand, backup = np.zeros((n, k), np.int32), np.zeros((n, max(bl, 1)), np.int32)
    eta = np.zeros((n, k), np.float32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    assert load().faco_lists_noalloc(p(xy), n, k, bl, p(cand), p(backup), p(eta), None) == 0
    return cand, backup[:, :bl], eta

check_short_lists(lists, {n}, {k}, {bl}, "{kind}")
"""


@pytest.mark.parametrize("n,k,bl,kind", [(32_768, 2, 0, "uniform"), (32_769, 4, 2, "heap"), (49_152, 5, 7, "uniform"),
                                         (49_152, 7, 0, "far")])
def test_short_lists_by_threads(emulated, n, k, bl, kind):
    emulated(SHORT_LISTS.format(n=n, k=k, bl=bl, kind=kind))


def test_tuner_lists_an_ant_once(emulated, monkeypatch):
    """A batch that times its per-ant kernels first: every table fills up in
    construction, in each of the timed passes."""
    monkeypatch.setenv("EMU_SM_SHARED", "17664")  # tables of 64 segments
    emulated("""
from paper_2203_02228_gb300 import Batch, inputs
b = Batch([inputs.uniform(160, seed=7), inputs.uniform(150, seed=8)], 8, seeds=[3, 4], min_new_edges=160)
b.iterate(3, 1)
b.sync()
b.set_plan(0)
b.iterate(3, 2)
assert b.stats(0).seg_cap == 64 and b.stats(0).redone_ants > 0
""")


@pytest.mark.parametrize("k,new_edges", [(16, 34), (24, 30)])
def test_batch_tables_full(emulated, monkeypatch, k, new_edges):
    """Tables of 64 segments that fill up in construction, in the search, or
    not at all."""
    monkeypatch.setenv("EMU_SM_SHARED", "17664")
    emulated("""
import numpy as np
import oracle
from paper_2203_02228_gb300 import Batch, inputs
xs = [inputs.uniform(400, seed=7), inputs.uniform(150, seed=8)]
b = Batch(xs, {k}, seeds=[3, 4], min_new_edges={e}, plan=0)
b.iterate(5, 2)
tours, lens = b.tours()
for i, x in enumerate(xs):
    o = oracle.Colony(x, {k}, seed=3 + i, min_new_edges={e}, threads=4)
    o.iterate(5, 2)
    np.testing.assert_array_equal(tours[i], o.best()[0])
    assert np.array_equal(b.tau(i).view(np.uint32), o.tau().view(np.uint32))
assert b.stats(0).seg_cap == 64 and b.stats(0).redone_ants > 0
""".format(k=k, e=new_edges), seed=k)
