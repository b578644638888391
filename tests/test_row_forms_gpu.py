"""Runs kept on the levels (by a barrier limit): a finished lane's RR set read off
its bit column, few or many lanes at a level, narrow and wide rows."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
LEVELS = dict(spin_limit=1 << 26)  # no one-by-one step


@pytest.fixture(scope="module")
def fbpt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as f
    f.build()
    return f


def assert_same(rr, ref, n):
    off, verts, starts, vcount = rr.to_host()
    assert np.array_equal(off, ref.offsets) and np.array_equal(verts, ref.verts)
    assert np.array_equal(starts, ref.starts)
    assert np.array_equal(vcount, np.bincount(ref.verts, minlength=n).astype(np.uint32))


def torus(k, p):
    """A k x k torus, four in-neighbours a vertex: sets of many levels."""
    v = np.arange(k * k).reshape(k, k)
    nb = np.stack([np.roll(v, 1, 0), np.roll(v, -1, 0), np.roll(v, 1, 1), np.roll(v, -1, 1)], -1).reshape(k * k, 4)
    nb.sort(axis=1)
    return synth.Graph(k * k, np.arange(0, 4 * k * k + 1, 4, dtype=np.uint64), nb.reshape(-1).astype(np.uint32),
                       np.full(4 * k * k, int(p * 2.0**32), np.uint32), "torus")


@pytest.mark.parametrize("words,slots,S", [(1, 1, 200), (1, 3, 700), (2, 4, 64), (1, 33, 3000), (8, 8, 4096), (4, 5, 1279)])
@pytest.mark.parametrize("launch", ["graph", "persistent", "host"])
def test_columns_of_few_and_many_lanes(fbpt, words, slots, S, launch):
    g = torus(31, 0.52)
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 3, 0, S)
    kw = dict(words=words, slots=slots, launch=launch, **LEVELS)
    for refill in ("lane", "batch"):
        assert_same(fbpt.sample(dg, 3, 0, S, refill=refill, **kw), ref, g.n)
    dg.set_order(np.random.default_rng(2).permutation(g.n), sorted_starts=True)
    assert_same(fbpt.sample(dg, 3, 0, S, **kw), ref, g.n)
    dg.close()


def test_deep_runs_with_wide_rows(fbpt):
    """A level that ends a few of 4,096 lanes reads their columns, not all of every row."""
    g = torus(1024, 0.49)
    dg = fbpt.Graph.from_synth(g)
    kw = dict(words=8, slots=8, launch="graph", **LEVELS)
    fbpt.sample(dg, 1, 0, 4096, **kw)
    rr = fbpt.sample(dg, 1, 0, 4096, **kw)
    assert rr.stats.ms_sweep < rr.stats.ms_expand
    assert_same(rr, oracle.rr_sets(g, 1, 0, 4096), g.n)
    dg.close()


@pytest.mark.parametrize("c,by_levels", [(0.9, False), (1.7, False), (2.5, True)])
def test_few_long_samples_of_a_small_graph(fbpt, c, by_levels):
    """Few samples go by levels at once where a run has shown most sets to outgrow a warp's list."""
    rp, col = synth.er_graph(1024, 1024 * 16, 3)
    g = synth.Graph(1024, rp, col, synth.thr_uniform(col.size, c / 16), "er")
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 3, 0, 500)
    kw = dict(words=8, slots=8, launch="graph")
    assert_same(fbpt.sample(dg, 3, 0, 500, **kw), ref, g.n)
    a, b = fbpt.sample(dg, 3, 0, 500, **kw), fbpt.sample(dg, 3, 0, 500, **kw, **LEVELS)
    assert_same(a, ref, g.n)
    assert ((a.stats.levels, a.stats.units_expanded) == (b.stats.levels, b.stats.units_expanded)) == by_levels
    dg.close()


@pytest.mark.parametrize("words,slots", [(1, 1), (1, 3), (8, 8)])
@pytest.mark.parametrize("launch", ["graph", "persistent"])
@pytest.mark.parametrize("kind", ["lists", "harvest"])
def test_short_sets_by_levels(fbpt, kind, words, slots, launch):
    """Sets that plain push calls draw one by one, through both ways that the levels write them."""
    n = 20001 if kind == "lists" else 2048
    rp, col = synth.er_graph(n, 6 * n, 7)
    g = synth.Graph(n, rp, col, synth.thr_uniform(col.size, 0.1 if kind == "lists" else 0.15), kind)
    ref = oracle.rr_sets(g, 11, 2**32 - 700, 1500)
    dg = fbpt.Graph.from_synth(g)
    for _ in range(2):
        rr = fbpt.sample(dg, 11, 2**32 - 700, 1500, words=words, slots=slots, launch=launch, **LEVELS)
        assert_same(rr, ref, g.n)
        assert rr.stats.ms_commit > 0  # levels
    one = fbpt.sample(dg, 11, 2**32 - 700, 1500, words=words, slots=slots, launch=launch)
    assert_same(one, ref, g.n)
    assert one.stats.ms_commit == 0  # all sets fit a warp's list
    dg.close()


@pytest.mark.parametrize("k,c", [(1500, 8), (3000, 50)])
def test_teams_share_rows(fbpt, k, c):
    """Sets beyond a warp's list whose rows are long enough for all warps of a CTA (256 groups and
    more), up to more of them in a round than its list of rows holds (1,024)."""
    rng = np.random.default_rng(k)
    n = 40 * k  # the other vertices are isolated: few samples are long
    degs = np.where(rng.random(k) < 0.1, 5, rng.integers(1025, 1041, k))
    rp = np.zeros(n + 1, np.uint64)
    rp[1:k + 1] = np.cumsum(degs)
    rp[k + 1:] = rp[k]
    col = np.concatenate([np.sort(rng.choice(k, d, replace=False)) for d in degs]).astype(np.uint32)
    g = synth.Graph(n, rp, col, synth.thr_uniform(col.size, c / 1030), "core")
    ref = oracle.rr_sets(g, 9, 0, 400)
    long = int((np.diff(ref.offsets) > 736).sum())
    assert 0 < long <= 400 // 16
    for launch in ("graph", "persistent"):
        for order in (None, np.random.default_rng(1).permutation(n)):
            dg = fbpt.Graph.from_synth(g)  # a first call: later ones know the mean and go by levels
            if order is not None:
                dg.set_order(order, sorted_starts=True)
            rr = fbpt.sample(dg, 9, 0, 400, words=1, slots=2, launch=launch)
            assert_same(rr, ref, n)
            assert rr.stats.ms_commit == 0  # none was left to the levels
            dg.close()
