"""Short IC samples drawn one by one (a warp each; those that outgrow its list a CTA
each; those that outgrow that by levels), against the oracle and against levels alone (host-driven): sets at the
list's limit, packed and wide rows of every alignment, always- and never-live
edges, a vertex order, the sample-id carry."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


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


def graph(n, mean):
    """Rows of 0 to 700 edges; about `mean` live edges a row, some of them certain."""
    rng = np.random.default_rng(n)
    degs = np.array([0, 1, 2, 3, 4, 5, 7, 31, 125, 128, 129, 131, 260, 700])[rng.integers(0, 14, n)]
    rp = np.concatenate([[0], np.cumsum(degs)]).astype(np.uint64)
    col = np.concatenate([np.sort(rng.choice(n, d, replace=False)) for d in degs]).astype(np.uint32)
    p = np.repeat(np.minimum(mean / np.maximum(degs, 1), 1.0), degs)
    thr = np.where(p >= 1, 0xFFFFFFFF, np.floor(p * 2.0**32)).astype(np.uint32)
    thr[rng.random(col.size) < 0.01] = 0
    return synth.Graph(n, rp, col, thr, "solo")


@pytest.mark.parametrize("n,mean,S", [(900, 0.9, 4000), (30000, 0.95, 20001), (30000, 1.03, 3000), (60000, 1.3, 300), (900, 0.5, 1)])
def test_solo_samples(fbpt, n, mean, S):
    g = graph(n, mean)
    ref = oracle.rr_sets(g, 21, 2**32 - 50, S)
    dg = fbpt.Graph.from_synth(g)
    for launch in ("persistent", "graph"):
        a = fbpt.sample(dg, 21, 2**32 - 50, S, words=8, slots=1, launch=launch)
        assert_same(a, ref, n)
    b = fbpt.sample(dg, 21, 2**32 - 50, S, words=8, slots=1, launch="host")
    assert_same(b, ref, n)
    if np.diff(ref.offsets).max() < 700:  # nothing was drawn twice
        assert a.stats.philox_calls == b.stats.philox_calls
    dg.set_order(np.random.default_rng(3).permutation(n), sorted_starts=True)
    assert_same(fbpt.sample(dg, 21, 2**32 - 50, S, words=8, slots=1), ref, n)
    dg.close()


@pytest.mark.parametrize("length", [735, 736, 737, 8191, 8192, 8193])
def test_sets_at_the_lists_limit(fbpt, length):
    """A cycle of always-live edges beside isolated vertices: sets of exactly `length`
    or one vertex, so the mean stays small."""
    n = 300 * length  # few samples start on the cycle
    rp = np.minimum(np.arange(n + 1), length).astype(np.uint64)
    col = ((np.arange(length) + 1) % length).astype(np.uint32)
    g = synth.Graph(n, rp, col, np.full(length, 0xFFFFFFFF, np.uint32), "cycle")
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 4, 0, 2000)
    assert np.diff(ref.offsets).max() == length
    for _ in range(2):  # the second run knows the mean, ~length / 300
        assert_same(fbpt.sample(dg, 4, 0, 2000, words=2, slots=1), ref, n)
    dg.close()
