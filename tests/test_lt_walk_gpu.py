"""LT samples as whole walks and by levels (a run with a trace) against the oracle:
row lengths around the 32-entry window, a vertex order, several tasks in one call,
walks that end by meeting themselves, and one longer than the path buffer."""
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


def graph(n, full):
    """Rows of 0 to 200 edges around the window's size; total weight 1 (full) or 0.6."""
    rng = np.random.default_rng(n)
    degs = np.array([0, 1, 2, 31, 32, 33, 34, 64, 65, 200])[rng.integers(0 if not full else 1, 10, n)]
    rp = np.concatenate([[0], np.cumsum(degs)]).astype(np.uint64)
    col = np.concatenate([np.sort(rng.choice(n, d, replace=False)) for d in degs]).astype(np.uint32)
    thr = [np.floor(w / w.sum() * (1.0 if full else 0.6) * (2.0**32 - d - 1)) if d else np.zeros(0)
           for d in degs for w in [rng.random(d) ** 4 + 1e-6]]
    return synth.Graph(n, rp, col, np.concatenate(thr).astype(np.uint32), "lt")


@pytest.mark.parametrize("n,S", [(300, 1), (300, 5000), (40000, 3001)])
@pytest.mark.parametrize("full", [False, True])
def test_walks_and_levels(fbpt, n, S, full):
    g = graph(n, full)
    ref = oracle.rr_sets(g, 5, 2**32 - 100, S, model="lt")
    dg = fbpt.Graph.from_synth(g)
    a = fbpt.sample(dg, 5, 2**32 - 100, S, words=4, slots=2, model="lt")
    b = fbpt.sample(dg, 5, 2**32 - 100, S, words=4, slots=2, model="lt", launch="graph", trace_cap=1 << 16)
    assert_same(a, ref, n)
    assert_same(b, ref, n)
    assert a.stats.philox_calls == b.stats.philox_calls and a.stats.edge_accesses == b.stats.edge_accesses
    dg.set_order(np.random.default_rng(2).permutation(n), sorted_starts=True)
    assert_same(fbpt.sample(dg, 5, 2**32 - 100, S, model="lt"), ref, n)
    outs, _ = fbpt.sample_batched([dg, dg], [5, 6], [2**32 - 100, 0], [S, 77], words=2, slots=1, model="lt")
    assert_same(outs[0], ref, n)
    assert_same(outs[1], oracle.rr_sets(g, 6, 0, 77, model="lt"), n)
    dg.close()


@pytest.mark.parametrize("length", [1023, 1024, 1025])
def test_walk_at_the_path_buffers_end(fbpt, length):
    """A cycle of `length` vertices: every walk goes all the way round."""
    rp = np.arange(length + 1, dtype=np.uint64)
    col = ((np.arange(length) + 1) % length).astype(np.uint32)
    g = synth.Graph(length, rp, col, np.full(length, 0xFFFFFFFF, np.uint32), "cycle")
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 9, 0, 40, model="lt")
    for _ in range(2):
        assert_same(fbpt.sample(dg, 9, 0, 40, words=1, slots=1, model="lt"), ref, length)
    dg.close()
