"""The linear-threshold edge search at row lengths around its 32-entry steps and
with weights that an equal-weight guess misses (one heavy edge at either end,
runs of zero weights, rows that keep nothing), bit-exact against the oracle."""
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


def graph(kind, seed):
    rng = np.random.default_rng(seed)
    n = 3000
    degs = np.array([1, 2, 31, 32, 33, 34, 63, 65, 100, 1000, 1089, 2999])[rng.integers(0, 12, n)]
    rp = np.concatenate([[0], np.cumsum(degs)]).astype(np.uint64)
    col = np.concatenate([np.sort(rng.choice(n, d, replace=False)) for d in degs]).astype(np.uint32)
    thr = []
    for d in degs:
        i = np.arange(d)
        w = {"first": np.exp(-i / 3.0), "last": np.exp((i - d + 1) / 3.0), "zeros": (i % 40 == 39) * 1.0,
             "random": rng.random(d) ** 8, "equal": np.ones(d)}[kind]
        s = w.sum()
        thr.append(np.floor(w / s * 0.95 * 2.0**32) if s else np.zeros(d))
    return synth.Graph(n, rp, col, np.concatenate(thr).astype(np.uint32), "lt-" + kind)


@pytest.mark.parametrize("launch", ["graph", "persistent"])
@pytest.mark.parametrize("kind", ["first", "last", "zeros", "random", "equal"])
def test_lt_search_bit_exact(fbpt, kind, launch):
    g = graph(kind, 17)
    dg = fbpt.Graph.from_synth(g)
    rr = fbpt.sample(dg, 99, 2**32 - 2000, 6000, words=8, slots=2, launch=launch, model="lt")
    ref = oracle.rr_sets(g, 99, 2**32 - 2000, 6000, model="lt")
    off, verts, starts, vcount = rr.to_host()
    assert np.array_equal(off, ref.offsets) and np.array_equal(verts, ref.verts)
    assert np.array_equal(starts, ref.starts)
    assert np.array_equal(vcount, np.bincount(ref.verts, minlength=g.n).astype(np.uint32))
    # one draw and, at most, one edge per visited vertex
    st = rr.stats
    assert st.edge_accesses <= st.philox_calls
    dg.close()
