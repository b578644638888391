"""The two ways a finished lane's RR set is written (entry lists, and the harvest of
its bit column) and the ordering of rows of every length class, against the oracle."""
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
    if ref.starts is not None:
        assert np.array_equal(starts, ref.starts)
    assert np.array_equal(vcount, np.bincount(ref.verts, minlength=n).astype(np.uint32))


def _graphs():
    rp, col = synth.rmat_graph(11, 12, 5)
    dense = synth.Graph(1 << 11, rp, col, synth.thr_uniform(col.size, 0.08), "dense")
    n = 20001  # more than 32 * 256 vertices and short sets: lists from the first run on
    rp, col = synth.er_graph(n, 6 * n, 7)
    return {"harvest": dense, "lists": synth.Graph(n, rp, col, synth.thr_uniform(col.size, 0.1), "lists")}


@pytest.fixture(scope="module")
def cases():
    return {k: (g, oracle.rr_sets(g, 11, 2**32 - 700, 1500)) for k, g in _graphs().items()}


@pytest.mark.parametrize("launch", ["host", "graph", "persistent"])
@pytest.mark.parametrize("words,slots,kw", [
    (1, 1, {}), (1, 3, {}), (2, 7, dict(schedule="filtered")), (4, 2, dict(schedule="learned")), (8, 8, {}),
    (2, 1, dict(refill="batch")), (1, 2, dict(unfused=True)), (4, 1, dict(compaction="scan")), (8, 1, dict(schedule="pull")),
])
@pytest.mark.parametrize("kind", ["harvest", "lists"])
def test_rows_of_every_form(fbpt, cases, kind, words, slots, kw, launch):
    g, ref = cases[kind]
    dg = fbpt.Graph.from_synth(g)
    for _ in range(2):  # the second run starts from what the first left, with its measured set size
        rr = fbpt.sample(dg, 11, 2**32 - 700, 1500, words=words, slots=slots, launch=launch, **kw)
        assert_same(rr, ref, g.n)
    dg.close()


@pytest.mark.parametrize("kind", ["harvest", "lists"])
def test_rows_with_a_vertex_order(fbpt, cases, kind):
    g, ref = cases[kind]
    dg = fbpt.Graph.from_synth(g)
    dg.set_order(np.random.default_rng(1).permutation(g.n), sorted_starts=True)
    for launch in ("graph", "persistent"):
        assert_same(fbpt.sample(dg, 11, 2**32 - 700, 1500, words=4, slots=3, launch=launch), ref, g.n)
    dg.close()


@pytest.mark.parametrize("n,S", [(1, 70), (300, 900), (8300, 700), (2**20 + 4001, 500)])
def test_row_lengths(fbpt, n, S):
    """Disjoint chains of up to 8,300 shuffled vertices, every edge always live: sets
    of every length up to that, so every ordering kernel and, with n above 2^20, a
    bitmap of two windows."""
    perm = np.random.default_rng(n).permutation(n)
    pos = np.argsort(perm)
    has = pos % 8300 != 0  # vertex at place p of the shuffle has the one at p - 1 as its in-neighbour
    rp = np.concatenate([[0], np.cumsum(has)]).astype(np.uint64)
    col = perm[pos[has] - 1].astype(np.uint32)
    g = synth.Graph(n, rp, col, np.full(col.size, 0xFFFFFFFF, np.uint32), "chains")
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 3, 0, S)
    for _ in range(2):
        assert_same(fbpt.sample(dg, 3, 0, S, words=8, slots=1, launch="persistent"), ref, n)
    dg.close()
