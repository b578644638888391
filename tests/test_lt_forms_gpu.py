"""The forms that LT calls take: whole walks where they apply, levels where the
caller asks for them or a walk outgrows its path buffer."""
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


def cycles(long, short, copies):
    """One cycle of `long` vertices and `copies` cycles of `short`: always-live edges."""
    n = long + short * copies
    v = np.arange(n)
    col = np.where(v < long, (v + 1) % long, long + (v - long) // short * short + (v - long + 1) % short)
    return synth.Graph(n, np.arange(n + 1, dtype=np.uint64), col.astype(np.uint32), np.full(n, 0xFFFFFFFF, np.uint32),
                       "cycles")


@pytest.mark.parametrize("long,copies", [(1500, 1), (1500, 400)])
def test_many_warps_meet_long_walks(fbpt, long, copies):
    """Walks that outgrow the buffer in many warps at once, among short ones."""
    g = cycles(long, 20, copies)
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 8, 0, 3000, model="lt")
    for _ in range(2):
        assert_same(fbpt.sample(dg, 8, 0, 3000, words=8, slots=1, model="lt", launch="graph"), ref, g.n)
    dg.close()


def test_asked_for_levels(fbpt):
    """Host-launched levels time their expands; a barrier limit keeps the levels and their barriers."""
    g = synth.rmat_wc(12)
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 4, 0, 3000, model="lt")
    for kw in (dict(launch="host"), dict(launch="graph", spin_limit=1 << 26), dict(launch="persistent", spin_limit=1 << 26)):
        rr = fbpt.sample(dg, 4, 0, 3000, words=2, slots=2, model="lt", **kw)
        assert_same(rr, ref, g.n)
        assert rr.stats.ms_commit > 0  # levels ran
        assert (rr.stats.ms_expand_events > 0) == (kw["launch"] == "host")
    rr = fbpt.sample(dg, 4, 0, 3000, words=2, slots=2, model="lt", launch="graph")
    assert_same(rr, ref, g.n)
    assert rr.stats.ms_commit == 0  # whole walks
    dg.close()


@pytest.mark.parametrize("long", [False, True])
def test_batch_is_one_run_on_one_stream(fbpt, long):
    """Graphs on streams of their own, several tasks on one graph, and walks that are too long: one batch,
    whose results belong to the first graph's stream."""
    import torch
    gs = [synth.rmat_wc(10), synth.rmat_wc(12), cycles(1500, 20, 30) if long else synth.rmat_wc(11)]
    dgs = [fbpt.Graph.from_synth(g, stream=s) for g, s in zip(gs, (0, torch.cuda.Stream(), torch.cuda.Stream()))]
    tasks = [0, 1, 2, 1, 2, 0]
    S = [700, 1, 400, 3000, 90, 64]
    for _ in range(2):  # the second batch knows which graph's walks are long
        outs, _ = fbpt.sample_batched([dgs[t] for t in tasks], [5 + i for i in range(6)], [100 * i for i in range(6)], S,
                                      words=2, slots=2, model="lt", launch="persistent")
        assert all(not o.c.stream for o in outs)
        for i, t in enumerate(tasks):
            assert_same(outs[i], oracle.rr_sets(gs[t], 5 + i, 100 * i, S[i], model="lt"), gs[t].n)
    for dg in dgs:
        dg.close()


@pytest.mark.parametrize("launch", ["graph", "persistent", "host"])
@pytest.mark.parametrize("kind", ["first", "last", "zeros", "random", "equal"])
def test_search_by_levels(fbpt, kind, launch):
    """The level form's edge search: the rows and weights of the whole-walk test, kept on the levels."""
    from test_lt_search_gpu import graph
    g = graph(kind, 17)
    dg = fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 99, 2**32 - 2000, 6000, model="lt")
    for refill in ("lane", "batch"):
        rr = fbpt.sample(dg, 99, 2**32 - 2000, 6000, words=8, slots=2, launch=launch, model="lt", refill=refill,
                         spin_limit=1 << 26)
        assert_same(rr, ref, g.n)
        assert rr.stats.ms_commit > 0 and rr.stats.edge_accesses <= rr.stats.philox_calls
    dg.close()
