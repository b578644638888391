"""The level loop's iterations of two and of six levels (chosen by the levels of the
last run on the graph): runs that end at any place within one, traces included."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1, 2, 3, 4, 5, 6, 7, 11, 12, 13, 23, 24, 25, 26])
def test_runs_of_every_length(length):
    """Chains of `length` vertices with always-live edges: exactly that many levels and the start's."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as fbpt
    fbpt.build()
    n = 40 * length
    v = np.arange(n)
    first = v % length == 0
    rp = np.concatenate([[0], np.cumsum(~first)]).astype(np.uint64)
    g = synth.Graph(n, rp, (v[~first] - 1).astype(np.uint32), np.full(int((~first).sum()), 0xFFFFFFFF, np.uint32), "chains")
    dg, other = fbpt.Graph.from_synth(g), fbpt.Graph.from_synth(g)
    ref = oracle.rr_sets(g, 2, 0, 300)

    def same(rr):
        off, verts, _, vcount = rr.to_host()
        return np.array_equal(off, ref.offsets) and np.array_equal(verts, ref.verts) and \
            np.array_equal(vcount, np.bincount(ref.verts, minlength=n).astype(np.uint32))

    kw = dict(words=1, slots=8, launch="graph", spin_limit=1 << 26)
    runs = [fbpt.sample(dg, 2, 0, 300, **kw) for _ in range(3)]  # six levels an iteration first, then by what is known
    runs.append(fbpt.sample(dg, 2, 0, 300, trace_cap=64, **kw))
    assert all(same(rr) for rr in runs)
    assert len({rr.stats.levels for rr in runs}) == 1 and runs[-1].stats.trace_rows == runs[0].stats.levels
    for _ in range(2):
        outs, _ = fbpt.sample_batched([dg, other, dg], [2] * 3, [0] * 3, [300] * 3, words=1, slots=8)
        assert all(same(rr) for rr in outs)
    dg.close()
    other.close()
