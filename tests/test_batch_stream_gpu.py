"""A batch runs, and its results lie, on one stream: the first graph's, also where
that is the default one and the other graphs have streams of their own."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_default_stream_batch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as fbpt
    fbpt.build()
    gs = [synth.rmat_wc(s) for s in (10, 12, 11)]
    dgs = [fbpt.Graph.from_synth(g, stream=s) for g, s in zip(gs, (0, torch.cuda.Stream(), torch.cuda.Stream()))]
    tasks, S = [0, 1, 2, 1], [700, 90, 3000, 64]
    for _ in range(2):
        outs, _ = fbpt.sample_batched([dgs[t] for t in tasks], [5, 6, 7, 8], [0] * 4, S, words=2, slots=2)
        assert all(not o.c.stream for o in outs)
        for i, t in enumerate(tasks):
            ref = oracle.rr_sets(gs[t], 5 + i, 0, S[i])
            off, verts, starts, vcount = outs[i].to_host()
            assert np.array_equal(off, ref.offsets) and np.array_equal(verts, ref.verts)
            assert np.array_equal(starts, ref.starts)
            assert np.array_equal(vcount, np.bincount(ref.verts, minlength=gs[t].n).astype(np.uint32))
    for dg in dgs:
        dg.close()
