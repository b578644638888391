"""Calls of both models on one graph: the size of one model's sets says nothing
about the other's, so neither makes the other's calls run twice."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_no_reruns_when_models_alternate():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as fbpt
    fbpt.build()
    g = synth.rmat_wc(14)
    dg = fbpt.Graph.from_synth(g)
    for _ in range(2):
        for model in ("ic", "lt"):
            rr = fbpt.sample(dg, 6, 0, 20000, words=8, slots=8, model=model, launch="graph")
            ref = oracle.rr_sets(g, 6, 0, 20000, model=model)
            off, verts, starts, _ = rr.to_host()
            assert np.array_equal(off, ref.offsets) and np.array_equal(verts, ref.verts)
            assert rr.stats.overflow_reruns == 0
    dg.close()
