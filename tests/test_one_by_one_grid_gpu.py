"""A grid set for the level kernels does not narrow the kernels that draw samples
one by one: one CTA of 152 x 4 to 6 would take many times as long."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_level_grid_leaves_one_by_one_alone(model):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2311_10201_gb300 as fbpt
    fbpt.build()
    rp, col = synth.er_graph(20000, 160000, 31)
    thr = synth.thr_wc(rp) if model == "lt" else synth.thr_uniform(col.size, 0.05)
    dg = fbpt.Graph.from_synth(synth.Graph(20000, rp, col, thr, "er"))

    def ms(blocks):
        return min(fbpt.sample(dg, 5, 0, 100000, model=model, launch="graph", blocks=blocks).stats.ms_total
                   for _ in range(5))

    assert ms(1) < 3 * ms(0)
    dg.close()
