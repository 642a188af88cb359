"""dp_debug_copy of a layer's input: rows past an atom's last neighbour read as zeros in
every layout, whatever the workspace held before the call."""

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16x", "fp16x", "bf16"])
@pytest.mark.parametrize("model", ["student", "default"])
def test_rows_past_the_last_neighbour(model, precision):
    import paper_2604_07276_gb300 as p

    cfg = synth.STUDENT_CONFIG if model == "student" else synth.DEFAULT_CONFIG
    m = p.DPA1(weight_file(cfg, synth.make_weights(cfg, seed=1), f"debugrows_{model}"), precision=precision)
    coord, atype, box = synth.lattice_system(200, seed=5, density=0.04)
    n, m1 = len(atype), cfg.embed[-1]
    m.reserve(n)
    m.debug_poison()
    m.compute(coord, box, atype)
    live = m.debug("nlist", (n, 128), dtype=np.int32) >= 0
    assert 0 < live.sum() < live.size
    for l in range(cfg.attn_layers + 1):
        G = m.debug(f"G{l}", (n, 128, m1))
        assert np.isfinite(G).all()
        assert (G[~live] == 0).all()
        assert (np.abs(G[live]).max(-1) > 0).all()
    m.close()
