"""The fitting net's column tiles narrow as the box shrinks (and the adjoint's dZ
moves into the product): a frame's results do not depend on it.  A frame alone
against the same frame inside ever larger batches, bit for bit."""

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16x", "bf16x", "fp32"])
@pytest.mark.parametrize("config", ["default", "student"])
def test_frame_independent_of_tiles(config, precision):
    import paper_2604_07276_gb300 as p

    cfg = synth.DEFAULT_CONFIG if config == "default" else synth.STUDENT_CONFIG
    w = synth.make_weights(cfg, seed=2, bias_scale=0.1)
    m = p.DPA1(weight_file(cfg, w, f"tiles_{config}"), precision=precision)
    frame = synth.lattice_system(213, seed=9)
    other = synth.lattice_system(700, seed=10)
    E, F, W, _ = m.compute(frame[0], frame[2], frame[1])
    for k in (1, 4, 9) if config == "default" else (2, 9, 20):
        e, f, v = m.compute_batch([(c, t, b) for c, t, b in [other] * k + [frame]])
        assert e[-1] == E and np.array_equal(f[-1], F) and np.array_equal(v[-1], W)
    m.close()
