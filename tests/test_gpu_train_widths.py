"""The training gradient for every embedding net with a kernel instance, on frames
whose live rows fill one block, leave a ragged last one, or are a single pair,
against the oracle's double backward (FP32 sums: 1e-5 relative, as for the
student)."""

import dataclasses

import numpy as np
import pytest

import synth
from oracle import OracleModel
from oracle.student import loss_and_grad

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


def _frame(which):
    if which == "pair":
        return np.array([[20.0, 20.0, 20.0], [21.2, 20.3, 19.9]]), np.array([0, 1], np.int32), np.full(3, 40.0)
    if which == "cluster":
        return synth.isolated_cluster(5, natoms=12)
    return synth.lattice_system(80, seed=4, density=0.03)


@pytest.mark.parametrize("frame", ["pair", "cluster", "box"])
@pytest.mark.parametrize("embed", [(16, 32, 64), (25, 50, 100), (32, 64, 128)])
def test_training_gradient(embed, frame):
    import torch

    import paper_2604_07276_gb300 as p

    cfg = dataclasses.replace(synth.STUDENT_CONFIG, embed=embed)
    w = synth.make_weights(cfg, seed=8, bias_scale=0.1, stats=True)
    coord, atype, box = _frame(frame)
    f_ref = np.random.default_rng(1).normal(size=(len(atype), 3))
    L, lE, lF, g = loss_and_grad(OracleModel.from_numpy(cfg, w), coord, box, atype, 1.5, f_ref)
    m = p.DPA1(weight_file(cfg, w, f"train_{embed[0]}"), precision="fp32")
    m.reserve(len(atype))
    m.debug_poison()
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    m.zero_grad()
    m.train_frame(dev(coord, torch.float64), dev(p.box9(box), torch.float64), dev(atype, torch.int32), 1.5,
                  dev(f_ref, torch.float64), loss)
    got = m.get_grad()
    assert np.linalg.norm(got - g) <= 1e-5 * np.linalg.norm(g)
    assert abs(float(loss[0]) - L) <= 1e-5 * abs(L)
    m.close()
