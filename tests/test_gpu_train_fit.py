"""The fitting net's weight gradient where its tiles and row slices end: layers of
widths below, at and past 64 with and without skips, on frames of 33 to 300 atoms (whole
and ragged groups of 32 rows), against the oracle's double backward (FP32 sums: 1e-5
relative, as for the student)."""

import dataclasses

import numpy as np
import pytest

import synth
from oracle import OracleModel
from oracle.student import loss_and_grad

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fitting,natoms", [((20, 24), 33), ((64, 64), 64), ((68, 68, 68), 65), ((64, 132), 96),
                                            ((36, 76, 76), 300)])
def test_fitting_gradient(fitting, natoms):
    import torch

    import paper_2604_07276_gb300 as p

    cfg = dataclasses.replace(synth.STUDENT_CONFIG, fitting=fitting)
    w = synth.make_weights(cfg, seed=9, bias_scale=0.1, stats=True)
    coord, atype, box = synth.lattice_system(natoms, seed=6, density=0.015)
    n = len(atype)
    f_ref = np.random.default_rng(2).normal(size=(n, 3))
    L, _, _, g = loss_and_grad(OracleModel.from_numpy(cfg, w), coord, box, atype, 2.5, f_ref)
    m = p.DPA1(weight_file(cfg, w, "trainfit_" + "_".join(map(str, fitting))), precision="fp32")
    m.reserve(n)
    m.debug_poison()
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    m.zero_grad()
    for _ in range(2):  # two frames add up
        m.train_frame(dev(coord, torch.float64), dev(p.box9(box), torch.float64), dev(atype, torch.int32), 2.5,
                      dev(f_ref, torch.float64), loss)
    got = m.get_grad()
    assert np.linalg.norm(got - 2 * g) <= 1e-5 * np.linalg.norm(2 * g)
    assert abs(float(loss[0]) - L) <= 1e-5 * abs(L)
    m.close()


def test_bias_gradients():
    """The energy biases' own gradients (small against the others): every type's and
    b_out's within 1e-5 of the oracle's."""
    import torch

    import paper_2604_07276_gb300 as p

    cfg = synth.STUDENT_CONFIG
    w = synth.make_weights(cfg, seed=9, bias_scale=0.1, stats=True)
    coord, atype, box = synth.lattice_system(1100, seed=6, density=0.05)
    n = len(atype)
    f_ref = np.zeros((n, 3))
    _, _, _, g = loss_and_grad(OracleModel.from_numpy(cfg, w), coord, box, atype, 5e3, f_ref)
    m = p.DPA1(weight_file(cfg, w, "trainbias"), precision="fp32")
    m.reserve(n)
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    m.zero_grad()
    m.train_frame(dev(coord, torch.float64), dev(p.box9(box), torch.float64), dev(atype, torch.int32), 5e3,
                  dev(f_ref, torch.float64), loss)
    got = m.get_grad()
    m.close()
    k = 1 + cfg.ntypes  # b_out, then a bias per type
    assert np.abs(g[-k:]).min() > 0
    assert (np.abs(got[-k:] - g[-k:]) <= 1e-5 * np.abs(g[-k:])).all()
