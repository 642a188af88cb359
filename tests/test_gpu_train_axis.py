"""The training gradient over descriptor axis widths (the tangent kernels spread the
axis columns' sums over the block: one column, an odd number, as many as the embedding
is wide), against the oracle's double backward (FP32 sums: 1e-5 relative, as for the
student)."""

import dataclasses

import numpy as np
import pytest

import synth
from oracle import OracleModel, energy_force_virial
from oracle.student import loss_and_grad

from gpu_helpers import BF16_ATOM_ENERGY, BF16_FORCE_RMSE, force_rmse, weight_file

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("embed,axis", [((16, 32, 64), 1), ((16, 32, 64), 64), ((25, 50, 100), 7), ((32, 64, 128), 40)])
def test_axis(embed, axis):
    import torch

    import paper_2604_07276_gb300 as p

    cfg = dataclasses.replace(synth.STUDENT_CONFIG, embed=embed, axis=axis, fitting=(32, 32))
    w = synth.make_weights(cfg, seed=10, bias_scale=0.1, stats=True)
    coord, atype, box = synth.lattice_system(70, seed=7, density=0.03)
    n = len(atype)
    f_ref = np.random.default_rng(3).normal(size=(n, 3))
    L, _, _, g = loss_and_grad(OracleModel.from_numpy(cfg, w), coord, box, atype, 0.5, f_ref)
    m = p.DPA1(weight_file(cfg, w, f"trainaxis_{embed[0]}_{axis}"), precision="fp32")
    m.reserve(n)
    m.debug_poison()
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    m.zero_grad()
    m.train_frame(dev(coord, torch.float64), dev(p.box9(box), torch.float64), dev(atype, torch.int32), 0.5,
                  dev(f_ref, torch.float64), loss)
    got = m.get_grad()
    assert np.linalg.norm(got - g) <= 1e-5 * np.linalg.norm(g)
    assert abs(float(loss[0]) - L) <= 1e-5 * abs(L)
    m.close()


@pytest.mark.parametrize("axis", [1, 7, 48, 64])
def test_axis_interleaved(axis):
    """The descriptor and its adjoint on the column-quad layout (fp16x), forces and
    atomic energies against the FP64 oracle."""
    import paper_2604_07276_gb300 as p

    cfg = dataclasses.replace(synth.STUDENT_CONFIG, axis=axis, fitting=(32, 32))
    w = synth.make_weights(cfg, seed=11, bias_scale=0.1, stats=True)
    coord, atype, box = synth.lattice_system(70, seed=8, density=0.03)
    _, re, rF, _ = energy_force_virial(OracleModel.from_numpy(cfg, w), coord, box, atype)
    m = p.DPA1(weight_file(cfg, w, f"axis_{axis}"), precision="fp16x")
    m.reserve(len(atype))
    m.debug_poison()
    _, F, _, e = m.compute(coord, box, atype, atom_energy=True)
    m.close()
    assert force_rmse(F, rF) <= BF16_FORCE_RMSE
    assert np.abs(e - re).max() <= BF16_ATOM_ENERGY
