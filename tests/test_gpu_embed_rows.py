"""The FP32 embedding net over live-row lists: nets without a tensor-core
instance (and models with more types than its tables hold), from one live row
up to several tiles with a ragged last one, against the oracle.  FP32 sums of
at most 128 terms: a relative force error of 1e-5 leaves a margin of ten."""

import dataclasses

import numpy as np
import pytest

import synth
from oracle import OracleModel, energy_force_virial

from gpu_helpers import weight_file, force_rmse

pytestmark = pytest.mark.gpu

STUDENT = synth.STUDENT_CONFIG
NINE = dataclasses.replace(synth.DEFAULT_CONFIG, ntypes=9, type_map=tuple("ABCDEFGHI"), attn_layers=0, out_scale=1.0)
CONFIGS = {
    "student": STUDENT,
    "student_concat": dataclasses.replace(STUDENT, tebd_input_mode="concat"),
    "nine_types": NINE,
}


def _system(which):
    if which == "pair":
        return np.array([[20.0, 20.0, 20.0], [21.2, 20.3, 19.9]]), np.array([0, 1], np.int32), np.full(3, 40.0)
    if which == "cluster":
        return synth.isolated_cluster(5, natoms=12)
    return synth.lattice_system(240, seed=3) if which == "box" else synth.lattice_system(70, seed=4, density=0.03)


@pytest.mark.parametrize("system", ["pair", "cluster", "sparse", "box"])
@pytest.mark.parametrize("name", ["student", "student_concat", "nine_types"])
@pytest.mark.parametrize("precision", ["fp16x", "fp32"])
def test_embed_rows(name, precision, system):
    import paper_2604_07276_gb300 as p

    cfg = CONFIGS[name]
    w = synth.make_weights(cfg, seed=6, bias_scale=0.1, stats=True)
    coord, atype, box = _system(system)
    E, e, F, W = energy_force_virial(OracleModel.from_numpy(cfg, w), coord, box, atype)
    m = p.DPA1(weight_file(cfg, w, f"rows_{name}"), precision=precision)
    m.reserve(len(atype))
    m.debug_poison()
    _, f, _, ae = m.compute(coord, box, atype, atom_energy=True)
    assert force_rmse(f, F) <= 1e-5 * np.sqrt(np.mean(F * F))
    assert np.abs(ae - e).max() <= 1e-5 * max(1.0, np.abs(e).max())
    m.close()
