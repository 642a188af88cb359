"""Ghost atoms are no centres: a local call against the oracle's evaluation of
the local centres alone, from a workspace that holds NaN patterns."""

import numpy as np
import pytest

import synth
from oracle import energy_force_virial

from gpu_helpers import weight_file, force_rmse, FP32_FORCE_RMSE, BF16_FORCE_RMSE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp16x", "bf16x"])
@pytest.mark.parametrize("nlocal", [1, 130, 239])
def test_local_centres_only(default_model, precision, nlocal):
    import paper_2604_07276_gb300 as p

    cfg, w, om = default_model
    coord, atype, box = synth.lattice_system(240, seed=31)
    m = p.DPA1(weight_file(cfg, w, "default"), precision=precision)
    m.reserve(240)
    m.debug_poison()
    E, F, W, ae = m.compute(coord, box, atype, atom_energy=True, nlocal=nlocal)
    rE, re, rF, rW = energy_force_virial(om, coord, box, atype, centres=np.arange(nlocal))
    tol = FP32_FORCE_RMSE if precision == "fp32" else BF16_FORCE_RMSE
    assert force_rmse(F, rF) <= tol
    assert np.abs(ae[:nlocal] - re).max() <= (1e-4 if precision == "fp32" else 1e-3) and not np.any(ae[nlocal:])
    assert np.abs(W - rW).max() <= 5e-3 * max(1.0, np.abs(rW).max())
    g = m.debug("g", (240, 128, 4))
    assert np.any(g[:nlocal]) and not np.any(g[nlocal:])
    assert m.stats()[0] == max(len(set(r[r >= 0])) for r in m.debug("nlist", (240, 128), np.int32))
    m.close()
