"""Host calls on both sides of the staging limit: the results are those of a call
on device arrays, with and without atomic energies, and errors are reported once."""

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [192, 4095, 4096, 4097])
def test_host_call_equals_device_call(default_model, n):
    import torch

    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    coord, atype, box = synth.lattice_system(n, seed=n)
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp16x")
    m.reserve(n)
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    f64 = torch.float64
    E, F, W, e = (torch.zeros(s, dtype=f64, device="cuda") for s in (1, (n, 3), 9, n))
    m.compute_device(dev(coord, f64), dev(p.box9(box), f64), dev(atype, torch.int32), E, F, W, e)
    torch.cuda.synchronize()  # the host call runs on the model's own stream
    for want in (True, False):
        hE, hF, hW, he = m.compute(coord, box, atype, atom_energy=want)
        assert hE == E.item() and np.array_equal(hF, F.cpu().numpy())
        assert np.array_equal(hW.reshape(9), W.cpu().numpy())
        assert np.array_equal(he, e.cpu().numpy()) if want else he is None
    m.close()


@pytest.mark.parametrize("n", [300, 4200])
def test_device_error_is_reported_and_cleared(default_model, n):
    """300 atoms within a cell edge of each other: more candidates around an atom
    than the search holds."""
    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp32")
    rng = np.random.default_rng(0)
    crowd = rng.uniform(0.0, 2.0, size=(300, 3)) + 10.0
    far, _, box = synth.lattice_system(8000, seed=1)
    far = far[np.linalg.norm(far - 11.0, axis=1) > 10.0][: n - 300]
    coord = np.concatenate([crowd, far])
    with pytest.raises(p.DPError) as ei:
        m.compute(coord, box, np.zeros(len(coord), np.int32))
    assert ei.value.code == -4
    c, t, b = synth.water_box(0)
    m.compute(c, b, t)  # the flag is clear again
    m.close()
