"""The neighbour search far from the origin: atoms thousands of boxes away, and boxes
thousands of angstroms wide, where single-precision coordinates are too coarse to tell
which pairs lie within the cutoff.  Half the pairs are placed within 1e-6 of it; the list
is the brute-force one of the same coordinates, entry for entry."""

import numpy as np
import pytest

import synth
from oracle.dpa1 import neighbor_list

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu

RCUT = 6.0


def _pairs(n, box, rng):
    """n atoms, the second half each near the cutoff from one of the first."""
    coord = rng.random((n, 3)) * box
    v = rng.normal(size=(n // 2, 3))
    v *= ((RCUT + rng.uniform(-1e-6, 1e-6, n // 2)) / np.linalg.norm(v, axis=1))[:, None]
    coord[n - n // 2:] = coord[:n // 2] + v
    return coord


def _check(coord, box, sel=120):
    import torch

    import paper_2604_07276_gb300 as p

    n = len(coord)
    nl = torch.full((n, 128), -7, dtype=torch.int32, device="cuda")
    nn = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    p.binding.nlist_noalloc(torch.tensor(coord, dtype=torch.float64, device="cuda"),
                            torch.tensor(p.box9(box), dtype=torch.float64, device="cuda"), RCUT, sel, nl, nn, st)
    assert int(st.item()) == 0
    ref, rnn, _ = neighbor_list(coord, box, RCUT, sel)
    assert np.array_equal(nn.cpu().numpy(), rnn)
    assert np.array_equal(nl.cpu().numpy()[:, :sel], ref)


@pytest.mark.parametrize("boxes", [0, 40, 5000])
@pytest.mark.parametrize("n", [300, 2048, 2500])
def test_far_atoms(n, boxes):
    rng = np.random.default_rng(n + boxes)
    box = np.array([14.0, 26.0, 19.0]) * max(1.0, n / 300.0) ** (1 / 3)
    coord = _pairs(n, box, rng)
    _check(coord + rng.integers(-boxes, boxes + 1, (n, 3)) * box, box)


@pytest.mark.parametrize("edge", [500.0, 3000.0, 50000.0])
def test_wide_boxes(edge):
    rng = np.random.default_rng(int(edge))
    box = np.array([edge, edge * 0.9, edge * 1.1])
    _check(_pairs(1000, box, rng), box)


def test_far_frames_of_a_batch(default_model):
    """A packed batch against the same frames one by one, and against the frames moved back."""
    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    rng = np.random.default_rng(8)
    near, far = [], []
    for k, n in enumerate((230, 301, 260)):
        coord, atype, box = synth.lattice_system(n, seed=60 + k, density=0.08)
        coord = np.round(coord * 2.0 ** 20) / 2.0 ** 20  # so that the shifts below are exact in FP64
        edge = np.ceil(np.asarray(box) * 4) / 4
        near.append((coord, atype, edge))
        far.append((coord + rng.integers(-30000, 30001, coord.shape) * edge, atype, edge))
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp32")
    e, f, v = m.compute_batch(far)
    for k, (coord, atype, box) in enumerate(far):
        one = m.compute(coord, box, atype)
        assert e[k] == one[0] and np.array_equal(f[k], one[1])
        home = m.compute(near[k][0], box, atype)
        # the same pairs, each displacement exact
        assert abs(e[k] - home[0]) <= 1e-5 * max(1.0, abs(home[0]))
        assert np.abs(f[k] - home[1]).max() <= 1e-4
    m.close()
