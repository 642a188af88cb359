"""The neighbour search against the brute-force list, entry for entry: candidate
counts at the edges of the register sort's sizes (32, 64, 128, 256), distances that
are equal or agree in the bits the sort sees first, and cells that wrap along one,
two or three axes with atoms given outside the box."""

import numpy as np
import pytest

from oracle.dpa1 import neighbor_list

pytestmark = pytest.mark.gpu

RCUT = 6.0


def _search(coord, box, sel):
    import torch
    import paper_2604_07276_gb300 as p

    n = len(coord)
    c = torch.tensor(coord, dtype=torch.float64, device="cuda")
    b = torch.tensor(p.box9(box), dtype=torch.float64, device="cuda")
    nl = torch.full((n, 128), -7, dtype=torch.int32, device="cuda")
    nn = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    p.binding.nlist_noalloc(c, b, RCUT, sel, nl, nn, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    return nl.cpu().numpy(), nn.cpu().numpy()


def _check(coord, box, sel=120):
    nl, nn = _search(coord, box, sel)
    ref, rnn, _ = neighbor_list(coord, box, RCUT, sel)
    assert np.array_equal(nn, rnn)
    assert np.array_equal(nl[:, :sel], ref)
    assert (nl[:, sel:] == -1).all()


def _ball(n, rng, radius):
    v = rng.normal(size=(n, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    return 10.0 + v * radius * rng.random((n, 1)) ** (1 / 3)


@pytest.mark.parametrize("cand", [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256])
@pytest.mark.parametrize("kind", ["random", "ties", "near"])
def test_candidate_counts(cand, kind):
    """cand + 1 atoms within half the cutoff of one point: cand candidates each."""
    rng = np.random.default_rng(1000 + cand)
    if kind == "random":
        coord = _ball(cand + 1, rng, 2.9)
    else:
        # sites 0.5 apart in a ball of radius 2.9 (every difference exact): shells of
        # equal distances; "near" moves them by 1e-8, below the sort's first 20 bits
        g = np.arange(-5, 6) * 0.5
        sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        sites = sites[(sites ** 2).sum(1) < 2.9 ** 2]
        coord = 10.0 + sites[rng.permutation(len(sites))[:cand + 1]]
        if kind == "near":
            coord = coord + rng.uniform(-1e-8, 1e-8, coord.shape)
    _check(coord, np.array([20.0, 20.0, 20.0]))


@pytest.mark.parametrize("box", [(12.5, 13.0, 14.0), (18.5, 12.5, 13.0), (12.5, 19.0, 25.0), (18.1, 18.2, 18.3),
                                 (40.0, 25.0, 19.0)])
@pytest.mark.parametrize("outside", [False, True])
def test_cells(box, outside):
    """One cell, three cells and more along an axis, in every mixture."""
    rng = np.random.default_rng(int(10 * sum(box)))
    box = np.array(box)
    n = int(0.06 * box.prod())
    coord = rng.random((n, 3)) * box
    coord[:6] = [[0, 0, 0], box, box * [1, 0, 0], box * [0, 0.5, 1], box * (1 - 1e-16), box * 1e-17]
    coord[:6] += rng.uniform(-0.3, 0.3, (6, 3)) * (np.arange(6)[:, None] % 2)
    if outside:
        coord = coord + rng.integers(-2, 3, (n, 3)) * box
    _check(coord, box)


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 2047, 2048, 2049])
def test_atom_counts(n):
    """Around the largest box whose cells one block sorts."""
    rng = np.random.default_rng(n)
    box = np.array([14.0, 19.0, 13.5]) * max(1.0, n / 280.0) ** (1 / 3)
    _check(rng.random((n, 3)) * box, box)


@pytest.mark.parametrize("edge", [96.5, 97.5, 195.0])
def test_many_cells(edge):
    """Few atoms in 4,096 cells and more."""
    rng = np.random.default_rng(int(edge))
    coord = rng.random((300, 3)) * edge
    coord[150:] = coord[:150] + rng.normal(size=(150, 3)) * 2.5
    _check(coord, np.array([edge, edge, edge]))
