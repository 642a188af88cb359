"""The force gather at the edges of its register sort: clusters in which every atom
is listed by 31 ... 256 others (places 32, 64, 128, 256), against the FP64 oracle,
and frames of a batch whose partial sums do and do not fill whole groups."""

import numpy as np
import pytest

import synth
from oracle import OracleModel, energy_force_virial, neighbor_list

from gpu_helpers import weight_file, force_rmse, FP32_FORCE_RMSE

pytestmark = pytest.mark.gpu


def _cluster(n, seed):
    """n sites 0.75 A apart, jittered, inside half the cutoff of one point."""
    g = np.arange(-4, 5) * 0.75
    s = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    s = s[np.argsort((s ** 2).sum(1), kind="stable")][:n]
    rng = np.random.default_rng(seed)
    s = s + rng.uniform(-0.1, 0.1, s.shape)
    return s[rng.permutation(n)] * min(1.0, 2.95 / np.linalg.norm(s, axis=1).max()) + 9.0


@pytest.mark.parametrize("others", [31, 32, 33, 64, 65, 119, 128, 129, 256])
def test_reverse_counts(default_model, others):
    import paper_2604_07276_gb300 as p

    cfg, w, om = default_model
    n = others + 1
    coord, box = _cluster(n, others), np.array([18.0, 18.5, 19.0])
    atype = (np.arange(n) % cfg.ntypes).astype(np.int32)
    nl, _, ncand = neighbor_list(coord, box, cfg.rcut, cfg.sel)
    rev = np.bincount(nl[nl >= 0], minlength=n)
    assert (ncand == others).all()
    assert (rev == others).all() if others <= cfg.sel else rev.max() > 128 or others == 128
    rE, re, rF, rW = energy_force_virial(om, coord, box, atype)
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp32")
    m.reserve(n)
    E, F, W, _ = m.compute(coord, box, atype)
    m.close()
    # FP32 rounding of up to 512 terms, relative to the forces of these close atoms
    assert force_rmse(F, rF) <= FP32_FORCE_RMSE + 1e-4 * np.sqrt((rF ** 2).mean())
    assert np.abs(W - rW).max() <= 5e-3 * max(1.0, np.abs(rW).max())
    assert abs(E - rE) <= 1e-5 * n * max(1.0, np.abs(re).max())


@pytest.mark.parametrize("sizes", [(1, 2, 7, 8, 9), (255, 256, 257, 2048), (2049, 40, 2300)])
def test_frame_sums(default_model, sizes):
    """Energy of a frame = sum of its atomic energies, whatever its block count."""
    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp16x")
    m.reserve(sum(sizes) + 64)
    frames = []
    for k, n in enumerate(sizes):
        rng = np.random.default_rng(k)
        box = np.full(3, max(13.0, 1.05 * (n / 0.08) ** (1 / 3)))
        frames.append((rng.random((n, 3)) * box, rng.integers(0, cfg.ntypes, n).astype(np.int32), box))
    E, _, _ = m.compute_batch(frames)
    for f, (c, t, b) in enumerate(frames):
        e1, f1, w1, ea = m.compute(c, b, t, atom_energy=True)
        assert abs(e1 - ea.sum()) <= 1e-12 * len(ea) * max(1.0, np.abs(ea).max())
        assert abs(E[f] - e1) <= 1e-6 * len(ea) * max(1.0, np.abs(ea).max())
    m.close()
