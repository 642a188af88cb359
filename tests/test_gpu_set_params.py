"""dp_set_params and dp_adam_step reach every copy of the trained weights: after either, a
model gives the same bits as one loaded from a file that holds those weights (the file's
values are FP32 ones, so both hold the same), in every precision and for each embedding
net with a kernel instance, and in MD steps replayed from a graph captured before."""

import dataclasses

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


def _fp32(w):
    return {k: np.asarray(v).astype(np.float32).astype(np.float64) for k, v in w.items()}


def _moved(w):
    """The trained arrays (embedding net, fitting net, energy biases) moved by a tenth of their size."""
    rng = np.random.default_rng(4)
    out = dict(w)
    for k, v in w.items():
        if k.startswith(("em_W", "em_b", "fit_", "ebias")):
            out[k] = v + 0.1 * np.abs(v).max() * rng.uniform(-1, 1, np.shape(v)) + 0.02 * rng.uniform(-1, 1, np.shape(v))
    if w["em_W0"].shape[0] > 1:  # concat: the type rows of the first layer are not trained
        out["em_W0"][1:] = w["em_W0"][1:]
    return _fp32(out)


CONFIGS = {
    "default": synth.DEFAULT_CONFIG,
    "concat": dataclasses.replace(synth.DEFAULT_CONFIG, tebd_input_mode="concat"),
    "paper": synth.PAPER_SIZE_CONFIG,
    "student": synth.STUDENT_CONFIG,
    "student25": dataclasses.replace(synth.STUDENT_CONFIG, embed=(25, 50, 100)),
    "student32": dataclasses.replace(synth.STUDENT_CONFIG, embed=(32, 64, 128)),
}


def _pair(name):
    cfg = CONFIGS[name]
    w = _fp32(synth.make_weights(cfg, seed=12, bias_scale=0.1))
    return weight_file(cfg, w, f"setp_{name}_a"), weight_file(cfg, _moved(w), f"setp_{name}_b")


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(np.asarray(x), np.asarray(y))


@pytest.mark.parametrize("name,precision", [
    ("default", "fp32"), ("default", "fp16x"), ("default", "bf16x"), ("default", "bf16"), ("concat", "fp16x"),
    ("concat", "bf16x"), ("paper", "bf16x"), ("student", "fp16x"), ("student25", "fp16x"), ("student25", "bf16x"),
    ("student32", "bf16x")])
def test_set_params(name, precision):
    import paper_2604_07276_gb300 as p

    first, moved = _pair(name)
    coord, atype, box = synth.lattice_system(300, seed=3, density=0.06)
    ref = p.DPA1(moved, precision=precision)
    want = ref.compute(coord, box, atype, atom_energy=True)
    m = p.DPA1(first, precision=precision)
    before = m.compute(coord, box, atype, atom_energy=True)
    assert abs(before[0] - want[0]) > 1e-2  # the move matters
    m.set_params(ref.get_params())
    _same(m.compute(coord, box, atype, atom_energy=True), want)
    ref.close()
    m.close()


@pytest.mark.parametrize("name", ["student", "student25", "student32"])
def test_adam_step(name):
    import torch

    import paper_2604_07276_gb300 as p

    first, _ = _pair(name)
    coord, atype, box = synth.lattice_system(300, seed=3, density=0.06)
    n = len(atype)
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    m = p.DPA1(first, precision="bf16x")
    m.reserve(n)
    before = m.compute(coord, box, atype, atom_energy=True)
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    m.zero_grad()
    m.train_frame(dev(coord, torch.float64), dev(p.box9(box), torch.float64), dev(atype, torch.int32), 1.0,
                  dev(np.zeros((n, 3)), torch.float64), loss)
    m.adam_step(0.02)
    torch.cuda.synchronize()
    got = m.compute(coord, box, atype, atom_energy=True)
    assert abs(got[0] - before[0]) > 1e-2
    # the parameter vector as weight arrays
    cfg = CONFIGS[name]
    w = _fp32(synth.make_weights(cfg, seed=12, bias_scale=0.1))
    theta, at = m.get_params().astype(np.float64), 0
    names = [f"em_{k}{l}" for l in range(len(cfg.embed)) for k in "Wb"]
    names += [f"fit_{k}{l}" for l in range(len(cfg.fitting) + 1) for k in "Wb"] + ["ebias"]
    for k in names:
        w[k] = theta[at:at + w[k].size].reshape(w[k].shape)
        at += w[k].size
    assert at == theta.size
    fresh = p.DPA1(weight_file(cfg, w, f"setp_{name}_trained"), precision="bf16x")
    _same(got, fresh.compute(coord, box, atype, atom_energy=True))
    fresh.close()
    m.close()


def test_captured_steps_follow():
    import torch

    import paper_2604_07276_gb300 as p
    from paper_2604_07276_gb300 import md

    first, moved = _pair("default")
    coord, atype, box = synth.water_box(0)
    vel = synth.maxwell_boltzmann(atype, 50.0, seed=11)
    ref = p.DPA1(moved, precision="fp16x")
    m = p.DPA1(first, precision="fp16x")
    state = md.MDState(coord, vel, synth.MASSES[atype], box, atype)
    x0, v0 = state.coord.clone(), state.vel.clone()
    md.run(m, state, dt=0.1, nsteps=3, graph=True)
    m.set_params(ref.get_params())
    state.coord.copy_(x0)
    state.vel.copy_(v0)
    got = md.run(m, state, dt=0.1, nsteps=3, graph=True)
    other = md.MDState(coord, vel, synth.MASSES[atype], box, atype)
    want = md.run(ref, other, dt=0.1, nsteps=3, graph=False)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and torch.equal(state.coord, other.coord)
    ref.close()
    m.close()
