"""Calls on the model's own stream after device calls that are still under way on others:
the results are those of the same calls one at a time."""

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


def _dev(a, t):
    import torch

    return torch.tensor(np.asarray(a), dtype=t, device="cuda")


def _device_args(p, frame):
    import torch

    coord, atype, box = frame
    f64 = torch.float64
    return [_dev(coord, f64), _dev(p.box9(box), f64), _dev(atype, torch.int32)] + [
        torch.zeros(s, dtype=f64, device="cuda") for s in (1, (len(atype), 3), 9, len(atype))]


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("precision", ["fp32", "fp16x", "bf16x"])
def test_host_calls_after_device_calls(default_model, precision, side_stream):
    import torch

    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    frames = [synth.lattice_system(n, seed=n, density=0.08) for n in (900, 301, 640)]
    m = p.DPA1(weight_file(cfg, w, "default"), precision=precision)
    m.reserve(1000)
    alone = [m.compute(c, b, t, atom_energy=True) for c, t, b in frames]
    batch = m.compute_batch(frames)
    args = _device_args(p, frames[0])
    stream = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    for k in (1, 2, 0):
        with torch.cuda.stream(stream):
            m.compute_device(*args)
        coord, atype, box = frames[k]
        got = m.compute(coord, box, atype, atom_energy=True)
        for a, b in zip(got, alone[k]):
            assert np.array_equal(a, b)
        assert args[3].item() == alone[0][0] and np.array_equal(args[4].cpu().numpy(), alone[0][1])
        with torch.cuda.stream(stream):
            m.compute_device(*args)
        e, f, v = m.compute_batch(frames)
        assert np.array_equal(e, batch[0]) and np.array_equal(v, batch[2])
        assert all(np.array_equal(a, b) for a, b in zip(f, batch[1]))
    m.close()


def test_host_call_after_replays(default_model):
    """A graph that the caller captured runs device calls the library does not see."""
    import torch

    import paper_2604_07276_gb300 as p

    cfg, w, _ = default_model
    frames = [synth.lattice_system(n, seed=n, density=0.08) for n in (900, 301)]
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp16x")
    m.reserve(1000)
    want = [m.compute(c, b, t) for c, t, b in frames]
    args = _device_args(p, frames[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        m.compute_device(*args)
    for _ in range(3):
        graph.replay()
        got = m.compute(frames[1][0], frames[1][2], frames[1][1])
        assert all(np.array_equal(a, b) for a, b in zip(got[:3], want[1][:3]))
        assert args[3].item() == want[0][0] and np.array_equal(args[4].cpu().numpy(), want[0][1])
    m.close()


def test_host_call_after_training_step():
    import torch

    import paper_2604_07276_gb300 as p

    cfg = synth.STUDENT_CONFIG
    m = p.DPA1(weight_file(cfg, synth.make_weights(cfg, seed=12, bias_scale=0.1), "order_student"), precision="fp32")
    coord, atype, box = synth.lattice_system(300, seed=3, density=0.06)
    m.reserve(300)
    c, b, t = _device_args(p, (coord, atype, box))[:3]
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    f_ref = torch.zeros((300, 3), dtype=torch.float64, device="cuda")
    before = m.compute(coord, box, atype)
    m.zero_grad()
    for _ in range(4):
        m.train_frame(c, b, t, 1.0, f_ref, loss)
    m.adam_step(0.02)
    got = m.compute(coord, box, atype)
    torch.cuda.synchronize()
    again = m.compute(coord, box, atype)
    assert got[0] == again[0] != before[0] and np.array_equal(got[1], again[1])
    m.close()


@pytest.mark.parametrize("graph", [False, True])
def test_md_behind_the_default_stream(default_model, graph):
    """The arrays of a run are filled by copies that wait behind other work of the default stream."""
    import torch

    import paper_2604_07276_gb300 as p
    from paper_2604_07276_gb300 import md

    cfg, w, _ = default_model
    coord, atype, box = synth.water_box(0)
    vel = synth.maxwell_boltzmann(atype, 50.0, seed=11)
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp16x")
    state = md.MDState(coord, vel, synth.MASSES[atype], box, atype)
    x0, v0 = state.coord.clone(), state.vel.clone()
    big = torch.zeros(1 << 28, device="cuda")
    runs = []
    for busy in (False, True):
        state.coord.zero_().add_(torch.arange(3 * len(atype), device="cuda").reshape(-1, 3) * 0.01)
        torch.cuda.synchronize()
        if busy:
            for _ in range(60):  # some milliseconds
                big.add_(1.0)
        state.coord.copy_(x0)
        state.vel.copy_(v0)
        thermo = md.run(m, state, dt=0.1, nsteps=2, graph=graph)
        runs.append((thermo.clone(), state.coord.clone(), state.vel.clone()))
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    m.close()


def test_training_calls_on_the_current_stream():
    """zero_grad and adam_step without a stream follow train_frame, which runs on PyTorch's current one."""
    import torch

    import paper_2604_07276_gb300 as p

    cfg = synth.STUDENT_CONFIG
    m = p.DPA1(weight_file(cfg, synth.make_weights(cfg, seed=12, bias_scale=0.1), "order_student"), precision="fp32")
    frame = synth.lattice_system(300, seed=3, density=0.06)
    m.reserve(300)
    c, b, t = _device_args(p, frame)[:3]
    loss = torch.zeros(3, dtype=torch.float64, device="cuda")
    f_ref = torch.zeros((300, 3), dtype=torch.float64, device="cuda")
    big = torch.zeros(1 << 28, device="cuda")
    m.zero_grad()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(40):  # some milliseconds
            big.add_(1.0)
        m.train_frame(c, b, t, 1.0, f_ref, loss)
        m.zero_grad()
        assert not m.get_grad().any()
        before = m.get_params()
        for _ in range(40):
            big.add_(1.0)
        m.train_frame(c, b, t, 1.0, f_ref, loss)
        m.adam_step(0.02)
        after = m.get_params()
    assert np.mean(after != before) > 0.9
    assert not m.get_grad().any()  # the step clears it
    m.close()
