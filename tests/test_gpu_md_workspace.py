"""Steps replayed from a captured graph after the workspace they were captured in has been
replaced by a larger one, or by another precision's and back: the same bits as eager steps."""

import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


def test_graph_after_reserve_and_precision(default_model):
    import torch

    import paper_2604_07276_gb300 as p
    from paper_2604_07276_gb300 import md

    cfg, w, _ = default_model
    coord, atype, box = synth.water_box(0)
    vel = synth.maxwell_boltzmann(atype, 50.0, seed=11)
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp16x")
    state, eager = (md.MDState(coord, vel, synth.MASSES[atype], box, atype) for _ in range(2))

    def same():
        a = md.run(m, state, dt=0.1, nsteps=3, graph=True)
        b = md.run(m, eager, dt=0.1, nsteps=3, graph=False)
        torch.cuda.synchronize()
        m.status()
        assert torch.equal(a, b) and torch.equal(state.coord, eager.coord) and torch.equal(state.vel, eager.vel)

    same()
    m.reserve(3000)
    same()
    m.reserve(3001)
    same()
    m.set_precision("fp32")
    same()
    m.set_precision("fp16x")
    same()
    m.close()
