"""``autograd.box_gradient`` is differentiable and transformable like the PyTorch
operations it stands for, on CUDA as on the CPU; the kernels behind the backward pass
against the same identity; and the backward pass with a batch of incoming gradients and
with saved tensors that come back in another layout."""

import numpy as np
import pytest

import synth

from gpu_helpers import weight_file

pytestmark = pytest.mark.gpu


def _inputs(n, seed, device):
    import torch

    g = torch.Generator().manual_seed(seed)
    rand = lambda *s: torch.randn(*s, generator=g, dtype=torch.float64)
    h = torch.diag(torch.tensor([20.0, 31.0, 17.0], dtype=torch.float64)) + rand(3, 3)
    return [t.to(device) for t in (rand(n, 3), h.reshape(9), rand(n, 3), rand(9))]


# FP64 sums of a few dozen terms of order 1 to 30 over cell edges of order 20
TOL = 1e-12


@pytest.mark.parametrize("which", range(4))
def test_forward_mode(which):
    import torch
    import torch.autograd.forward_ad as fw

    from paper_2604_07276_gb300.autograd import box_gradient

    tangent = {}
    for device in ("cpu", "cuda"):
        args, dirs = _inputs(7, 1, device), _inputs(7, 2, device)
        with fw.dual_level():
            args[which] = fw.make_dual(args[which], dirs[which])
            tangent[device] = fw.unpack_dual(box_gradient(*args)).tangent
        assert tangent[device] is not None
        # torch.func's own forward mode
        args = _inputs(7, 1, device)
        f = lambda t: box_gradient(*args[:which], t, *args[which + 1:])
        _, jv = torch.func.jvp(f, (args[which],), (dirs[which],))
        assert (jv - tangent[device]).abs().max() <= TOL
    assert tangent["cpu"].abs().max() > 1e-3
    assert (tangent["cuda"].cpu() - tangent["cpu"]).abs().max() <= TOL


def test_vmap_and_grad():
    import torch

    from paper_2604_07276_gb300.autograd import box_gradient

    frames = [_inputs(5, s, "cuda") for s in range(4)]
    ref = torch.stack([box_gradient(*f) for f in frames])
    got = torch.func.vmap(box_gradient)(*[torch.stack(t) for t in zip(*frames)])
    assert (got - ref).abs().max() <= TOL
    x, h, f, w = frames[0]
    g = torch.func.grad(lambda hh: box_gradient(x, hh, f, w).sum())(h)
    hr = h.clone().requires_grad_()
    gr, = torch.autograd.grad(box_gradient(x, hr, f, w).sum(), hr)
    assert gr.abs().max() > 1e-3 and (g - gr).abs().max() <= TOL


def test_tracing():
    import torch
    from torch.fx.experimental.proxy_tensor import make_fx

    from paper_2604_07276_gb300.autograd import box_gradient

    traced = make_fx(box_gradient)(*_inputs(6, 3, "cuda"))
    other = _inputs(6, 4, "cuda")
    assert (traced(*other) - box_gradient(*other)).abs().max() <= TOL


@pytest.mark.parametrize("n", [0, 1, 1023, 1025, 200000])
def test_kernels(n):
    """One block of the sums and several; the tolerance is n eps of the largest partial sums."""
    import torch

    from paper_2604_07276_gb300.autograd import box_gradient
    from paper_2604_07276_gb300.binding import box_gradient as kernels

    ref = box_gradient(*_inputs(n, n, "cpu"))
    got = kernels(*_inputs(n, n, "cuda")).cpu()
    assert (got - ref).abs().max() <= 1e-12 * max(1.0, n ** 0.5)
    args = _inputs(n, n, "cuda")
    args[1] = torch.zeros_like(args[1])
    with pytest.raises(torch.linalg.LinAlgError):
        kernels(*args)


def test_backward(default_model):
    import torch

    import paper_2604_07276_gb300 as p
    from paper_2604_07276_gb300 import autograd

    cfg, w, _ = default_model
    m = p.DPA1(weight_file(cfg, w, "default"), precision="fp32")
    coord, atype, box = synth.water_box(seed=0)
    t = torch.tensor(atype, dtype=torch.int32, device="cuda")

    def leaves():
        return (torch.tensor(coord, dtype=torch.float64, device="cuda").requires_grad_(),
                torch.tensor(p.box9(box), dtype=torch.float64, device="cuda").requires_grad_())

    x, h = leaves()
    e = autograd.energy(x, m, h, t)
    launched = p.kernel_launches()
    gx, gh = torch.autograd.grad(e, (x, h), retain_graph=True)
    assert p.kernel_launches() - launched == 2  # the two kernels of dE/dh
    E, F, W, _ = m.compute(coord, box, atype)
    ref = autograd.box_gradient(*(torch.tensor(np.asarray(a), dtype=torch.float64) for a in (coord, p.box9(box), F, W.reshape(9))))
    scale = max(1.0, float(ref.abs().max()))
    assert (gh.cpu() - ref).abs().max() <= 1e-10 * scale
    # a batch of incoming gradients
    up = torch.tensor([1.0, -2.0, 0.5], dtype=torch.float64, device="cuda")
    bx, bh = torch.autograd.grad(e, (x, h), up, is_grads_batched=True)
    for k in range(3):
        assert torch.equal(bx[k], up[k] * gx) and torch.equal(bh[k], up[k] * gh)
    # saved tensors that a hook gives back column by column
    with torch.autograd.graph.saved_tensors_hooks(lambda s: s, lambda s: s.t().contiguous().t() if s.dim() == 2 else s):
        x, h = leaves()
        e = autograd.energy(x, m, h, t)
        _, gs = torch.autograd.grad(e, (x, h))
    assert (gs - gh).abs().max() <= 1e-10 * scale
    m.close()
