"""dE/dh by the library against the same 3 x 3 identity in PyTorch, for one block
and several, diagonal and general cells; a singular cell is refused by both."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 1023, 1025, 200000])
@pytest.mark.parametrize("general", [False, True])
def test_box_gradient(n, general):
    import torch

    from paper_2604_07276_gb300.autograd import box_gradient

    g = torch.Generator().manual_seed(n)
    x, f = (torch.randn(n, 3, generator=g, dtype=torch.float64) for _ in range(2))
    w = torch.randn(9, generator=g, dtype=torch.float64)
    h = torch.diag(torch.tensor([20.0, 31.0, 17.0], dtype=torch.float64))
    if general:
        h = (h + torch.randn(3, 3, generator=g, dtype=torch.float64))[[1, 0, 2]]
    ref = box_gradient(x, h.reshape(9), f, w)
    got = box_gradient(x.cuda(), h.reshape(9).cuda(), f.cuda(), w.cuda()).cpu()
    # sums of n FP64 products in another order: n eps of the largest partial sums
    tol = 1e-13 * max(1.0, n ** 0.5) * 10
    assert np.abs((got - ref).numpy()).max() <= tol


@pytest.mark.parametrize("device", ["cpu", "cuda"])
def test_singular_cell(device):
    import torch

    from paper_2604_07276_gb300.autograd import box_gradient

    x = torch.ones(4, 3, dtype=torch.float64, device=device)
    h = torch.zeros(9, dtype=torch.float64, device=device)
    with pytest.raises(torch.linalg.LinAlgError):
        box_gradient(x, h, x, torch.ones(9, dtype=torch.float64, device=device))
