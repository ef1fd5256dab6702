"""Loss and gradient of the boundary network at the edges of the training kernel's tiles (16 rows), blocks (64)
and grid (152 blocks), against the FP64 oracle."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

# A gradient is a product of at most five values that were rounded to BF16 (weights, activations and dz; half a unit
# is 2^-9 of the value): 1e-2 to first order, taken twice.  The targets lie far from the outputs, so that the
# residual is no small difference.
TOL = 2e-2


@pytest.mark.parametrize("rows", [1, 7, 8, 15, 16, 17, 63, 64, 65, 200, 152 * 64 - 1, 152 * 64 + 1, 2 * 152 * 64 + 17])
def test_loss_and_gradient(gpu_lib, rows):
    import torch

    lee = gpu_lib
    p = omlp.init_params(3)
    rng = np.random.default_rng(rows)
    x = rng.normal(size=(rows, 16)).astype(np.float32)
    t = (3 * rng.choice([-1.0, 1.0], size=rows)).astype(np.float32)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    with lee.Mlp(p.astype(np.float32)) as m:
        grad = torch.empty(lee.MLP_NPARAM, device="cuda")
        loss = torch.empty(1, device="cuda")
        m.loss_grad(xd, td, rows, grad, loss)
        torch.cuda.synchronize()
    L, g = omlp.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64))
    assert float(loss.item()) == pytest.approx(L, rel=TOL)
    gg = grad.cpu().numpy().astype(np.float64)
    for name, (a, b) in {"W1": (0, 1024), "b1": (1024, 1088), "W2": (1088, 5184), "b2": (5184, 5248),
                         "W3": (5248, 5312), "b3": (5312, 5313)}.items():
        err = np.linalg.norm(gg[a:b] - g[a:b]) / np.linalg.norm(g[a:b])
        assert err < TOL, (name, err)
