"""Gradient of the warm-start network at the edges of the backward kernel's row split (single
rows, chunks of 16, 64 and 65 rows, one row past what fills the GPU evenly, unaligned outputs
through the C ABI) against a float64 evaluation with the same bfloat16 roundings.

Bound: float32 sums of n terms in chains of at most 64 rows and then of partial gradients, so a
relative 2-norm error of about sqrt(64 + 152) * 2^-24 = 8.8e-7 of sums without cancellation;
rows whose hidden values round to another bfloat16 (a relative 2^-8 of one of 128 units, in
about one row per thousand) and cancellation in the residuals y - t leave 3e-5."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_oracle as mo  # noqa: E402
from paper_2503_13075_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 16, 17, 64, 65, 152 * 16 + 1, 152 * 64 + 1])
def test_gradient_row_splits(n):
    rng = np.random.default_rng(n)
    theta = mo.init_params(5).astype(np.float32)
    # features on a coarse grid: bfloat16 holds them exactly, so the oracle's rounded inputs are
    # the kernel's in every product
    X = (rng.integers(-64, 65, size=(n, 16)) / 64.0).astype(np.float32)
    t = rng.normal(size=n).astype(np.float32)
    loss, grad = mo.loss_and_grad(theta.astype(np.float64), X, t, bf16_mode=True)
    mlp = B.Mlp(max_batch=n, seed=1)
    mlp.set_params(theta)
    xd, td = torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda()
    g, l0 = mlp.gradient(xd, td)
    assert np.linalg.norm(g.cpu().numpy() - grad) <= 3e-5 * np.linalg.norm(grad)
    assert abs(l0.item() - loss) <= 1e-5 * loss
    g2, l2 = mlp.gradient(xd, td)
    assert torch.equal(g, g2) and torch.equal(l0, l2)  # a fixed order of summation
    buf = torch.zeros(mlp.n_params + 2, device="cuda")  # a gradient that starts off a 16-byte boundary
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    code = B.lib().ilves_mlp_gradient(mlp._h, B._ptr(xd), B._ptr(td), n, ctypes.c_void_p(buf.data_ptr() + 4), None, s)
    assert code == 0 and torch.equal(buf[1:-1], g) and buf[0].item() == 0 and buf[-1].item() == 0
    assert mlp.check() == 0
