"""Rounding of the gradient's accumulation over the CTAs of a batch.  The gradient of 256 (and 512) samples is
compared with the FP64 sum of the gradients of its groups of four (one CTA each, the same arithmetic, exactly
scaled), so that only the accumulation differs.  Adding n partial sums one after another in FP32 leaves a relative
error of about 0.43 2^-24 sqrt(n / 2): 1.03e-7 for the 32 CTAs of eight samples of a batch of 256, 1.45e-7 for 64
of four; 1.45e-7 and 2.05e-7 at 512.  The bounds lie half-way."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,bound", [(256, 1.24e-7), (512, 1.75e-7)])
def test_gradient_accumulation(B, bound):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    rng = np.random.default_rng(B)
    P = mlp.param_count()
    p = torch.from_numpy((mlp.init_params(3) + 0.05 * rng.standard_normal(P)).astype(np.float32)).cuda()
    x = torch.from_numpy(rng.standard_normal((B, 256)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.standard_normal((B, 128)).astype(np.float32)).cuda()
    g, loss = torch.empty(P, device="cuda"), torch.empty(1, device="cuda")
    total = torch.zeros(P, dtype=torch.float64, device="cuda")
    for i in range(0, B, 4):
        abi.fftenkf_mlp_gradient(p, x[i:i + 4].contiguous(), y[i:i + 4].contiguous(), 4, g, loss, 0)
        total += g.double() * (4.0 / B)
    errs = []
    for _ in range(5):   # the order of the additions is free
        abi.fftenkf_mlp_gradient(p, x, y, B, g, loss, 0)
        errs.append(float((g.double() - total).norm() / total.norm()))
    assert sorted(errs)[2] <= bound, errs
