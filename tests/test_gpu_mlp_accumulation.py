"""Rounding of the gradient's accumulation over the CTAs of a batch: no more than that of eight samples per CTA,
added to the result in FP32 in free order.  The gradients of the batch's groups of four samples (one CTA each, the
same arithmetic, exactly scaled) give the exact sum in FP64, and the expected error of adding groups of four, or of
eight, one after another in FP32; the bound lies between the two."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402

pytestmark = pytest.mark.gpu


def _expected(parts, total):
    """Relative error of adding the parts in FP32 one after another, mean of five orders."""
    errs = []
    for seed in range(5):
        acc = torch.zeros_like(parts[0])
        for i in np.random.default_rng(seed).permutation(len(parts)):
            acc += parts[i]
        errs.append(float((acc.double() - total).norm() / total.norm()))
    return sum(errs) / len(errs)


@pytest.mark.parametrize("B", [256, 512])
def test_gradient_accumulation(B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    rng = np.random.default_rng(B)
    P = mlp.param_count()
    p = torch.from_numpy((mlp.init_params(3) + 0.05 * rng.standard_normal(P)).astype(np.float32)).cuda()
    x = torch.from_numpy(rng.standard_normal((B, 256)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.standard_normal((B, 128)).astype(np.float32)).cuda()
    g, loss = torch.empty(P, device="cuda"), torch.empty(1, device="cuda")
    fours = []
    for i in range(0, B, 4):
        abi.fftenkf_mlp_gradient(p, x[i:i + 4].contiguous(), y[i:i + 4].contiguous(), 4, g, loss, 0)
        fours.append(g * (4.0 / B))
    total = sum(f.double() for f in fours)
    of_four, of_eight = _expected(fours, total), _expected([a + b for a, b in zip(fours[::2], fours[1::2])], total)
    assert of_eight < of_four
    errs = []
    for _ in range(9):   # the order of the additions is free
        abi.fftenkf_mlp_gradient(p, x, y, B, g, loss, 0)
        errs.append(float((g.double() - total).norm() / total.norm()))
    assert sum(errs) / len(errs) <= (of_four * of_eight) ** 0.5, (errs, of_four, of_eight)
