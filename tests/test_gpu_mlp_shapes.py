"""The spectrum network's kernels at every launch shape on a real GB300: one sample per CTA and eight
(forward), four and eight (gradient), ragged last CTAs, and arrays aligned to one float only."""

from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlp  # noqa: E402


def _offset(a, off):
    """Device copy of a flat array that starts `off` floats after an allocation's start."""
    a = np.asarray(a, np.float32).ravel()
    t = torch.empty(a.size + off, device="cuda")
    t[off:] = torch.from_numpy(a).cuda()
    return t[off:]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("B", [1, 6, 304, 307, 608, 613])
def test_forward_and_gradient(B, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    abi.lib()
    rng = np.random.default_rng(B)
    P = mlp.param_count()
    theta = (mlp.init_params(3) + 0.05 * rng.standard_normal(P)).astype(np.float32)
    X = rng.standard_normal((B, 256)).astype(np.float32)
    Y = rng.standard_normal((B, 128)).astype(np.float32)
    used, at = theta.astype(np.float64), 0
    for i, o in mlp.LAYERS:   # the kernels round the weights to BF16
        used[at:at + i * o] = torch.from_numpy(theta[at:at + i * o]).to(torch.bfloat16).double().numpy()
        at += i * o + o
    ref, _ = mlp.forward(used, X)
    ref_g = mlp.backward(used, X.astype(np.float64), Y.astype(np.float64))
    pt, Xt, Yt = _offset(theta, off), _offset(X, off), _offset(Y, off)
    out, g, loss = torch.empty(B, 128, device="cuda"), _offset(np.ones(P), off), torch.ones(1, device="cuda")
    abi.fftenkf_mlp_forward(pt, Xt, B, out, 0)
    abi.fftenkf_mlp_gradient(pt, Xt, Yt, B, g, loss, 0)
    rel = lambda a, b: float(np.linalg.norm(a - b) / np.linalg.norm(b))   # noqa: E731
    assert rel(out.cpu().numpy().astype(np.float64), ref) <= 1e-4
    assert rel(g.cpu().numpy().astype(np.float64), ref_g) <= 1e-3
    assert abs(float(loss) - mlp.loss(ref, Y)) <= 1e-4 * mlp.loss(ref, Y)
