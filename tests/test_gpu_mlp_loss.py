"""Rounding of the training loss, the FP32 sum of the CTAs' losses in free order: no more than that of eight samples per
CTA.  The losses of the batch's groups of four samples (one CTA each, the same arithmetic, exactly scaled) give the
exact sum in FP64 and the expected error of adding groups of four, or of eight, one after another in FP32; the bound
on the root mean square over many batches lies between the two."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402

pytestmark = pytest.mark.gpu


def _square_errors(parts, total, rng):
    out = []
    for _ in range(10):
        acc = np.float32(0)
        for v in rng.permutation(parts):
            acc = np.float32(acc + v)
        out.append((float(acc) / total - 1.0) ** 2)
    return out


@pytest.mark.parametrize("B", [256, 600])
def test_loss_accumulation(B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    rng = np.random.default_rng(B)
    P = mlp.param_count()
    p = torch.from_numpy((mlp.init_params(3) + 0.05 * rng.standard_normal(P)).astype(np.float32)).cuda()
    g = torch.empty(P, device="cuda")
    four, eight, got = [], [], []
    for _ in range(24):
        x = torch.from_numpy(rng.standard_normal((B, 256)).astype(np.float32)).cuda()
        y = torch.from_numpy(rng.standard_normal((B, 128)).astype(np.float32)).cuda()
        part, loss = torch.empty(B // 4, device="cuda"), torch.empty(5, device="cuda")
        for i in range(B // 4):
            abi.fftenkf_mlp_gradient(p, x[4 * i:4 * i + 4].contiguous(), y[4 * i:4 * i + 4].contiguous(), 4, g, part[i:i + 1], 0)
        for i in range(5):
            abi.fftenkf_mlp_gradient(p, x, y, B, g, loss[i:i + 1], 0)
        fours = part.cpu().numpy()                        # of B = 4; the scale 4 / B is exact, or cancels in the ratio
        total = float(fours.astype(np.float64).sum())
        four += _square_errors(fours, total, rng)
        eight += _square_errors(np.float32(fours[::2] + fours[1::2]), total, rng)
        got += [(float(v) / (total * 4.0 / B) - 1.0) ** 2 for v in loss.cpu().numpy().astype(np.float64)]
    rms = [float(np.sqrt(np.mean(e))) for e in (got, four, eight)]
    assert rms[2] < rms[1]
    assert rms[0] <= np.sqrt(rms[1] * rms[2]), rms
