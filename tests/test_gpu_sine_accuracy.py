"""FP32 analyses of the real sine variant through its own passes are no further from the FP64 oracle than through the
periodic analysis of the odd extension (which transforms real lines of the same length by half-length complex ones):
mean error over six draws, small grids, where a line has the fewest stages and formed twiddle powers weigh most."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sine  # noqa: E402
from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx,N,observed", [(65, 65, 5, [1, 0]), (129, 257, 6, [1, 1, 0])])
def test_sine_error_against_the_extension(ny, nx, N, observed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import torch_api
    from tests import gpu_util
    from tests.test_gpu_sine_passes import _odd
    M, n_obs = len(observed), sum(observed)
    own, general = [], []
    for seed in range(6):
        S = [fields.matern32_spectrum(ny, nx, l, 1.0) for l in (8.0, 20.0, 12.0)[:M]]
        p = fields.make_problem(ny, nx, N, S, observed, np.full((n_obs, ny, nx // 2 + 1), 0.1), seed=seed, storage="f32", rho=0.6)
        rhat = np.full((n_obs, ny - 2, nx - 2), 0.1)
        ref = sine.analyze(p.ensemble, p.data, p.perturbations, rhat, p.observed)
        ens, data, pert, _ = gpu_util.to_device(p)
        r = torch.from_numpy(rhat).cuda()
        e_ens = _odd(ens).contiguous()
        e_r = torch.full((n_obs, 2 * (ny - 1), nx), 0.1, dtype=torch.float64, device="cuda")
        plan = torch_api.Plan(2 * (ny - 1), 2 * (nx - 1), M, N, torch.float32, observed)
        plan.analyze(e_ens, _odd(data).contiguous(), _odd(pert).contiguous(), e_r)
        plan.close()
        gen = ens.clone()
        gen[..., 1:-1, 1:-1] = e_ens[..., 1:ny - 1, 1:nx - 1]
        plan = torch_api.SinePlan(ny, nx, M, N, torch.float32, observed)
        plan.analyze(ens, data, pert, r)
        plan.close()
        own.append(gpu_util.rel_l2(ens.cpu().numpy(), ref))
        general.append(gpu_util.rel_l2(gen.cpu().numpy(), ref))
    assert sum(own) <= sum(general), (own, general)
