"""Tall narrow grids with many members on a real GB300: the inverse row pass's CTAs take several items
each and read their staged forecast rows with 16 rows of 16 or 32 points to a warp, so that a stage's
next copy must wait for reads still queued behind bank conflicts."""

from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import enkf  # noqa: E402
from synth import fields  # noqa: E402


@pytest.mark.parametrize("sched", [[0], [0, 0, 1]])   # all default; the pipelined passes, inverse rows default
@pytest.mark.parametrize("ny,nx,N,observed", [(2048, 32, 19, [1, 1, 0, 0]), (1536, 64, 19, [1, 0]), (1024, 48, 25, [0, 1, 0])])
def test_narrow_grid(ny, nx, N, observed, sched):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    spectra = [fields.matern32_spectrum(ny, nx, 3.0 + 2.0 * b, 1.0) for b in range(len(observed))]
    rh = np.full((sum(observed), ny, nx // 2 + 1), 0.1)
    p = fields.make_problem(ny, nx, N, spectra, observed, rh, seed=ny + nx, storage="f32", rho=0.6)
    plan = gu.plan_for(p)
    abi.fftenkf_set_schedule(plan.handle, sched)
    ens, data, pert, rhat = gu.to_device(p)
    plan.analyze(ens, data, pert, rhat)
    assert plan.device_status() == 0
    ua = ens.cpu().numpy().astype(np.float64)
    plan.close()
    ref = enkf.analyze(p.ensemble, p.data, p.perturbations, p.rhat, p.observed)
    assert gu.rel_l2(ua, ref) <= 1e-5
    assert gu.rel_l2(ua - p.ensemble, ref - p.ensemble) <= 1e-4
