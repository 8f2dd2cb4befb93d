"""The gains' float-pair arithmetic over the range of doubles that it accepts: data-error variances and caller
spectra from 0 through subnormal and far outside a float's range, on every column path, against the FP64
oracle.  Tolerances as in test_gpu_split: state 1e-5, increment 1e-4."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coupled, enkf, sine  # noqa: E402
from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu

R = [0.0, 1e-300, 3e-41, 2e-24, 4.7e-23, 0.02, 1.0, 1e30, 2e36, 1e300]   # both sides of 2^-74 and 2^120
C = [1e-290, 1e-60, 3e-41, 2e-24, 4.7e-23, 0.5, 3.0, 1e30, 2e36, 1e40]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    abi.lib()


def _pattern(ny, nxh, n, step):
    """an index per half-spectrum wavenumber, even in k_y"""
    ky = np.minimum(np.arange(ny), ny - np.arange(ny))[:, None]
    return (step * ky + np.arange(nxh)[None, :]) % n


def _problem(ny, nx, observed, values):
    spectra = [fields.matern32_spectrum(ny, nx, 3.0 + 2.0 * b, 1.0) for b in range(len(observed))]
    rh = np.stack([np.asarray(values)[_pattern(ny, nx // 2 + 1, len(values), 3 + 2 * i)] for i in range(sum(observed))])
    p = fields.make_problem(ny, nx, 6, spectra, observed, np.full(rh.shape, 0.1), seed=77 + ny, storage="f32", rho=0.6)
    p.rhat = rh
    return p


# split passes; fused columns; separate passes (three observed blocks, and columns of 3 * 2^a)
PLANS = [(64, 32, [1, 0], False), (512, 32, [1, 0, 1], True), (512, 32, [1, 1, 0, 1], True), (96, 48, [0, 1], True)]


@pytest.mark.parametrize("ny,nx,observed,pipelined", PLANS)
@pytest.mark.parametrize("supplied", [False, True])
def test_gain_range(ny, nx, observed, pipelined, supplied):
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    p = _problem(ny, nx, observed, R)
    tab = spec_d = None
    if supplied:
        n_obs, n_un = sum(observed), len(observed) - sum(observed)
        K = ny * (nx // 2 + 1)
        tab = np.zeros(n_obs * K + 2 * n_obs * n_un * K)
        for i in range(n_obs):
            c = np.asarray(C)[_pattern(ny, nx // 2 + 1, len(C), 5 + i)]
            tab[i * K:(i + 1) * K] = c.ravel()
            for u in range(n_un):   # real and even: a real field's spectrum
                at = n_obs * K + 2 * (i * n_un + u) * K
                tab[at:at + 2 * K:2] = (0.3 - 0.5 * u) * c.ravel()
        spec_d = torch.from_numpy(tab).cuda()
    ref = enkf.analyze(p.ensemble, p.data, p.perturbations, p.rhat, p.observed, spectrum=tab)
    plan = gu.plan_for(p)
    if pipelined:
        abi.fftenkf_set_schedule(plan.handle, [0, 1])
    ens, data, pert, rhat = gu.to_device(p)
    plan.analyze(ens, data, pert, rhat, spec_d) if supplied else plan.analyze(ens, data, pert, rhat)
    assert plan.device_status() == 0
    plan.close()
    ua = ens.cpu().numpy().astype(np.float64)
    assert gu.rel_l2(ua, ref) <= 1e-5
    assert gu.rel_l2(ua - p.ensemble, ref - p.ensemble) <= 1e-4


@pytest.mark.parametrize("observed", [[1, 0], [1, 0, 1]])
def test_gain_range_coupled(observed):
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    p = _problem(64, 32, observed, [0.02, 1.0, 1e30, 2e36, 1e300])
    ref = coupled.analyze(p.ensemble, p.data, p.perturbations, p.rhat, p.observed)
    plan = gu.plan_for(p)
    abi.fftenkf_set_coupled(plan.handle, True)
    ens, data, pert, rhat = gu.to_device(p)
    plan.analyze(ens, data, pert, rhat)
    assert plan.device_status() == 0
    plan.close()
    ua = ens.cpu().numpy().astype(np.float64)
    assert gu.rel_l2(ua, ref) <= 1e-5
    assert gu.rel_l2(ua - p.ensemble, ref - p.ensemble) <= 1e-4


def test_gain_range_sine():
    from paper_1001_1588_gb300 import torch_api
    from tests import gpu_util as gu
    ny = nx = 33
    S = [fields.matern32_spectrum(ny, nx, l, 1.0) for l in (3.0, 5.0)]   # energy at every wavenumber
    p = fields.make_problem(ny, nx, 6, S, [1, 0], np.full((1, ny, nx // 2 + 1), 0.1), seed=5, storage="f32", rho=0.6)
    rhat = np.asarray(R)[_pattern(ny - 2, nx - 2, len(R), 3)][None]
    ref = sine.analyze(p.ensemble, p.data, p.perturbations, rhat, p.observed)
    plan = torch_api.SinePlan(ny, nx, 2, 6, torch.float32, [1, 0])
    ens, data, pert, _ = gu.to_device(p)
    plan.analyze(ens, data, pert, torch.from_numpy(np.ascontiguousarray(rhat)).cuda())
    assert plan.device_status() == 0
    plan.close()
    ua = ens.cpu().numpy().astype(np.float64)
    assert gu.rel_l2(ua, ref) <= 1e-5
    assert gu.rel_l2(ua - p.ensemble, ref - p.ensemble) <= 1e-4
