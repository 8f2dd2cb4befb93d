"""The fused column pass on its own dispatch: wide columns of every length it covers (the lengths that large
analyses run), one and two observed blocks beside unobserved ones, perturbations given and drawn, pinned to the
pipelined passes by the anomaly rows' schedule with the column entries left at the wide plan.  The profiling
counters say which passes ran, so that a change of the dispatch cannot empty the tests."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import enkf, perturb  # noqa: E402
from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu
PINNED = [0, 1]   # anomaly rows narrow: no split passes


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    abi.lib()


def _problem(ny, nx, N, observed, storage):
    spectra = [fields.matern32_spectrum(ny, nx, 3.0 + 4.0 * b, 1.0) for b in range(len(observed))]
    kk = fields.radial_wavenumber_half(ny, nx)
    rh = np.stack([(0.05 + 0.05 * i) / np.maximum(kk, 1.0) for i in range(sum(observed))])
    return fields.make_problem(ny, nx, N, spectra, observed, rh, seed=6100 + ny + nx, storage=storage, rho=0.6)


def _launches(plan, call):
    from paper_1001_1588_gb300 import abi
    abi.fftenkf_set_profiling(plan.handle, True)
    call()
    n = {k: v[1] for k, v in abi.fftenkf_pass_times(plan.handle).items()}
    abi.fftenkf_set_profiling(plan.handle, False)
    return n


CASES = [(512, 64, [1, 0, 1, 0], "f32"), (1024, 48, [0, 1, 0], "f32"), (1024, 96, [1, 1, 0, 0], "bf16"),
         (2048, 32, [1, 1, 0], "f32"), (2048, 48, [0, 0, 1], "bf16"), (2048, 16, [1], "f32"), (4096, 32, [1, 0], "f32")]


@pytest.mark.parametrize("ny,nx,observed,storage", CASES)
def test_wide_fused_columns(ny, nx, observed, storage):
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    tol = {"f32": 1e-5, "bf16": 5e-3}[storage]
    p = _problem(ny, nx, 5, observed, storage)
    plan = gu.plan_for(p)
    abi.fftenkf_set_schedule(plan.handle, PINNED)
    ens, data, pert, rhat = gu.to_device(p)
    drawn = ens.clone()
    tables = []
    n = _launches(plan, lambda: tables.append(plan.estimate_spectrum(ens)))
    assert (n["row_fwd_anomaly"], n["col_fused"], n["col_stats"]) == (1, 1, 0)
    tab = enkf.spectrum_to_tables(enkf.estimate_spectrum(p.ensemble, p.observed), p.observed)
    assert gu.rel_l2(tables[0].cpu().numpy(), tab) <= tol
    e = perturb.perturbations(p.ny, p.nx, p.rhat, 99, p.N)
    for u, e_k, call in ((ens, p.perturbations, lambda: plan.analyze(ens, data, pert, rhat)),
                         (drawn, e, lambda: plan.analyze_seeded(drawn, data, rhat, 99))):
        n = _launches(plan, call)
        # the split columns read rhat as it is and take both kinds of rows in one launch
        assert (n["rhat_transpose"], n["row_fwd_anomaly"], n["row_fwd_innovation"], n["col_fused"]) == (1, 1, 1, 1)
        assert n["col_stats"] == n["col_update"] == 0
        ref = enkf.analyze(p.ensemble, p.data, e_k, p.rhat, p.observed)
        got = u.float().cpu().numpy().astype(np.float64)
        assert gu.rel_l2(got, ref) <= tol
        assert gu.rel_l2(got - p.ensemble, ref - p.ensemble) <= 10 * tol
    assert plan.device_status() == 0
    plan.close()


@pytest.mark.parametrize("ny,nx,observed", [(96, 64, [1, 0]), (64, 96, [1, 1, 1, 0]), (768, 48, [0, 1])])
def test_separate_columns_drawn(ny, nx, observed):
    """Columns that the fused pass does not cover: statistics and update, perturbations drawn in the update."""
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    p = _problem(ny, nx, 6, observed, "f32")
    plan = gu.plan_for(p)
    abi.fftenkf_set_schedule(plan.handle, PINNED)
    ens, data, _, rhat = gu.to_device(p)
    n = _launches(plan, lambda: plan.analyze_seeded(ens, data, rhat, 7))
    assert (n["col_stats"], n["col_update"], n["col_fused"]) == (1, 1, 0)
    assert plan.device_status() == 0
    plan.close()
    ref = enkf.analyze(p.ensemble, p.data, perturb.perturbations(p.ny, p.nx, p.rhat, 7, p.N), p.rhat, p.observed)
    got = ens.cpu().numpy().astype(np.float64)
    assert gu.rel_l2(got, ref) <= 1e-5
    assert gu.rel_l2(got - p.ensemble, ref - p.ensemble) <= 1e-4
