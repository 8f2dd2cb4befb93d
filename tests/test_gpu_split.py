"""The split passes (independent CTAs per row tile and per wavenumber column) on a real GB300: against
the FP64 oracle at the edges of their tiles and member groups, and against the pipelined passes of the
same plan, over block masks, storage types and given, drawn and caller-supplied inputs."""

from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import enkf  # noqa: E402
from synth import fields  # noqa: E402

TOL = {"f32": 1e-5, "bf16": 5e-3}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    abi.lib()


# shortest lines and fewest members; one row tile; lines of less than a warp with a last round of members
# that does not fill the groups; every 3 * 2^a plan (radices 6, 12, 24); many blocks; the longest lines
CASES = [
    (16, 16, 2, [1], "f32"), (24, 24, 3, [1, 0], "bf16"), (32, 48, 17, [1, 1, 1, 1], "f32"),
    (48, 96, 19, [0, 1, 1, 0], "f32"), (96, 192, 7, [1, 0, 0, 0, 0, 0], "bf16"), (192, 384, 5, [1, 1], "f32"),
    (384, 768, 3, [0, 1], "f32"), (768, 64, 9, [1, 1, 0], "f32"), (768, 1536, 2, [1], "bf16"),
    (1024, 32, 4, [1, 1, 1, 0], "f32"), (2048, 16, 3, [1], "f32"), (512, 2048, 2, [1, 0], "bf16"), (16, 8192, 2, [1], "f32"),
    (256, 6144, 2, [1], "f32"), (128, 128, 33, [1], "f32"),
]


def _problem(ny, nx, N, observed, storage):
    spectra = [fields.matern32_spectrum(ny, nx, 3.0 + 2.0 * b, 1.0) for b in range(len(observed))]
    kk = fields.radial_wavenumber_half(ny, nx)
    rh = np.stack([(0.05 + 0.05 * i) / np.maximum(kk, 1.0) for i in range(sum(observed))])
    return fields.make_problem(ny, nx, N, spectra, observed, rh, seed=9000 + ny + nx + N, storage=storage, rho=0.6)


@pytest.mark.parametrize("ny,nx,N,observed,storage", CASES)
def test_split_parity(ny, nx, N, observed, storage):
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    p = _problem(ny, nx, N, observed, storage)
    ref = enkf.analyze(p.ensemble, p.data, p.perturbations, p.rhat, p.observed)
    tab = enkf.spectrum_to_tables(enkf.estimate_spectrum(p.ensemble, p.observed), p.observed)
    plan = gu.plan_for(p)
    ens, data, pert, rhat = gu.to_device(p)
    forecast = ens.clone()

    def call(kind):
        u = forecast.clone()
        if kind == "given":
            plan.analyze(u, data, pert, rhat)
        elif kind == "drawn":
            plan.analyze_seeded(u, data, rhat, 31)
        else:
            plan.analyze(u, data, pert, rhat, spec)
        assert plan.device_status() == 0
        return u.float().cpu().numpy().astype(np.float64)

    spec = plan.estimate_spectrum(forecast)
    assert gu.rel_l2(spec.cpu().numpy(), tab) <= TOL[storage]
    got = {k: call(k) for k in ("given", "drawn", "spectrum")}
    assert gu.rel_l2(got["given"], ref) <= TOL[storage]
    assert gu.rel_l2(got["given"] - p.ensemble, ref - p.ensemble) <= 10 * TOL[storage]
    # the pipelined passes (any schedule entry set): the same analysis to FP32 rounding of the transforms
    # and, in BF16, to the storage rounding of the result (2^-9 of a value; the forecast dominates it)
    abi.fftenkf_set_schedule(plan.handle, [0, 1])
    spec = plan.estimate_spectrum(forecast)
    for kind, u in got.items():
        other = call(kind)
        assert gu.rel_l2(u, other) <= TOL[storage], kind
    plan.close()
