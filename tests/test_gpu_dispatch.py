"""Which passes a call takes, by the profiling counters, on both sides of the dispatch's lines, and that the mixed
forms (split rows with pipelined columns) compute the same: with a caller's spectrum, given and drawn perturbations,
against the pipelined passes of the same plan."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu

# shape, members, observed, storage; split columns in an analysis, with a caller's spectrum, in an estimate
CASES = [
    ((64, 64, 5, [1], "f32"), (True, True, True)),
    ((768, 48, 25, [1, 1, 1, 1], "f32"), (True, False, True)),
    ((1024, 48, 25, [1, 1, 0, 0], "bf16"), (True, False, True)),
    ((192, 192, 3, [1, 1, 1], "f32"), (True, False, True)),
    ((512, 48, 25, [1, 0, 0], "f32"), (True, False, True)),
    ((512, 192, 25, [1, 0, 0], "f32"), (True, True, True)),
    ((1024, 1024, 5, [1], "f32"), (True, True, True)),
    ((1024, 2048, 3, [1, 1], "bf16"), (False, True, False)),
    ((768, 2048, 3, [1, 1, 1, 1], "bf16"), (True, False, False)),
]


@pytest.mark.parametrize("shape,split", CASES)
def test_dispatch(shape, split):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    ny, nx, N, observed, storage = shape
    tol = {"f32": 1e-5, "bf16": 5e-3}[storage]
    spectra = [fields.matern32_spectrum(ny, nx, 3.0 + 2.0 * b, 1.0) for b in range(len(observed))]
    kk = fields.radial_wavenumber_half(ny, nx)
    rh = [0.1 * (i + 1) / (1.0 + kk) for i in range(sum(observed))]
    p = fields.make_problem(ny, nx, N, spectra, observed, np.stack(rh), seed=ny + nx + N, storage=storage, rho=0.6)
    plan = gu.plan_for(p)
    forecast, data, pert, rhat = gu.to_device(p)

    def calls():
        got = {}
        spec = plan.estimate_spectrum(forecast)
        kinds = {"given": lambda u: plan.analyze(u, data, pert, rhat), "drawn": lambda u: plan.analyze_seeded(u, data, rhat, 5),
                 "supplied": lambda u: plan.analyze(u, data, pert, rhat, spec),
                 "supplied drawn": lambda u: plan.analyze_seeded(u, data, rhat, 5, spec),
                 "estimate": lambda u: plan.estimate_spectrum(u)}
        for kind, call in kinds.items():
            u = forecast.clone()
            abi.fftenkf_set_profiling(plan.handle, True)
            out = call(u)
            n = {k: v[1] for k, v in abi.fftenkf_pass_times(plan.handle).items()}
            abi.fftenkf_set_profiling(plan.handle, False)
            columns = n["col_fused"] == 1 and n["rhat_transpose"] + n["gain"] == 0
            if kind == "estimate":   # the fused pass and the split columns share a counter here
                columns = n["col_fused"] == 1 and n["col_stats"] == 0
            got[kind] = (out.double().cpu().numpy(), columns)
        assert plan.device_status() == 0
        return got

    default = calls()
    given, supplied, estimate = split
    assert [default[k][1] for k in ("given", "drawn", "supplied", "supplied drawn")] == [given, given, supplied, supplied]
    if ny != 1024:   # columns that the fused pass covers count as fused either way
        assert default["estimate"][1] == estimate
    abi.fftenkf_set_schedule(plan.handle, [0, 1])
    pipelined = calls()
    plan.close()
    for kind, (out, _) in default.items():
        assert gu.rel_l2(out, pipelined[kind][0]) <= tol, kind
