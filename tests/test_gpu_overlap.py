"""Overlapped launches of the split passes cost nothing: a call among others takes no longer than its passes timed
one by one (with events between them, which keep them apart), within 10 %."""

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx,N,observed", [(48, 128, 25, [1, 1, 0, 0]), (1024, 48, 25, [1, 1, 1, 1]), (768, 64, 25, [1, 1, 0, 0])])
def test_a_call_is_no_slower_than_its_passes(ny, nx, N, observed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi, torch_api
    M, n_obs = len(observed), sum(observed)
    plan = torch_api.Plan(ny, nx, M, N, torch.float32, observed)
    ens, pert = torch.randn(M, N, ny, nx, device="cuda"), torch.randn(N, n_obs, ny, nx, device="cuda")
    data = torch.randn(n_obs, ny, nx, device="cuda")
    rhat = torch.full((n_obs, ny, nx // 2 + 1), 0.1, dtype=torch.float64, device="cuda")

    def calls():
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(20):
            plan.analyze(ens, data, pert, rhat)
        e1.record()
        e1.synchronize()
        return e0.elapsed_time(e1) / 20

    calls()
    together = sorted(calls() for _ in range(9))[4]
    abi.fftenkf_set_profiling(plan.handle, True)
    calls()
    passes = {k: v for k, v in abi.fftenkf_pass_times(plan.handle).items() if v[1]}
    plan.close()
    assert set(passes) == {"row_fwd_anomaly", "col_fused", "row_inv"}
    apart = sum(ms / n for ms, n in passes.values())
    assert together <= 1.1 * apart, (together, apart)
