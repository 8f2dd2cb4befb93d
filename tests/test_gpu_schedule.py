"""Schedule entries of passes without transforms are ignored: on a small grid the default launches run and the
result stays the same bit for bit.  An entry of a pass with transforms selects the passes."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu


def test_entries_without_transforms_are_ignored():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    from tests import gpu_util as gu
    p = fields.make_config2(ny=128, nx=128)
    plan = gu.plan_for(p)
    names = [abi.fftenkf_pass_name(i) for i in range(abi.fftenkf_pass_count())]
    idle = [int(n in ("mean", "gain", "chat_out", "rhat_transpose")) for n in names]
    assert sum(idle) == 4

    def run(sched):
        abi.fftenkf_set_schedule(plan.handle, sched)
        ens, data, pert, rhat = gu.to_device(p)
        abi.fftenkf_set_profiling(plan.handle, True)
        plan.analyze(ens, data, pert, rhat)
        n = {k: v[1] for k, v in abi.fftenkf_pass_times(plan.handle).items()}
        abi.fftenkf_set_profiling(plan.handle, False)
        assert plan.device_status() == 0
        return ens.cpu().numpy(), n

    want, n0 = run([0] * len(names))
    assert (n0["row_fwd_anomaly"], n0["row_fwd_innovation"], n0["col_fused"], n0["rhat_transpose"]) == (1, 0, 1, 0)
    got, n = run(idle)
    assert n == n0
    np.testing.assert_array_equal(got, want)
    for i, name in enumerate(names):
        if not idle[i]:
            _, n = run([int(j == i) for j in range(len(names))])
            assert n["row_fwd_innovation"] == n["rhat_transpose"] == 1, name
    plan.close()
