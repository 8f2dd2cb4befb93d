"""The batched autotuner times the passes as real inputs run them: its scratch rhat is a positive, ordinary double (with
rhat = 0 every denominator vanishes, and every wavenumber takes a branch that real inputs do not); and for a batch of one shape
(its passes in series, in the tuner and in the replay) the tuned sum is the replay's time, within 20 % (three launches'
gaps of a few us on about 0.5 ms, and the spread of runs)."""

import os
import re
import struct

import pytest

torch = pytest.importorskip("torch")

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc", "batch_api.cu")


def test_scratch_rhat_is_an_ordinary_variance():
    with open(SOURCE, encoding="utf-8") as f:
        fill = re.search(r"cudaMemsetAsync\(scratch \+ field_bytes, (0x[0-9a-f]{2}), bytes - field_bytes, s\);", f.read())
    rhat, = struct.unpack("<d", bytes([int(fill.group(1), 16)]) * 8)
    assert 1e-6 < rhat < 1e3


@pytest.mark.gpu
def test_tuned_time_is_the_time_of_real_inputs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    ny, nx, N, count = 1024, 1024, 5, 8
    b = abi.fftenkf_plan_batched([(ny, nx, N)] * count, abi.FFTENKF_F32)
    ws = torch.empty(abi.fftenkf_batch_workspace_size(b), dtype=torch.uint8, device="cuda")
    tuned = abi.fftenkf_batch_autotune(b, ws, 0)
    ens = [torch.randn(N, ny, nx, device="cuda") for _ in range(count)]
    data = [torch.randn(ny, nx, device="cuda") for _ in range(count)]
    pert = [torch.randn(N, ny, nx, device="cuda") for _ in range(count)]
    rhat = [torch.full((ny, nx // 2 + 1), 0.1, dtype=torch.float64, device="cuda") for _ in range(count)]
    ms = []
    for _ in range(9):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        abi.fftenkf_analyze_batched(b, ens, data, pert, rhat, ws, int(torch.cuda.current_stream().cuda_stream))
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
    abi.fftenkf_batch_destroy(b)
    assert tuned <= 1.2 * sorted(ms)[4], (tuned, sorted(ms))
