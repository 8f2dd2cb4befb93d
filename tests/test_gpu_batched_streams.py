"""Batched analyses issued on two streams with their own inputs and workspaces: the second call's pointer table
must not reach the first call's kernels, which may still be running.  Bitwise against the same calls one after
the other."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SPECS = [(1024, 1024, 9), (512, 1024, 9), (512, 512, 5)]


def _inputs(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)   # noqa: E731
    return ([r(N, ny, nx) for ny, nx, N in SPECS], [r(ny, nx) for ny, nx, _ in SPECS], [r(N, ny, nx) for ny, nx, N in SPECS],
            [torch.full((ny, nx // 2 + 1), 0.1, dtype=torch.float64, device="cuda") for ny, nx, _ in SPECS])


@pytest.fixture()
def batch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    b = abi.fftenkf_plan_batched(SPECS, abi.FFTENKF_F32)
    yield abi, b
    abi.fftenkf_batch_destroy(b)


def test_two_streams_with_their_own_pointers(batch):
    abi, b = batch
    n = abi.fftenkf_batch_workspace_size(b)
    sets = [(_inputs(1), torch.empty(n, dtype=torch.uint8, device="cuda")),
            (_inputs(2), torch.empty(n, dtype=torch.uint8, device="cuda"))]
    want = []
    for (ens, data, pert, rhat), ws in sets:
        u = [e.clone() for e in ens]
        abi.fftenkf_analyze_batched(b, u, data, pert, rhat, ws, 0)
        torch.cuda.synchronize()
        want.append(u)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        got = [[e.clone() for e in ens] for (ens, _, _, _), _ in sets]
        torch.cuda.synchronize()
        for s, u, ((_, data, pert, rhat), ws) in zip(streams, got, sets):
            abi.fftenkf_analyze_batched(b, u, data, pert, rhat, ws, int(s.cuda_stream))
        torch.cuda.synchronize()
        for u, w in zip(got, want):
            assert all(torch.equal(x, y) for x, y in zip(u, w))
    assert abi.fftenkf_batch_last_device_status(b, 0) == 0
