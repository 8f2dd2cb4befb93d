"""The real sine variant's own row and column passes (k_sine.cuh) at the edges of their tiles and groups,
against the FP64 oracle and against the periodic analysis of the odd extension, which the shapes outside
their range (row extensions above 4096 points, ny - 1 or nx - 1 no multiple of 8, sums beyond shared memory)
go through.  Tolerances as in test_gpu_sine: FP32 storage 1e-5, BF16 5e-3; tables 1e-5."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sine  # noqa: E402
from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    abi.lib()


def _problem(ny, nx, M, N, observed, storage):
    S = [fields.se_spectrum(ny, nx, l, 1.0) for l in (4.0, 9.0, 16.0, 6.0, 5.0, 3.0)[:M]]
    n_obs = int(np.sum(observed))
    p = fields.make_problem(ny, nx, N, S, observed, np.full((n_obs, ny, nx // 2 + 1), 0.1), seed=ny + 3 * nx,
                            storage=storage, rho=0.6)
    ky, kx = np.arange(1, ny - 1)[:, None], np.arange(1, nx - 1)[None, :]
    rhat = np.stack([0.1 * (i + 1) / np.sqrt(ky ** 2 + kx ** 2) for i in range(n_obs)])
    return p, rhat


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _odd(x):
    """odd extension of [..., ny, nx] (float32 torch), boundary taken as zero"""
    x = x.clone()
    x[..., 0, :] = 0
    x[..., -1, :] = 0
    x[..., :, 0] = 0
    x[..., :, -1] = 0
    x = torch.cat([x, -x[..., 1:-1, :].flip(-2)], -2)
    return torch.cat([x, -x[..., :, 1:-1].flip(-1)], -1)


SHAPES = [
    (9, 9, 1, 2, [1], "f32"),              # one thread per line, one tile
    (17, 25, 2, 3, [1, 1], "bf16"),        # extension rows of 48, no unobserved block, an odd row count
    (13, 17, 2, 3, [1, 0], "f32"),         # ny - 1 no multiple of the tile: through the extension
    (25, 97, 3, 33, [0, 1, 0], "f32"),     # more members than groups
    (129, 33, 6, 7, [1, 0, 1, 0, 1, 1], "bf16"),   # four observed blocks
    (65, 385, 4, 20, [0, 1, 1, 1], "f32"),
    (769, 17, 2, 3, [1, 0], "f32"),        # columns of 1536
    (2049, 9, 2, 3, [0, 1], "bf16"),       # the longest columns
    (9, 1537, 1, 4, [1], "bf16"),          # rows of 3072
    (9, 2049, 2, 2, [1, 0], "f32"),        # the longest rows
    (9, 4097, 1, 2, [1], "f32"),           # longer: through the extension
]


@pytest.mark.parametrize("ny,nx,M,N,observed,storage", SHAPES)
def test_sine_passes(ny, nx, M, N, observed, storage):
    from paper_1001_1588_gb300 import torch_api
    from tests import gpu_util
    p, rhat = _problem(ny, nx, M, N, observed, storage)
    dt = torch.float32 if storage == "f32" else torch.bfloat16
    ens, data, pert, _ = gpu_util.to_device(p)
    r = torch.from_numpy(np.ascontiguousarray(rhat)).cuda()

    # the general path: the periodic analysis of the odd extension, interior taken
    plan = torch_api.Plan(2 * (ny - 1), 2 * (nx - 1), M, N, dt, observed)
    e_ens = _odd(ens.float()).to(dt).contiguous()
    e_r = torch.ones(len(rhat), 2 * (ny - 1), nx, dtype=torch.float64, device="cuda")
    e_r[:, 1:ny - 1, 1:nx - 1] = r
    e_r[:, ny:, 1:nx - 1] = r.flip(1)
    plan.analyze(e_ens, _odd(data).contiguous(), _odd(pert.float()).to(dt).contiguous(), e_r)
    general = ens.clone()
    general[..., 1:-1, 1:-1] = e_ens[..., 1:ny - 1, 1:nx - 1]
    plan.close()

    plan = torch_api.SinePlan(ny, nx, M, N, dt, observed)
    tables = plan.estimate_spectrum(ens).cpu().numpy()
    plan.analyze(ens, data, pert, r)
    assert plan.device_status() == 0
    plan.close()
    ref_t = sine.spectrum_tables(p.ensemble, p.observed)
    for t, row in enumerate(ref_t):
        assert _rel(tables.reshape(ref_t.shape)[t], row) <= 1e-5, t
    ua = ens.float().cpu().numpy().astype(np.float64)
    ref = sine.analyze(p.ensemble, p.data, p.perturbations, rhat, p.observed)
    tol = 1e-5 if storage == "f32" else 5e-3
    assert _rel(ua, ref) <= tol
    assert _rel(ua, general.float().cpu().numpy()) <= tol
    for sl in (np.s_[..., 0, :], np.s_[..., -1, :], np.s_[..., :, 0], np.s_[..., :, -1]):
        np.testing.assert_array_equal(ua[sl], p.ensemble[sl])


def test_sine_passes_status_and_capture():
    """A non-finite member is reported, and a captured analysis equals the direct one."""
    from paper_1001_1588_gb300 import abi, torch_api
    from tests import gpu_util
    p, rhat = _problem(33, 49, 3, 5, [1, 0, 1], "f32")
    ens, data, pert, _ = gpu_util.to_device(p)
    r = torch.from_numpy(np.ascontiguousarray(rhat)).cuda()
    plan = torch_api.SinePlan(33, 49, 3, 5, torch.float32, [1, 0, 1])
    direct = ens.clone()
    plan.analyze(direct, data, pert, r)
    held = ens.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.analyze(held, data, pert, r)
    assert torch.equal(held, ens)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(held, direct)
    bad = ens.clone()
    bad[0, 1, 5, 5] = float("nan")
    plan.analyze(bad, data, pert, r)
    assert plan.device_status() == abi.FFTENKF_ENONFINITE
    assert plan.device_status() == 0
    plan.close()
