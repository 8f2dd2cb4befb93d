"""The morphing forward transform's tiles of 16 and of 8 rows: ragged right and bottom tiles, displacements
beyond the staged halo (which gather from global memory); and no tiles, for few nodes and for narrow
planes.  Against the FP64 oracle.  Tolerance as in test_gpu_morph: relative L2 1e-5."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import morph  # noqa: E402
from synth import fields  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,ny,nx,amp", [(3, 20, 250, 250, 2.5), (2, 10, 256, 224, 9.0), (1, 21, 245, 225, 12.0),
                                            (2, 3, 61, 90, 4.0), (1, 5, 600, 70, 7.0)])
def test_morph_forward_tiles(M, K, ny, nx, amp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_1588_gb300 import abi
    u = fields.smooth_members(31, M, K, ny, nx, ell=12.0)
    u_ref = fields.smooth_members(32, M, 1, ny, nx, ell=12.0)[:, 0]
    T = fields.smooth_mappings(33, K, ny, nx, amp=amp, ell=40.0)
    ext = torch.zeros((M + 2, K, ny, nx), dtype=torch.float32, device="cuda")
    ext[:2] = torch.from_numpy(np.ascontiguousarray(T, dtype=np.float32)).cuda()
    dev = [torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (u, u_ref)]
    abi.fftenkf_morph_forward(dev[0], dev[1], ext, M, K, ny, nx, 20, 0.0)
    torch.cuda.synchronize()
    got = ext.cpu().numpy().astype(np.float64)
    ref = morph.morph_forward(u, u_ref, T, 20, 0.0)
    assert np.linalg.norm(got[2:] - ref) <= 1e-5 * np.linalg.norm(ref)
