"""FP32 moments of nodes whose velocity, or whose momentum, leaves the FP32 range: as the FP64
moments of the same state round to FP32, infinities included, beside ordinary nodes.
"""
import numpy as np
import pytest

from gpu_helpers import W9, gpu_params
from paper_2006_12910_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f64", "f32"])
def test_velocities_beyond_fp32(store):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny = 37, 6
    ctx = lbm.Context(gpu_params(dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5), store))
    f = np.broadcast_to(W9[:, None, None], (9, ny, nx)).copy()
    # density 1e-29 with momentum +-2e10, and momentum beyond FP32 with density 1
    f[:, 1, 3] = f[:, 4, 36] = 0.0
    f[[0, 1, 3], 1, 3] = 1e-29, 1e10, -1e10
    f[[0, 2, 4], 4, 36] = 1e-29, -1e10, 1e10
    f[:, 2, 8] = 0.0
    f[[0, 1, 3], 2, 8] = 1.0, 2e38, -2e38
    ctx.set_populations(f)
    out = [torch.full((ny, nx), float("nan"), device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    ctx.moments_device(*out)
    ctx.sync()
    with np.errstate(over="ignore"):
        want = [m.astype(np.float32) for m in ctx.moments()]
    for a, b in zip(out, want):
        assert np.allclose(a.cpu().numpy(), b, rtol=2.0 ** -23, atol=1e-12, equal_nan=True)
    assert np.isinf(want[1][1, 3]) and np.isinf(want[2][4, 36])
