"""FP32 moments on the device (lbm_moments_device) against FP64 moments of the same stored
populations, at the sizes and pointers where the vector path can go wrong.

Tolerance: the sums carry at least 40 bits, so an output is the FP32 rounding of the exact
value or its neighbour: one ulp (2^-23 relative), plus 2^-40 of the largest term where the
momentum sum cancels (terms are at most about 1).
"""
import numpy as np
import pytest

from gpu_helpers import gpu_params
from paper_2006_12910_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu
EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def expected(f, solid, gx, gy):
    fluid = solid == 0
    with np.errstate(all="ignore"):
        rho = f.sum(0)
        u = [np.where(fluid, (np.tensordot(e, f, 1) - 0.5 * rho * g) / rho, 0.0) for e, g in ((EX, gx), (EY, gy))]
    return [np.where(fluid, rho, 0.0)] + u


@pytest.mark.parametrize("store", ["f64", "f32", "f32s", "f16s", "bf16s"])
@pytest.mark.parametrize("nx,ny,shift", [(3, 3, 0), (5, 4, 0), (64, 7, 0), (64, 7, 1), (129, 33, 0), (1026, 3, 2)])
def test_moments_device_round_to_fp32(store, nx, ny, shift):
    import torch
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=3e-3, gy=-1e-4)
    solid = np.zeros((ny, nx), np.uint8)
    solid[1, nx // 2] = 1
    ctx = lbm.Context(gpu_params(base, store), solids=[solid])
    ctx.set_populations(workloads.random_populations(nx, ny, 5, 0.02, solid))
    buf = torch.full((3, nx * ny + 8), -7.0, device="cuda")
    torch.cuda.synchronize()
    out = [buf[k, shift:shift + nx * ny] for k in range(3)]
    ctx.moments_device(*out)
    ctx.sync()
    for got, want in zip(out, expected(ctx.populations(), solid, base["gx"], base["gy"])):
        np.testing.assert_allclose(got.cpu().numpy().reshape(ny, nx), want, rtol=2.0 ** -23, atol=2.0 ** -40)
    assert bool((buf[:, shift + nx * ny:] == -7.0).all()) and bool((buf[:, :shift] == -7.0).all())


def test_moments_device_of_numbers_that_are_not_ordinary():
    import torch
    nx, ny = 24, 5
    ctx = lbm.Context(gpu_params(dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8), "f32"))
    f = workloads.random_populations(nx, ny, 5, 0.02)
    f[:, 0, 1] = 0.0
    f[1, 1, 2] = np.nan
    f[2, 2, 3] = np.inf
    f[0, 3, 4] = -5.0
    f[:, 4, 5] = 3e38
    ctx.set_populations(f)
    out = torch.zeros(3, ny * nx, device="cuda")
    torch.cuda.synchronize()
    ctx.moments_device(*out)
    ctx.sync()
    with np.errstate(all="ignore"):
        want = [w.astype(np.float32) for w in expected(f.astype(np.float32).astype(np.float64), np.zeros((ny, nx)), 0.0, 0.0)]
    for got, w in zip(out.cpu().numpy().reshape(3, ny, nx), want):
        np.testing.assert_allclose(got, w, rtol=2.0 ** -23, atol=2.0 ** -40)


def test_moments_of_several_domains_in_one_buffer_keep_call_order():
    import torch
    base = dict(nx=512, ny=300, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8)
    ctx = lbm.Context([gpu_params(base, "f32s") for _ in range(6)])
    for d in range(6):
        ctx.set_populations(workloads.random_populations(512, 300, d, 0.02), dom=d)
    out = torch.zeros(3, 512 * 300, device="cuda")
    torch.cuda.synchronize()
    for d in range(6):
        ctx.moments_device(*out, dom=d)
    ctx.step(3)
    want = torch.zeros_like(out)
    ctx2 = lbm.Context(gpu_params(base, "f32s"))
    ctx2.set_populations(workloads.random_populations(512, 300, 5, 0.02))
    torch.cuda.synchronize()
    ctx2.moments_device(*want)
    ctx.sync()
    ctx2.sync()
    assert torch.equal(out, want)
