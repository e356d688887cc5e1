"""The fixed-point collision of the FP64 store against the FP64 oracle over the range of its
format and beyond it, where single nodes fall back to FP64 arithmetic.

One collision of either kind is good to about 1e-16 of rho0 (half of what FP64 rounds to);
over 3 steps, whose streaming mixes nodes, the largest difference is held to 2e-14 of the
largest population.  The checkerboard puts in-range and out-of-range nodes into every warp.
"""
import numpy as np
import pytest

from gpu_helpers import W9, pair
from paper_2006_12910_gb300 import lbm

pytestmark = pytest.mark.gpu
EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def flow(nx, ny, rho0, umax, seed):
    """Populations near equilibrium with velocities up to umax."""
    rng = np.random.default_rng(seed)
    u, v = rng.uniform(-umax, umax, (2, ny, nx))
    r = rho0 * (1 + 0.05 * rng.standard_normal((ny, nx)))
    eu = EX[:, None, None] * u + EY[:, None, None] * v
    f = W9[:, None, None] * r * (1 + 3 * eu + 4.5 * eu ** 2 - 1.5 * (u * u + v * v))
    return f * (1 + 0.02 * rng.standard_normal(f.shape))


def agree(base, f0, steps=3):
    ref, ctx = pair(base, "f64", f0=f0)
    ref.step(steps)
    ctx.step(steps)
    a, b = ref.populations(), ctx.populations()
    assert np.isfinite(b).all()
    assert np.abs(a - b).max() <= 2e-14 * np.abs(a).max()
    ctx.sync()


@pytest.mark.parametrize("rho0", [1.0, 0.999, 1.999, 1000.0, 3e-7])
@pytest.mark.parametrize("tau,g", [(0.52, 0.0), (0.8, 1e-5), (1.9, -3e-3), (40.0, 1e-7), (0.500005, 0.0)])
def test_collision_over_the_range(rho0, tau, g):
    base = dict(nx=67, ny=8, periodic_x=1, periodic_y=1, walls_y=0, tau=tau, gx=g, gy=-0.3 * g, rho0=rho0)
    agree(base, flow(67, 8, rho0, 0.1, 3))


@pytest.mark.parametrize("what", ["fast", "small", "tiny", "zero", "negative", "dense", "all"])
def test_nodes_out_of_range(what):
    nx, ny = 70, 9
    f = flow(nx, ny, 1.0, 0.02, 5)
    odd = (np.add.outer(np.arange(ny), np.arange(nx)) % 2).astype(bool)
    if what in ("fast", "all"):
        f[:, odd] = flow(nx, ny, 1.0, 0.35, 6)[:, odd]
    if what in ("small", "all"):
        f[5, 2, ::3] = 2.0 ** -12
    if what in ("tiny", "all"):
        f[6, 4, ::5] = 1e-30
    if what in ("zero", "all"):
        f[7, 6, ::4] = 0.0
    if what in ("negative", "all"):
        f[8, ::2, ::7] = -1e-3
    if what in ("dense", "all"):
        f[:, 7, ::2] *= 5.0
    agree(dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.9, gx=1e-4), f)


def test_unstable_density_is_still_reported():
    base = dict(nx=40, ny=6, periodic_x=1, periodic_y=1, walls_y=0, tau=0.9)
    f = flow(40, 6, 1.0, 0.02, 5)
    f[0, 3, 7] = np.nan
    ctx = lbm.Context(lbm.make_params(store="f64", **base))
    ctx.set_populations(f)
    ctx.step(1)
    with pytest.raises(lbm.LbmError):
        ctx.sync()


def test_moments_of_a_small_density_and_of_zero_populations():
    import torch
    nx, ny = 34, 5
    for rho0 in (3e-7, 1e-25):
        f = flow(nx, ny, rho0, 0.05, 9)
        f[1, 2, 3] = 0.0
        ctx = lbm.Context(lbm.make_params(nx=nx, ny=ny, store="f64", rho0=rho0, tau=0.8))
        ctx.set_populations(f)
        out = torch.zeros(3, nx * ny, device="cuda")
        torch.cuda.synchronize()
        ctx.moments_device(*out)
        ctx.sync()
        rho = f.sum(0)
        want = [rho, np.tensordot(EX, f, 1) / rho, np.tensordot(EY, f, 1) / rho]
        for got, w in zip(out.cpu().numpy().reshape(3, ny, nx), want):
            np.testing.assert_allclose(got, w, rtol=2.0 ** -23, atol=2.0 ** -40 * np.abs(w).max())
