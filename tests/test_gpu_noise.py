"""FP32 noise of the stream-collide kernels at its edges: a variance that vanishes in FP32,
one near the smallest normal number, and chunks cut by the row end, against the oracle.

One step from rest at rho = 1 leaves f - omega_i rho0 equal to the noise, so the populations
are compared relative to the noise's largest value: 1e-5, the bound of the pointwise noise
tests (the hardware sine and cosine are good to 4e-7 of it).
"""
import numpy as np
import pytest

from gpu_helpers import W9, pair

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def rest(nx, ny):
    return np.broadcast_to(W9[:, None, None], (9, ny, nx)).copy()


@pytest.mark.parametrize("launch", [(1, 128, 0), (2, 64, 2)])
@pytest.mark.parametrize("nx", [3, 6, 129, 258])
@pytest.mark.parametrize("tau,kT,power_law", [(1.0, 1e-5, 0), (0.55, 3e-4, 0), (1.3, 1e-33, 0), (0.8, 2e-6, 1)])
def test_noise_of_one_step_from_rest(tau, kT, power_law, nx, launch):
    base = dict(nx=nx, ny=5, periodic_x=1, periodic_y=1, walls_y=0, tau=tau, kT=kT, seed=2 ** 63 - 25, domain_id=7,
                power_law=power_law, n_pl=1.5, xi_pl=0.1, tau_min=0.6, tau_max=1.5)
    ref, ctx = pair(base, "f32s", f0=rest(nx, 5))
    ctx.set_launch(*launch)
    ref.step(1)
    ctx.step(1)
    noise = ref.populations() - W9[:, None, None]
    got = ctx.populations() - W9[:, None, None]
    if kT > 1e-20:
        assert np.abs(got - noise).max() <= 1e-5 * np.abs(noise).max() + 2.0 ** -52
    else:  # below the resolution of the FP64 populations read back
        assert np.abs(got).max() <= 2.0 ** -52


def test_variance_that_vanishes_in_fp32_adds_no_noise():
    """tau = 1/2 + 1e-12: omega rounds to 2 in FP32 and omega (2 - omega) is 1.6e-11 or 0."""
    base = dict(nx=70, ny=6, periodic_x=1, periodic_y=1, walls_y=0, tau=0.5 + 1e-12, kT=1e-8, seed=5)
    for store in ("f32", "f32s"):
        _, ctx = pair(base, store, f0=rest(70, 6))
        ctx.step(3)
        ctx.sync()
        got = ctx.populations() - W9[:, None, None]
        assert np.isfinite(got).all() and np.abs(got).max() < 1e-6
