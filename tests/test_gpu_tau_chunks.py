"""tau* of a node does not depend on the nodes solved in step with it: a field moved along the
periodic direction, so that other nodes share its chunks and its warps, gives the moved result
bit for bit (last-place differences of tau* would grow where the strain is small).
"""
import numpy as np
import pytest

from gpu_helpers import W9, gpu_params
from paper_2006_12910_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32s", "f32", "f64"])
@pytest.mark.parametrize("n", [0.5, 0.75, 1.5])
def test_moved_field_gives_the_moved_result(n, store):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny = 134, 12
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=0, walls_y=1, tau=1.0, gx=2e-5, power_law=1, n_pl=n, xi_pl=0.01,
                tau_min=0.51, tau_max=2.0)
    rng = np.random.default_rng(4)
    f0 = W9[:, None, None] * (1 + 0.02 * rng.standard_normal((9, ny, nx)) * np.logspace(-3, 0, nx))
    first = None
    for move in (0, 1, 2, 3, 129):
        ctx = lbm.Context(gpu_params(base, store))
        ctx.set_populations(np.roll(f0, move, axis=2))
        ctx.step(12)
        f = np.roll(ctx.populations(), -move, axis=2)
        first = f if first is None else first
        assert np.array_equal(f, first), move
