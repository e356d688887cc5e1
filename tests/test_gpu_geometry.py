"""lbm_set_geometry on a context that has run: nodes that stay fluid keep their populations,
nodes that turn fluid start at rest with density rho0, solid ones read as zero.

A quarter of the nodes are solid, so that chunks mix solid and fluid nodes (whose vector
stores leave meaningless values in the solid slots); an eighth of all nodes change.  Rest is
exact up to one rounding of the store and of f - omega_i rho0 in FP64.
"""
import numpy as np
import pytest

from gpu_helpers import W9, assert_close, compare_state, oracle_params, pair
from oracle import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("rho0", [1.0, 0.9])
@pytest.mark.parametrize("store", ["f64", "f32", "f32s", "f16s", "bf16s"])
def test_nodes_that_turn_fluid_start_at_rest(store, rho0):
    nx, ny = 131, 24
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=0, walls_y=1, tau=0.8, gx=1e-5, rho0=rho0)
    rng = np.random.default_rng(17)
    solid = (rng.random((ny, nx)) < 0.25).astype(np.uint8)
    _, ctx = pair(base, store, solid=solid)
    ctx.step(11)
    before = ctx.populations()
    other = solid ^ (rng.random((ny, nx)) < 0.125)
    ctx.set_geometry(0, other)
    after = ctx.populations()
    stay, fresh = (solid == 0) & (other == 0), (solid != 0) & (other == 0)
    assert fresh.sum() > 50
    assert np.array_equal(after[:, stay], before[:, stay])
    assert np.all(after[:, other != 0] == 0.0)
    assert np.abs(after[:, fresh] - rho0 * W9[:, None]).max() <= (2.0 ** -25 if store == "f32" else 2.0 ** -53)
    ref = oracle.Domain(oracle_params(base), solid=other, f0=after)
    ref.step(10)
    ctx.step(10)
    ctx.sync()
    if rho0 == 1.0:  # the inputs have density 1: shifted by 0.9 they are outside what the store bounds are for
        errs, tols = compare_state(ref, ctx, store, other, rho0=rho0)
        assert_close(errs, tols, store)
