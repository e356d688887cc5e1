"""Bounce-back, row ends and ragged chunks of both stream-collide kernels against the oracle.

A quarter of the nodes are solid at random, so that every combination of bounced directions,
enclosed fluid nodes, solid chunks and solid nodes at the row ends occurs; the widths cover
every remainder of the chunk (4 nodes, 2 in FP64) and of the row segment (32 chunks), and
rows shorter than one chunk.  Tolerances are those of the parity tests after 20 steps.
"""
import numpy as np
import pytest

from gpu_helpers import assert_close, compare_state, pair

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("store", ["f64", "f32", "f32s", "f16s"])
@pytest.mark.parametrize("ends", ["periodic", "walls", "open"])
@pytest.mark.parametrize("nx", [3, 5, 6, 7, 127, 128, 129, 130, 259])
def test_random_solids(nx, ends, store):
    ny = 9
    base = dict(nx=nx, ny=ny, periodic_x=int(ends != "open"), inlet_outlet=int(ends == "open"),
                periodic_y=int(ends == "periodic"), walls_y=int(ends != "periodic"), tau=0.8, gx=1e-5, gy=-2e-6,
                rho_in=1.001, rho_out=0.999)
    rng = np.random.default_rng(100 * nx + len(ends))
    solid = (rng.random((ny, nx)) < 0.25).astype(np.uint8)
    if ends == "open":
        solid[:, :2] = solid[:, -2:] = 0
    for launch in [(1, 128, 0), (2, 64, 2)]:
        ref, ctx = pair(base, store, solid=solid)
        ctx.set_launch(*launch)
        ref.step(20)
        ctx.step(20)
        errs, tols = compare_state(ref, ctx, store, solid)
        assert_close(errs, tols, f"{store} {launch}")
        if launch[0] == 1:
            first = ctx.populations()
    assert np.array_equal(first, ctx.populations())
