"""Disks that cross the periodic seams, against the oracle, step by step.

The centre is stored wrapped, so in the step of the crossing the boxes of the disk at t and
t+1 lie at opposite ends of the domain.  The rasterisation of that step must hold every node
once: the counts of changed nodes, whole numbers, are equal at every step, and forces and
states are within the bounds of the moving-particle tests (FP64 1e-12 and 1e-10 of the force,
shifted FP32 1e-6 and 1e-4).
"""
import numpy as np
import pytest

from gpu_helpers import pair, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# R = 36: a box of more nodes than the shared bitmap holds
@pytest.mark.parametrize("store", ["f64", "f32s"])
@pytest.mark.parametrize("R,nx,ny", [(3.0, 40, 33), (10.0, 514, 64), (36.0, 140, 96)])
@pytest.mark.parametrize("ux,uy", [(0.31, 0.0), (-0.31, 0.0), (0.0, 0.27), (0.0, -0.27), (0.31, 0.27), (-0.31, 0.27)])
def test_disk_crosses_the_seam(ux, uy, R, nx, ny, store):
    x = nx - 0.5 if ux > 0 else (0.5 if ux < 0 else 0.4 * nx)
    y = ny - 0.4 if uy > 0 else (0.4 if uy < 0 else 0.4 * ny)
    parts = [dict(x=x, y=y, R=R, rho_p=1.1, U=ux, V=uy, Omega=0.002)]
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5)
    ref, ctx = pair(base, store, particles=parts)
    last, crossed = parts[0], False
    for _ in range(8):
        ref.step(1)
        ctx.step(1)
        dg, do = ctx.particle_forces(0), ref.diag(0)
        assert np.array_equal(dg[9:11], do[9:11])
        assert rel(dg[:6], do[:6]) < (1e-10 if store == "f64" else 1e-4)
        q = ref.particles()[0]
        crossed |= abs(q["x"] - last["x"]) > nx / 2 or abs(q["y"] - last["y"]) > ny / 2
        last = q
    assert crossed
    pg = ctx.particles()[0]
    assert max(abs(last[k] - pg[k]) for k in ("x", "y", "U", "V", "Omega")) < (1e-12 if store == "f64" else 1e-6)
