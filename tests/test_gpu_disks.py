"""Rasterised disks whose rim touches nodes and whose box ends on them, against the oracle.

The box of a disk is taken from FP32 offsets around its nearest node; where the centre plus or
minus the radius is a node, or misses one by less than FP32 resolves, the box must still hold
every node of the disk and the ring around it.  Link counts are whole numbers and must be equal;
states after 12 steps are those of the FP64 contact tests (1e-12).
"""
import numpy as np
import pytest

from gpu_helpers import pair

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("off", [0.0, 0.5, 1e-7, -1e-7, 1e-12])
@pytest.mark.parametrize("R", [2.0, 2.5, 5.0, 8.0, 13.0])
def test_disk_boxes(R, off):
    nx, ny = 96, 48
    # on the rim exactly: held still; across the periodic corner; and one that sweeps over nodes
    parts = [dict(x=24.0 + off, y=24.0 + off, R=R, rho_p=1.1, fixed=1),
             dict(x=(off if off >= 0 else nx + off), y=2.0, R=R, rho_p=1.1, fixed=1),
             dict(x=60.0 + 1e-7, y=22.0 - 1e-7, R=R, rho_p=1.2, U=0.093, V=-0.071, Omega=0.002)]
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5, lj_psi=1e-4, lj_rit=2.5)
    ref, ctx = pair(base, "f64", particles=parts)
    for _ in range(12):
        ref.step(1)
        ctx.step(1)
        for i in range(3):
            assert np.array_equal(ctx.particle_forces(i)[9:11], ref.diag(i)[9:11])
    pr, pg = ref.particles(), ctx.particles()
    assert max(abs(a[k] - b[k]) for a, b in zip(pr, pg) for k in ("x", "y", "U", "V", "Omega")) < 1e-12
