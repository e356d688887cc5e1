"""Disks whose rim moves through the short last row segment, against the oracle.

The stream-collide pass leaves the moments of nodes that a disk covers or uncovers for the
next force launch, in the work items (row segments of 32 chunks) marked near the disk.  Where
the width is no multiple of a segment, the last one is a few nodes wide, and a disk beside the
periodic seam, or beside an open end, has rim nodes in it and beyond it.  Counts of changed
nodes are whole numbers and must be equal; states after 12 steps are within the bounds of the
contact tests (1e-12 in FP64, 1e-6 in shifted FP32).
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


@pytest.mark.parametrize("ends", ["periodic", "open"])
@pytest.mark.parametrize("last", [2, 5])
@pytest.mark.parametrize("store", ["f64", "f32s"])
def test_rims_in_the_short_last_segment(store, last, ends):
    nx, ny = {"f64": 96, "f32s": 128}[store] + last, 48
    base = dict(nx=nx, ny=ny, periodic_x=int(ends == "periodic"), inlet_outlet=int(ends == "open"), periodic_y=0,
                walls_y=1, tau=0.8, rho_in=1.001, rho_out=0.999)
    # the rim sweeps over nodes on both sides of the end of the row
    parts = [dict(x=nx - 6.05, y=14.0, R=5.0, rho_p=1.1, U=-0.09, V=0.02)]
    if ends == "periodic":
        parts.append(dict(x=3.9, y=33.0, R=5.0, rho_p=1.1, U=0.09, V=-0.02))
    ref, ctx = pair(base, store, particles=parts)
    changed = 0.0
    for _ in range(12):
        ref.step(1)
        ctx.step(1)
        for i in range(len(parts)):
            d = ref.diag(i)[9:11]
            changed += d.sum()
            assert np.array_equal(ctx.particle_forces(i)[9:11], d)
    assert changed > 0
    pr, pg = ref.particles(), ctx.particles()
    assert max(abs(a[k] - b[k]) for a, b in zip(pr, pg) for k in ("x", "y", "U", "V", "Omega")) < \
        (1e-12 if store == "f64" else 1e-6)
