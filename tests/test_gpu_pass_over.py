"""Disks that follow one another so closely that a node leaves one and enters the next in the
same step: both take the node's moments, against the oracle at every step.

Gaps of 0.15 nodes at speeds of 0.3 without the Eq. MP2 force; two disks, and three in a row
with a crowd of nodes that pass between them.  Counts of changed nodes are equal, forces and
states within the bounds of the moving-particle tests.
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


@pytest.mark.parametrize("store", ["f64", "f32s"])
@pytest.mark.parametrize("dx,dy", [(1, 0), (-1, 0), (0, 1), (0, -1)])
@pytest.mark.parametrize("n", [2, 3])
def test_nodes_passed_from_disk_to_disk(n, dx, dy, store):
    R, gap = 6.0, 0.15
    parts = [dict(x=32.05 + dx * k * (2 * R + gap), y=32.0 + dy * (0.05 + k * (2 * R + gap)) * 1.0, R=R, rho_p=1.5,
                  U=0.3 * dx, V=0.3 * dy) for k in range(n)]
    base = dict(nx=90, ny=88, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8)
    ref, ctx = pair(base, store, particles=parts)
    both = 0
    owner = owners(parts, base)
    for _ in range(5):
        ref.step(1)
        ctx.step(1)
        was, owner = owner, owners(ref.particles(), base)
        both += int(((was > 0) & (owner > 0) & (was != owner)).sum())
        for i in range(n):
            dg, do = ctx.particle_forces(i), ref.diag(i)
            assert np.array_equal(dg[9:11], do[9:11])
            assert rel(dg[:6], do[:6]) < (1e-10 if store == "f64" else 1e-4)
    assert both > 0
    pr, pg = ref.particles(), ctx.particles()
    assert max(abs(a[k] - b[k]) for a, b in zip(pr, pg) for k in ("x", "y", "U", "V", "Omega")) < \
        (1e-12 if store == "f64" else 1e-6)


def owners(parts, base):
    """Number (from 1) of the disk that covers each node, 0 for none."""
    y, x = np.mgrid[0:base["ny"], 0:base["nx"]]
    o = np.zeros(x.shape, int)
    for i, p in enumerate(parts):
        ex = (x - p["x"] + base["nx"] / 2) % base["nx"] - base["nx"] / 2
        ey = (y - p["y"] + base["ny"] / 2) % base["ny"] - base["ny"] / 2
        o[ex * ex + ey * ey < p["R"] ** 2] = i + 1
    return o
