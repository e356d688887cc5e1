"""The overlapped chains of a step graph against the same launches one after another.

A lattice of more work items than the split rule's runs its FAR passes beside the force
launches, whose link exchange rewrites slots of the items near the disks.  Disks lie a few
nodes from item borders and from the periodic seam, so that the FAR items beside them read up
to the last node that the exchange leaves alone.  lbm_profile_steps runs every launch of a
step after the one before it; populations and particle states must be the same bits.
"""
import numpy as np
import pytest

from gpu_helpers import gpu_params
from paper_2006_12910_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("launch", [(1, 128, 0), (3, 128, 0), (2, 64, 2)])
@pytest.mark.parametrize("store,kT", [("f64", 0.0), ("f32s", 0.0), ("f32s", 1e-6), ("f16s", 0.0)])
def test_chains_equal_the_launches_in_sequence(store, kT, launch):
    nx, ny, R = 516, 1000, 6.0
    # left rims 0.3 to 9.3 nodes right of an item border (x = 128, 256), right rims left of one
    # (x = 384) and of the seam; every one moves
    parts = [dict(x=b + s * (R + 1.3 + k), y=60.0 + 90.0 * k + 25.0 * (j % 2), R=R, rho_p=1.1, U=0.02 * s, V=0.01)
             for j, (b, s) in enumerate([(128, 1), (256, 1), (384, -1), (516, -1)]) for k in range(10)]
    base = dict(nx=nx, ny=ny, periodic_x=1, periodic_y=0, walls_y=1, tau=0.8, gx=1e-6, lj_psi=1e-4, lj_rit=2.5,
                kT=kT, seed=11)
    f0 = workloads.random_populations(nx, ny, seed=3, amp=0.01)
    got = []
    for run in ("step", "profile_steps"):
        ctx = lbm.Context(gpu_params(base, store, len(parts)), particles=[parts])
        ctx.set_populations(f0)
        ctx.set_launch(*launch)
        for n in (1, 20, 7):
            getattr(ctx, run)(n)
        ctx.sync()
        got.append((ctx.populations(), ctx.particles_array()))
        ctx.close()
    assert np.array_equal(got[0][0], got[1][0])
    assert np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("before", [0, 1, 2])
def test_restored_at_an_odd_step(before, tmp_path):
    """The launches take the step's parity (their copies of states and lists) from the host;
    a checkpoint of step 7 restored into a context that has itself done 0, 1 or 2 steps
    continues as the run it was taken from."""
    base = dict(nx=96, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5, lj_psi=1e-4, lj_rit=2.5)
    parts = [dict(x=30.2, y=30.7, R=7.3, rho_p=1.2, U=0.05, V=-0.03, Omega=0.003),
             dict(x=60.6, y=33.1, R=6.1, rho_p=0.9, U=-0.04, V=0.02)]

    def ctx():
        c = lbm.Context(gpu_params(base, "f32s", 2), particles=[parts])
        c.set_populations(workloads.random_populations(96, 64, seed=9, amp=0.01))
        return c

    a, b = ctx(), ctx()
    a.step(7)
    a.save(tmp_path / "ck.bin")
    b.step(before)
    b.load_checkpoint(tmp_path / "ck.bin")
    for n in (1, 4, 6):
        a.step(n)
        b.step(n)
    assert b.step_count == 18
    assert np.array_equal(a.populations(), b.populations())
    assert a.particles() == b.particles()
