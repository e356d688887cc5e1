"""A disk added during a run, far from another, leaves that one's motion as it is.

The force of covered and uncovered nodes belongs to the change of rasterisation at the end of
the step before; adding particles rasterises anew and must not lose it.  Until the flow around
the new disk arrives (a node a step), the first disk's states are the same bits as without it.
"""
import numpy as np
import pytest

from gpu_helpers import gpu_params, pair, rel
from paper_2006_12910_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f64", "f32s"])
@pytest.mark.parametrize("at", [7, 8, 9, 10])
def test_first_disk_moves_on_unchanged(at, store):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    base = dict(nx=300, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5, lj_psi=1e-4, lj_rit=2.5)
    first = dict(x=60.2, y=30.7, R=7.3, rho_p=1.2, U=0.21, V=-0.17, Omega=0.003)
    runs = []
    for late in (False, True):
        c = lbm.Context(gpu_params(base, store, 2), particles=[[first]])
        c.set_populations(workloads.random_populations(300, 64, seed=9, amp=0.01))
        c.step(at)
        if late:
            c.add_particles(0, [dict(x=210.3, y=33.0, R=6.1, rho_p=0.9, U=-0.05, V=0.02)])
        states, changed = [], 0.0
        for _ in range(8):
            c.step(1)
            changed += c.particle_forces(0)[9:11].sum()
            states.append(c.particles_array()[0])
        runs.append((np.array(states), changed))
    assert runs[0][1] > 0 and runs[0][1] == runs[1][1]
    assert np.array_equal(runs[0][0], runs[1][0])


@pytest.mark.parametrize("store", ["f64", "f32s", "f16s"])
@pytest.mark.parametrize("at", [6, 7, 8, 9])
def test_replaced_populations_carry_the_next_force(at, store):
    """lbm_set_populations between two steps: the covered / uncovered force of the next step is
    taken from the new populations, as in the oracle (1e-10 of the force in FP64; 1e-4 and 5e-2
    in the stores that round them)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    base = dict(nx=96, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5)
    parts = [dict(x=60.2, y=30.7, R=7.3, rho_p=1.2, U=0.21, V=-0.17, Omega=0.003)]
    ref, ctx = pair(base, store, particles=parts)
    changed = 0.0
    f1 = workloads.random_populations(96, 64, seed=31, amp=0.02)
    for n in (at, 1):
        ref.step(n)
        ctx.step(n)
        f1 = 0.97 * f1
        ref.set_populations(f1)
        ctx.set_populations(f1)
        ref.step(1)
        ctx.step(1)
        dg, do = ctx.particle_forces(0), ref.diag(0)
        changed += do[9:11].sum()
        assert np.array_equal(dg[9:11], do[9:11])
        assert rel(dg[:6], do[:6]) < {"f64": 1e-10, "f32s": 1e-4, "f16s": 5e-2}[store]
    assert changed > 0
