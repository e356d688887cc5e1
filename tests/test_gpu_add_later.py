"""A disk added during a run, far from another, leaves that one's motion as it is.

The force of covered and uncovered nodes belongs to the change of rasterisation at the end of
the step before; adding particles rasterises anew and must not lose it.  Until the flow around
the new disk arrives (a node a step), the first disk's states are the same bits as without it.
"""
import numpy as np
import pytest

from gpu_helpers import gpu_params
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
