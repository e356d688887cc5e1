"""Side changes of nodes: their tags belong to one run and lead to the right slots.

A checkpoint of one small disk at step 10 is restored into a context that has itself run 40
steps with three larger disks over the same nodes; it must continue as the run it was taken
from, bit for bit (no tag of the context's earlier run may be taken for one of a step to come).
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


@pytest.mark.parametrize("store", ["f64", "f32s"])
def test_restored_over_a_longer_run(store, tmp_path):
    base = dict(nx=100, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5)

    def ctx(parts):
        c = lbm.Context(gpu_params(base, store, 3), particles=[parts])
        c.set_populations(workloads.random_populations(100, 64, seed=9, amp=0.01))
        return c

    a = ctx([dict(x=40.2, y=30.7, R=3.3, rho_p=1.2, U=0.2, V=-0.1, Omega=0.003)])
    b = ctx([dict(x=36.0, y=31.0, R=9.0, rho_p=1.2, U=0.11, V=-0.13), dict(x=57.0, y=30.0, R=9.5, rho_p=1.2, U=0.21, V=0.05),
             dict(x=80.0, y=30.0, R=10.0, rho_p=1.2, U=-0.03, V=0.2)])
    a.step(10)
    a.save(tmp_path / "ck.bin")
    b.step(40)
    b.sync()
    b.load_checkpoint(tmp_path / "ck.bin")
    for n in (1, 8, 21):
        a.step(n)
        b.step(n)
    assert np.array_equal(a.populations(), b.populations())
    assert a.particles() == b.particles()
