"""A device allocation that fails (injected on the host) while particles are added or restored:
the call returns LBM_E_NOMEM, and the context goes on without particles instead of replaying
step graphs that hold the freed arrays; particles added afterwards behave as in a new context.
"""
import numpy as np
import pytest

from gpu_helpers import gpu_params
from paper_2006_12910_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu
BASE = dict(nx=96, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5, lj_psi=1e-4, lj_rit=2.5)
P = [dict(x=30.2, y=30.7, R=7.3, rho_p=1.2, U=0.05, V=-0.03, Omega=0.003), dict(x=60.6, y=33.1, R=6.1, rho_p=0.9, U=-0.04)]


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def context(parts=None):
    c = lbm.Context(gpu_params(BASE, "f32s", 2), particles=[parts] if parts else None)
    c.set_populations(workloads.random_populations(96, 64, seed=9, amp=0.01))
    return c


@pytest.mark.parametrize("call", ["add", "load"])
def test_goes_on_without_particles(call, tmp_path):
    src = context(P)
    src.step(3)
    src.save(tmp_path / "ck.bin")
    failed = 0
    for nth in range(1, 30):
        c = context(P[:1])
        c.step(5)
        lbm.debug_fail_alloc(nth)
        try:
            c.add_particles(0, P[1:]) if call == "add" else c.load_checkpoint(tmp_path / "ck.bin")
        except lbm.LbmError as e:
            assert e.code == -2
            failed += 1
            assert c.particles() == []
            c.step(6)
            c.sync()
            assert c.particles() == [] and np.isfinite(c.checks()).all()
            # from here on as a context that never had particles
            f = c.populations()
            d = context()
            for x in (c, d):
                x.set_populations(f)
                x.add_particles(0, P)
                x.step(7)
            assert np.array_equal(c.populations(), d.populations())
            assert c.particles() == d.particles()
        else:
            break
        finally:
            lbm.debug_fail_alloc(0)
    assert failed >= 8
