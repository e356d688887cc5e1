"""Ensembles that mix power-law and Newtonian domains, with and without noise, against one
oracle per domain: the kernels are the power-law variants for every domain then, and a
Newtonian domain must still have its own relaxation time and noise variance.

Pointwise after 10 steps, over the largest |f - omega_i rho0|, with the bounds of the
pointwise noise tests.
"""
import numpy as np
import pytest

from gpu_helpers import W9, gpu_params, oracle_params
from oracle import oracle
from paper_2006_12910_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def run(store, newtonian, first):
    """Largest pointwise error of each domain: a power-law one at index `first`, Newtonian ones around it."""
    common = dict(periodic_x=1, periodic_y=1, walls_y=0, seed=77)
    doms = [dict(common, nx=70, ny=20, kT=1e-5, domain_id=1, tau=0.9, **newtonian(0.9)),
            dict(common, nx=33, ny=24, kT=0.0, domain_id=2, tau=0.62, **newtonian(0.62))]
    doms.insert(first, dict(common, nx=48, ny=16, kT=2e-5, domain_id=3, tau=1.0, power_law=1, n_pl=1.5, xi_pl=0.1,
                            tau_min=0.6, tau_max=1.5))
    ctx = lbm.Context([gpu_params(b, store) for b in doms])
    refs = []
    for d, b in enumerate(doms):
        f0 = workloads.random_populations(b["nx"], b["ny"], seed=40 + d, amp=0.01)
        ctx.set_populations(f0, dom=d)
        refs.append(oracle.Domain(oracle_params(b), f0=f0))
        refs[d].step(10)
    ctx.step(10)
    ctx.sync()
    return [np.abs(ctx.populations(dom=d) - r.populations()).max() / np.abs(r.populations() - W9[:, None, None]).max()
            for d, r in enumerate(refs)]


LIMIT = {"f64": 1e-12, "f32s": 1e-5, "f16s": 1e-3}


@pytest.mark.parametrize("first", [0, 1, 2])
@pytest.mark.parametrize("store", list(LIMIT))
def test_noise_variance(store, first):
    """xi = (tau - 1/2) / 3 is the viscosity the kernels take tau from."""
    errs = run(store, lambda tau: dict(xi_pl=(tau - 0.5) / 3, tau_min=0.51, tau_max=2.0), first)
    assert max(errs) < LIMIT[store], errs


@pytest.mark.parametrize("given", [dict(), dict(xi_pl=0.3, tau_min=0.51, tau_max=0.7, n_pl=0.5)])
@pytest.mark.parametrize("store", list(LIMIT))
def test_own_relaxation_time(store, given):
    """Power-law parameters of a domain without the power law, the defaults or any others, do nothing."""
    errs = run(store, lambda tau: given, 1)
    assert max(errs) < LIMIT[store], errs
