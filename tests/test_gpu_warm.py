"""After the first step no call builds a graph: whatever count warmed the context up, later
counts are launched and nothing else (no capture, instantiation or upload in a running
simulation, no failure that belongs to set-up)."""
import pytest

from gpu_helpers import gpu_params
from paper_2006_12910_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", ["step", "prepare"])
@pytest.mark.parametrize("parts", [[], [dict(x=30.2, y=30.7, R=7.3, rho_p=1.2, U=0.02)]])
def test_later_counts_only_launch(parts, warm):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from torch.profiler import ProfilerActivity, profile
    base = dict(nx=96, ny=64, periodic_x=1, periodic_y=1, walls_y=0, tau=0.8, gx=1e-5)
    ctx = lbm.Context(gpu_params(base, "f32s", len(parts)), particles=[parts] if parts else None)
    if warm == "prepare":
        ctx.prepare_steps(20)
    ctx.step(20)
    ctx.sync()
    kinds = [ProfilerActivity.CPU, ProfilerActivity.CUDA]
    with profile(activities=kinds):  # the first one of a process starts the recording late
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
    with profile(activities=kinds) as prof:
        for n in (1, 2, 7, 20, 64, 65):
            ctx.step(n)
        ctx.sync()
    names = [e.name for e in prof.events()]
    if "cudaGraphLaunch" not in names:
        pytest.skip("the profiler records no runtime calls here")
    assert not [n for n in names if "Capture" in n or "Instantiate" in n or "GraphUpload" in n]
