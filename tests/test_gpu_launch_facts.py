"""After one step outside a capture no launch of another length makes an attribute or occupancy query: the calls of the CUDA
runtime that a launch of many steps makes, as the profiler lists them, where its block size is another than one step's (many
small grids without auto-reset)."""
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2512_06102_gb300 import jwf, scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


def _runtime_calls(f):
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return [e.name for e in p.events()]


@pytest.mark.parametrize("kernel", [jwf.KERNEL_RESIDENT, jwf.KERNEL_FUSED])
@pytest.mark.parametrize("first,then", [(1, 24), (24, 1)])
def test_a_launch_of_another_length_makes_no_query(kernel, first, then):
    require_gpu()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # more than 1024 threads an SM at 256 a grid, fewer than 1970; a shape of its own for every case (the facts outlive a context)
    H = 37 + 2 * (kernel == jwf.KERNEL_FUSED) + (first > then)
    scn = scenarios.make_scenario(H, 61, N=6 * sms, seed=5)
    sim = make_sim(scn, seed=3)
    sim.precompute_probs(*[to(a) for a in (scn.cls, scn.dem, scn.wind_speed, scn.wind_dir)])
    sim.set_kernel(kernel)
    sim.load_state(to(scn.F0))
    _runtime_calls(lambda: torch.zeros(1, device="cuda"))     # (the profiler's own start)
    queries = ("cudaFuncSetAttribute", "cudaFuncGetAttributes", "cudaOccupancy")
    made = [[n for n in _runtime_calls(lambda: sim.step(k)) if n.startswith(queries)] for k in (first, then, then)]
    sim.close()
    if not made[0]:
        pytest.skip("the profiler lists no calls of the runtime here")
    assert made[1] == [] and made[2] == []
