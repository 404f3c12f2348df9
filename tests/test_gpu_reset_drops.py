"""Launches of several steps with auto-reset and drop lists in which a grid has no drop at some steps (a negative centre),
so that grids restart in front of steps with and without one: states, counts and done flags equal the C oracle's, for the
block sizes of the resident step, with the table and fused."""
import numpy as np
import pytest

from oracle import discrete
from paper_2512_06102_gb300 import jwf, scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [jwf.KERNEL_RESIDENT, jwf.KERNEL_FUSED])
@pytest.mark.parametrize("threads", [32, 64, 128, 256, 512, 1024])
def test_restart_in_front_of_a_step_without_a_drop(kernel, threads):
    require_gpu()
    side = np.array([40, 61, 17, 96, 33] * 12, np.int32)
    scn = scenarios.make_scenario(side, side[::-1].copy(), seed=11)
    sim = make_sim(scn, seed=6, auto_reset=True, t_max=3)
    sim.precompute_probs(*[to(a) for a in (scn.cls, scn.dem, scn.wind_speed, scn.wind_dir)])
    q = sim.probs()[0].cpu().numpy().copy()
    sim.set_kernel(kernel, threads)
    sim.load_state(to(scn.F0))
    T = 48
    drops = scenarios.drops(T, scn.H, scn.W, seed=5, p_drop=0.3)
    assert (drops[..., 0] < 0).any() and (drops[..., 0] >= 0).any()
    got = [x.cpu().numpy() for x in sim.step(T, to(drops))]
    state = sim.state().cpu().numpy()
    sim.close()
    ro = discrete.Rollout(scn.H, scn.W, scn.F0, q, scn.params.p_continue, seed=6, t_max=3, auto_reset=True)
    want = ro.step(T, drops)
    np.testing.assert_array_equal(state, ro.F)
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
