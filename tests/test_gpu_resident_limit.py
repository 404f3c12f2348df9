"""Grids near the limit of shared memory: with the table and 32 threads the resident kernel takes 663 x 663 (as large as it
once took), and fewer grids than SMs that nearly fill an SM are tiled by the automatic choice, as many as SMs resident (seen
by the counters of the work done, which differ between the two kernels)."""
import numpy as np
import pytest
import torch

from oracle import discrete
from paper_2512_06102_gb300 import jwf, scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [659, 663])
@pytest.mark.parametrize("threads", [0, 32])
def test_largest_resident_grid(side, threads):
    require_gpu()
    scn = scenarios.make_scenario(side, side, N=1, seed=5)
    sim = make_sim(scn, seed=3, auto_reset=True, t_max=7)
    sim.precompute_probs(*[to(a) for a in (scn.cls, scn.dem, scn.wind_speed, scn.wind_dir)])
    q = sim.probs()[0].cpu().numpy().copy()
    sim.set_class_threads(3, 32)
    sim.set_kernel(jwf.KERNEL_RESIDENT, threads)
    sim.load_state(to(scn.F0))
    drops = scenarios.drops(10, scn.H, scn.W, seed=2)
    got = [x.cpu().numpy() for x in sim.step(10, to(drops))]
    state = sim.state().cpu().numpy()
    sim.close()
    ro = discrete.Rollout(scn.H, scn.W, scn.F0, q, scn.params.p_continue, seed=3, t_max=7, auto_reset=True)
    want = ro.step(10, drops)
    np.testing.assert_array_equal(state, ro.F)
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("H,W,many,same_as", [(617, 641, False, jwf.KERNEL_TILED_FUSED), (617, 641, True, None),
                                              (600, 600, False, None)])
def test_few_large_grids_are_tiled(H, W, many, same_as):
    require_gpu()
    n = torch.cuda.get_device_properties(0).multi_processor_count if many else 1
    scn = scenarios.make_scenario(H, W, N=1, seed=5)
    terrain = [to(scn.cls).repeat(n), to(scn.dem).repeat(n), to(scn.wind_speed).repeat(n), to(scn.wind_dir).repeat(n)]
    F0 = to(scn.F0).repeat(n)
    work, state = {}, {}
    for kernel in (jwf.KERNEL_FUSED, jwf.KERNEL_TILED_FUSED):
        sim = jwf.Sim(H, W, n_envs=n, n_classes=len(scn.params.mu_veg), seed=1)
        sim.set_params(scn.params)
        sim.set_terrain(*terrain)
        sim.set_kernel(kernel)
        sim.load_state(F0)
        counter = torch.zeros(4, dtype=torch.int64, device="cuda")
        sim.set_pair_counter(counter)
        sim.step(32)
        work[kernel] = counter[:3].tolist()
        state[kernel] = sim.state().clone()
        sim.close()
    assert torch.equal(state[jwf.KERNEL_FUSED], state[jwf.KERNEL_TILED_FUSED])
    equal = work[jwf.KERNEL_FUSED] == work[jwf.KERNEL_TILED_FUSED]
    assert equal == (same_as is not None)


def test_few_large_grids_with_auto_reset():
    """The automatic choice steps them one step a launch on the plain kernel and several on the resident one, in turn."""
    require_gpu()
    scn = scenarios.make_scenario(617, 641, N=2, seed=5)
    sim = make_sim(scn, seed=3, auto_reset=True, t_max=5)
    sim.precompute_probs(*[to(a) for a in (scn.cls, scn.dem, scn.wind_speed, scn.wind_dir)])
    q = sim.probs()[0].cpu().numpy().copy()
    sim.load_state(to(scn.F0))
    drops = scenarios.drops(12, scn.H, scn.W, seed=2, p_drop=0.5)
    outs, t = [], 0
    for k in (1, 3, 1, 1, 6):
        outs.append([x.cpu().numpy() for x in sim.step(k, to(drops[t:t + k]))])
        t += k
    state = sim.state().cpu().numpy()
    sim.close()
    ro = discrete.Rollout(scn.H, scn.W, scn.F0, q, scn.params.p_continue, seed=3, t_max=5, auto_reset=True)
    want = ro.step(12, drops)
    np.testing.assert_array_equal(state, ro.F)
    for i in range(3):
        np.testing.assert_array_equal(np.concatenate([o[i] for o in outs]), want[i])
