"""dL/dp_continue of the on-chip adjoint (jwf_relaxed_bwd_rates) over many steps: adjoints saturated at 1e35 under a p_burn of
one add up beyond float's range, and the sum stays the one in double."""
import numpy as np
import pytest
import torch

from paper_2512_06102_gb300 import scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("masked", [False, True])
def test_saturated_adjoints_add_up_beyond_float(masked):
    require_gpu()
    side, n_env, T = 128, 4, 1100
    scn = scenarios.make_scenario(side, side, N=n_env, seed=2)
    scn.params.p_continue = 1.0
    n = scn.F0.size
    sim = make_sim(scn, keep_rates=True)
    sim.precompute_probs(to(scn.cls), to(scn.dem), to(scn.wind_speed), to(scn.wind_dir))
    assert sim.relaxed_on_chip(masked)
    PU, PB = torch.zeros((T, n), device="cuda"), torch.ones((T, n), device="cuda")
    gu, gb = torch.zeros(n, device="cuda"), torch.full((n,), 1e35, device="cuda")
    au, ab = torch.empty_like(gu), torch.empty_like(gu)
    gpc = torch.zeros(1, dtype=torch.float64, device="cuda")
    sim.relaxed_bwd_rates(PU, PB, gu, gb, au, ab, torch.empty((2 * T, n), device="cuda"),
                          torch.zeros((n, 8), device="cuda"), masks=torch.zeros((T, n), device="cuda") if masked else None,
                          gpc=gpc)
    want = float(np.float32(1e35)) * n * T
    assert want / n_env / side ** 2 * 4 > float(np.finfo(np.float32).max)      # four rows of a column over the steps
    assert bool((ab == gb).all())
    # a column of 32 rows over two steps is summed in float, the columns in double
    assert abs(float(gpc) - want) <= 64 * 2.0 ** -24 * want
    sim.close()
