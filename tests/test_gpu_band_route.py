"""Both sides of the rule that sends a batch to the on-chip adjoint or to the column sweeps: many large grids, of which only a
few fit the GPU at once, go to the sweeps, few grids and small ones stay on chip; and on both sides the two ways give the same
results bit for bit (dL/dp_continue: the same float sums added in another order in double)."""
import numpy as np
import pytest
import torch

from paper_2512_06102_gb300 import scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


# faster: on chip for a fit, for a sampled trajectory (None: not asked)
@pytest.mark.parametrize("H,W,n_env,masked,faster", [(220, 180, 100, False, (False, False)), (220, 180, 8, False, (True, True)),
                                                     (123, 236, 137, True, (False, None)), (123, 236, 8, True, (True, None)),
                                                     (128, 128, 256, False, (False, True)), (128, 128, 80, True, (True, None)),
                                                     (33, 40, 700, False, (True, True))])
def test_both_ways_of_the_rate_adjoint(H, W, n_env, masked, faster):
    require_gpu()
    T = 4
    scn = scenarios.make_scenario(H, W, N=1, seed=9)
    one = [to(a) for a in (scn.cls, scn.dem, scn.wind_speed, scn.wind_dir)]
    scn.H, scn.W = np.full(n_env, H, np.int32), np.full(n_env, W, np.int32)
    sim = make_sim(scn, keep_rates=True)
    sim.precompute_probs(*[a.repeat(n_env) for a in one])
    assert sim.relaxed_on_chip(masked)
    for sparse, want in zip((False, True), faster):
        assert want is None or sim.relaxed_on_chip_faster(masked, sparse) == want
    n = n_env * H * W
    g = torch.Generator(device="cuda").manual_seed(1)
    f = lambda *s: torch.rand(s, device="cuda", generator=g)
    PU, PB = torch.zeros((T + 1, n), device="cuda"), torch.zeros((T + 1, n), device="cuda")
    PB[0] = (f(n) < 0.03) * f(n)
    PU[0] = 1 - PB[0]
    masks = f(T, n) * (f(T, n) < 0.1) if masked else None
    sim.relaxed_fwd_steps(PU[0], PB[0], PU[1:], PB[1:], masks=masks)
    gu, gb = f(n) - 0.5, f(n) - 0.5
    out = []
    for call in (False, True):
        au, ab = torch.empty_like(gu), torch.empty_like(gu)
        gr = torch.full((n, 8), 0.25, device="cuda")
        gpc = torch.zeros(1, dtype=torch.float64, device="cuda")
        scratch = torch.full((2 * T, n), float("nan"), device="cuda")
        if call:
            sim.relaxed_bwd_rates(PU[:T], PB[:T], gu, gb, au, ab, scratch, gr, masks=masks, gpc=gpc)
        else:
            sim.relaxed_bwd_steps(PU[:T], PB[:T], gu, gb, au, ab, masks=masks, glam=scratch[:T], gpc=gpc)
            sim.rates_accumulate(scratch[:T], PB[:T], gr, mask=masks)
        out.append((au, ab, gr, float(gpc)))
    for x, y in zip(out[0][:3], out[1][:3]):
        assert torch.equal(x, y)
    assert abs(out[0][3] - out[1][3]) <= 1e-12 * max(1.0, float((PB[:T].abs().sum())))
    sim.close()
