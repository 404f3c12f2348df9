"""Infinities and NaN in the relaxed kernels that pass over cells without a burning neighbour: rates and p_un that are not
finite, ahead of the fire and at it, give in the on-chip kernels what they give in single steps and in the column sweeps, and
a dL/dlam that is not finite reaches the rate adjoint of a cell without a burning neighbour (its product with 0 is NaN)."""
import numpy as np
import pytest
import torch

from paper_2512_06102_gb300 import scenarios
from tests.gpu_util import make_sim, require_gpu, to

pytestmark = pytest.mark.gpu


def same(x, y):
    torch.testing.assert_close(x, y, rtol=0, atol=0, equal_nan=True)


def _case(H, W):
    scn = scenarios.make_scenario(np.array(H, np.int32), np.array(W, np.int32), seed=9)
    sim = make_sim(scn, keep_rates=True)
    sim.precompute_probs(to(scn.cls), to(scn.dem), to(scn.wind_speed), to(scn.wind_dir))
    n = scn.F0.size
    rng = np.random.default_rng(3)
    pb = np.where(scn.F0 == 2, 1.0, (rng.random(n) < 0.01) * rng.random(n)).astype(np.float32)
    return scn, sim, n, rng, pb, (1 - pb).astype(np.float32)


@pytest.mark.parametrize("H,W,masked", [([33], [31], False), ([128] * 3, [128] * 3, False), ([37, 90], [61, 117], True)])
@pytest.mark.parametrize("wild", ["p_un", "rates"])
def test_on_chip_equals_sweeps_beyond_finite_values(H, W, masked, wild):
    require_gpu()
    T = 4
    scn, sim, n, rng, pb, pu = _case(H, W)
    q, r = (x.clone() for x in sim.probs())
    at = torch.from_numpy(rng.choice(n, 12, replace=False)).cuda()
    values = torch.tensor([float("inf"), float("nan"), -float("inf")], device="cuda").repeat(4)
    pu = to(pu)
    if wild == "p_un":
        pu[at] = values
    else:
        inside = r[at, 2] != 0                              # a rate whose source lies in the grid
        r[at[inside], 2] = values[inside]
        sim.set_probs(q, r)
    f = lambda *s: to(rng.random(s).astype(np.float32))
    masks = f(T, n) * (f(T, n) < 0.1) if masked else None
    PU, PB = torch.zeros((T + 1, n), device="cuda"), torch.zeros((T + 1, n), device="cuda")
    PU[0], PB[0] = pu, to(pb)
    assert sim.relaxed_on_chip(masked)
    sim.relaxed_fwd_steps(PU[0], PB[0], PU[1:], PB[1:], masks=masks)
    for t in range(T):
        u, b = sim.relaxed_fwd(PU[t].clone(), PB[t].clone(), None if masks is None else masks[t])
        same(PU[t + 1], u)
        same(PB[t + 1], b)
    # the adjoint along states with finite p_burn
    PB = torch.nan_to_num(PB, nan=0.25, posinf=0.5, neginf=0.0).contiguous()
    gu, gb = f(n) - 0.5, f(n) - 0.5
    out = []
    for on_chip in (False, True):
        au, ab = torch.empty_like(gu), torch.empty_like(gu)
        gr = torch.zeros((n, 8), device="cuda")
        scratch = torch.empty((2 * T, n), device="cuda")
        if on_chip:
            sim.relaxed_bwd_rates(PU[:T], PB[:T], gu, gb, au, ab, scratch, gr, masks=masks)
        else:
            sim.relaxed_bwd_steps(PU[:T], PB[:T], gu, gb, au, ab, masks=masks, glam=scratch[:T])
            sim.rates_accumulate(scratch[:T], PB[:T], gr, mask=masks)
        out.append((au, ab, gr))
    for x, y in zip(*out):
        same(y, x)
    sim.close()


@pytest.mark.parametrize("masked", [False, True])
def test_rate_adjoint_of_an_infinite_dlam(masked):
    require_gpu()
    T = 3
    scn, sim, n, rng, pb, _ = _case([40, 33], [70, 31])
    PB = torch.zeros((T, n), device="cuda")
    PB[:, to(pb) > 0] = 0.5
    glam = to(rng.standard_normal((T, n)).astype(np.float32))
    at = torch.from_numpy(rng.choice(n, 9, replace=False)).cuda()
    mask = torch.zeros((T, n), device="cuda") if masked else None
    want, got = torch.zeros((n, 8), device="cuda"), torch.zeros((n, 8), device="cuda")
    sim.rates_accumulate(glam, PB, want, mask=mask)
    glam[1, at] = torch.tensor([float("inf"), float("nan"), -float("inf")], device="cuda").repeat(3)
    sim.rates_accumulate(glam, PB, got, mask=mask)
    quiet = torch.ones(n, dtype=torch.bool, device="cuda")
    quiet[at] = False
    same(got[quiet], want[quiet])
    # inf x 0 and NaN x anything are NaN, inf x 0.5 is inf
    assert not bool(torch.isfinite(got[at]).any()) and bool(torch.isnan(got[at]).any())
    sim.close()
