"""The backward passes where device memory holds the column sweeps' scratch but not the on-chip adjoint's, and where the
library finds the sweeps faster: the sweeps run, over the same blocks of steps and with their scratch (CPU: a simulator that
records its calls, an allocator that refuses the larger tensor)."""
import types

import pytest
import torch

from paper_2512_06102_gb300 import relaxed

CELLS = 6


class RecordingSim:
    cells, grad_size, n_classes, tables_version = CELLS, 7, 1, 0

    def __init__(self, faster=True):
        self.calls, self.faster, self.asked = [], faster, []

    def relaxed_on_chip(self, with_masks=False):
        return True

    def relaxed_on_chip_faster(self, with_masks=False, sparse=False):
        self.asked.append((with_masks, sparse))
        return self.faster

    def relaxed_bwd_rates(self, su, sb, gu, gb, ngu, ngb, scratch, gr, masks=None, gpc=None):
        self.calls.append(("on chip", su.shape[0], scratch.shape[0]))

    def relaxed_bwd_steps(self, su, sb, gu, gb, ngu, ngb, masks=None, glam=None, gpc=None):
        self.calls.append(("sweeps", su.shape[0], glam.shape[0]))

    def rates_accumulate(self, glam, sb, gr, mask=None):
        self.calls.append(("rates", sb.shape[0], glam.shape[0]))

    def rates_contract(self, *args):
        pass

    def state_planes(self, states, pu, pb):
        pass


def _backward(kind, sim, T):
    g = torch.zeros(CELLS)
    ctx = types.SimpleNamespace(sim=sim, T=T, seg=T, masks=None, scene=(None,) * 4, tables_version=0, keep_all=True,
                                ckpts=[(torch.zeros(T + 1, CELLS), torch.zeros(T + 1, CELLS))], theta_device="cpu",
                                F0=torch.zeros(CELLS, dtype=torch.uint8), hist=torch.zeros(T, CELLS, dtype=torch.uint8))
    return kind.backward(ctx, g, g)


@pytest.mark.parametrize("kind", [relaxed.RelaxedRollout, relaxed.StraightThroughRollout])
def test_sweeps_where_the_larger_scratch_does_not_fit(kind, monkeypatch):
    T, empty = 20, torch.empty

    def tight(*shape, **kw):
        if shape[0] == (2 * relaxed.CHUNK, CELLS):
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(*shape, **kw)

    sim = RecordingSim()
    _backward(kind, sim, T)
    assert sim.calls == [("on chip", 4, 8), ("on chip", 16, 32)]
    monkeypatch.setattr(torch, "empty", tight)
    sim = RecordingSim()
    _backward(kind, sim, T)
    assert sim.calls == [("sweeps", 4, 4), ("rates", 4, 4), ("sweeps", 16, 16), ("rates", 16, 16)]


@pytest.mark.parametrize("kind", [relaxed.RelaxedRollout, relaxed.StraightThroughRollout])
def test_sweeps_where_they_are_faster(kind):
    sim = RecordingSim(faster=False)
    _backward(kind, sim, 20)
    assert sim.calls == [("sweeps", 4, 4), ("rates", 4, 4), ("sweeps", 16, 16), ("rates", 16, 16)]
    assert sim.asked == [(False, kind is relaxed.StraightThroughRollout)]
