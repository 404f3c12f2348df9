"""GraphTankerRollout runs all its steps in one call only where the env's step and its simulator's are the package's own: a
step replaced on the env object, on its class or in a subclass, and a simulator with its own agent step, are called for every
step (CPU: a simulator that only counts)."""
import types

import pytest
import torch

from paper_2512_06102_gb300 import jwf, tanker


class CountingSim:
    N = 3

    def __init__(self):
        self.calls = []

    def agent_step(self, actions, agent, water0, random_fire, burn_penalty, reward, done, obs_k, obs):
        self.calls.append(actions.clone())
        reward.fill_(len(self.calls))
        done.fill_(len(self.calls) % 2)


class OneCallSim(CountingSim):
    # the package's agent step, and all of them in one call
    agent_step = jwf.Sim.agent_step

    def agent_rollout(self, *args):
        self.calls.append("all")


def _env(sim, cls=tanker.TankerEnv):
    return cls(sim, torch.zeros(12, dtype=torch.uint8))


def _steps(env, T=4):
    actions = torch.arange(T * 3, dtype=torch.int32).reshape(T, 3)
    roll = tanker.GraphTankerRollout(env, actions, capture=False)
    roll.run()
    return actions, roll


def _check(sim, actions, roll):
    assert len(sim.calls) == len(actions) and all(torch.equal(x, y) for x, y in zip(sim.calls, actions))
    assert roll.rewards[:, 0].tolist() == [1, 2, 3, 4] and roll.dones[:, 0].tolist() == [1, 0, 1, 0]


def test_a_simulator_with_its_own_step_is_called_step_by_step():
    sim = CountingSim()
    _check(sim, *_steps(_env(sim)))


@pytest.mark.parametrize("where", ["object", "class", "subclass"])
def test_a_replaced_step_is_called_step_by_step(where, monkeypatch):
    sim = OneCallSim()

    def step(self, actions):
        CountingSim.agent_step(self.sim, actions, None, 0, 0, 0, self.reward, self.done, 0, None)
        return self.obs, self.reward, self.done

    if where == "subclass":
        env = _env(sim, type("Env", (tanker.TankerEnv,), {"step": step}))
    else:
        env = _env(sim)
        if where == "object":
            env.step = types.MethodType(step, env)
        else:
            monkeypatch.setattr(tanker.TankerEnv, "step", step)
    _check(sim, *_steps(env))


def test_the_packages_own_steps_are_one_call():
    sim = OneCallSim()
    _steps(_env(sim))
    assert sim.calls == ["all"]
