"""The tensor-core control roll-outs lose nothing against fp32 arithmetic: their states are no further from the fp64 oracle's
than those of the fp32 runtime-shape kernel are, from the first step on and after errors have fed back over many.

The measure is the geometric mean over the members of a member's RMS error (relative to the RMS of each state component), which
a few chaotic members cannot move.  Both kernels' roundings are independent, so with 64 members the ratio of two
equally accurate kernels scatters by a few per cent; 1.2 leaves room for that and none for a lost bit."""
import numpy as np
import pytest
import torch

from helpers import oracle_fitness
from paper_2202_05008_b200 import Solver, workloads as W
from paper_2202_05008_b200.binding import ROLLOUT_AUTO, ROLLOUT_GENERIC

pytestmark = pytest.mark.gpu

STEPS = (1, 2, 5, 20, 60)


def _traces(w, theta, T, kernel):
    s = Solver(w, trace_steps=T, rollout_kernel=kernel)
    rows = s.padded_rows(w.pop_size)
    rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    trace = torch.zeros(w.pop_size, w.episodes, T, 4 if w.layer_sizes[0] == 5 else 28, device="cuda")
    s.rollout(rows, trace=trace)
    assert s.sync_status() == 0
    s.close()
    return trace.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("sizes,pop,episodes", [
    ((28, 128, 128, 8), 64, 4), ((28, 128, 128, 8), 300, 4), ((28, 64, 64, 8), 64, 8), ((28, 64, 64, 64, 8), 64, 4),
    ((28, 20, 8), 64, 8), ((5, 16, 16, 1), 64, 4), ((5, 64, 64, 1), 64, 8), ((5, 128, 90, 1), 300, 4), ((5, 40, 40, 40, 1), 64, 8)])
def test_states_are_as_close_to_the_oracle_as_those_of_the_fp32_kernel(sizes, pop, episodes):
    base, T = (W.CFG2, max(STEPS)) if sizes[0] == 5 else (W.CFG4, max(STEPS))
    # (the oracle computes with the task constants as fp32 numbers, which the kernels get)
    w = base.with_(pop_size=pop, episodes=episodes, horizon=T, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes),
                   task_param=tuple(float(np.float32(x)) for x in base.task_param))
    rng = np.random.default_rng(sum(sizes) + pop)
    noise = rng.standard_normal((pop // 2, w.param_dim)) * 0.1                 # a population in mid-training
    centre = rng.standard_normal(w.param_dim) * 0.05
    theta = np.empty((pop, w.param_dim), np.float32)
    theta[0::2], theta[1::2] = centre + noise, centre - noise
    members = list(range(32)) + list(range(pop - 32, pop))
    want = np.array(oracle_fitness(w, theta[members], 0, T, want_trace=True)[1])
    rms = np.sqrt((want ** 2).mean(axis=(0, 1, 2)))
    at = [t - 1 for t in STEPS]
    err = {}
    for kernel in (ROLLOUT_AUTO, ROLLOUT_GENERIC):
        e = (_traces(w, theta, T, kernel)[members][:, :, at] - want[:, :, at]) / rms
        err[kernel] = np.exp(np.log(np.sqrt((e ** 2).mean(axis=(1, 3)))).mean(axis=0))       # one per step
    assert (err[ROLLOUT_AUTO] < 1.2 * err[ROLLOUT_GENERIC]).all(), (err[ROLLOUT_AUTO] / err[ROLLOUT_GENERIC]).round(2)
