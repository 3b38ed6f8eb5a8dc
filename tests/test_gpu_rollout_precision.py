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


def _workload(sizes, pop, episodes):
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    # (the oracle computes with the task constants as fp32 numbers, which the kernels get)
    return base.with_(pop_size=pop, episodes=episodes, horizon=max(STEPS), layer_sizes=sizes, param_dim=W.mlp_param_count(sizes),
                      task_param=tuple(float(np.float32(x)) for x in base.task_param))


def _population(w, seed):
    """A population in mid-training."""
    rng = np.random.default_rng(seed)
    noise = rng.standard_normal((w.pop_size // 2, w.param_dim)) * 0.1
    centre = rng.standard_normal(w.param_dim) * 0.05
    theta = np.empty((w.pop_size, w.param_dim), np.float32)
    theta[0::2], theta[1::2] = centre + noise, centre - noise
    return theta


def _check_against_fp32(w, theta):
    members = list(range(32)) + list(range(w.pop_size - 32, w.pop_size))
    want = np.array(oracle_fitness(w, theta[members], 0, w.horizon, want_trace=True)[1])
    rms = np.sqrt((want ** 2).mean(axis=(0, 1, 2)))
    at = [t - 1 for t in STEPS]
    err = {}
    for kernel in (ROLLOUT_AUTO, ROLLOUT_GENERIC):
        e = (_traces(w, theta, w.horizon, kernel)[members][:, :, at] - want[:, :, at]) / rms
        err[kernel] = np.exp(np.log(np.sqrt((e ** 2).mean(axis=(1, 3))) + 1e-30).mean(axis=0))       # one per step
    ratio = err[ROLLOUT_AUTO] / err[ROLLOUT_GENERIC]
    assert (ratio < 1.2).all(), ratio.round(2)


@pytest.mark.parametrize("sizes,pop,episodes", [
    ((28, 128, 128, 8), 64, 4), ((28, 128, 128, 8), 300, 4), ((28, 64, 64, 8), 64, 8), ((28, 64, 64, 64, 8), 64, 4),
    ((28, 20, 8), 64, 8), ((5, 16, 16, 1), 64, 4), ((5, 64, 64, 1), 64, 8), ((5, 128, 90, 1), 300, 4), ((5, 40, 40, 40, 1), 64, 8),
    # one, three and four hidden layers with the weights in registers, wide ones and such that take the other tanh
    ((28, 128, 8), 64, 4), ((28, 49, 8), 64, 4), ((28, 128, 128, 128, 8), 64, 4), ((28, 100, 90, 80, 8), 64, 8), ((28, 70, 20, 100, 8), 64, 4),
    ((28, 52, 56, 60, 8), 64, 8), ((28, 64, 64, 64, 64, 8), 64, 4), ((28, 128, 128, 128, 128, 8), 64, 8), ((28, 100, 66, 70, 90, 8), 64, 4),
    ((5, 100, 1), 64, 8), ((5, 128, 128, 128, 1), 64, 8), ((5, 64, 64, 64, 64, 1), 64, 8), ((5, 128, 128, 128, 128, 1), 64, 4), ((5, 128, 20, 20, 1), 64, 4)])
def test_states_are_as_close_to_the_oracle_as_those_of_the_fp32_kernel(sizes, pop, episodes):
    w = _workload(sizes, pop, episodes)
    _check_against_fp32(w, _population(w, sum(sizes) + pop))


@pytest.mark.parametrize("sizes", [(28, 64, 64, 8), (28, 20, 8), (28, 100, 90, 80, 8), (28, 52, 56, 60, 8), (28, 128, 128, 128, 128, 8), (28, 128, 90, 8),
                                   (5, 64, 64, 1), (5, 100, 1), (5, 40, 40, 40, 1), (5, 64, 64, 64, 64, 1)])
def test_the_same_of_eight_episodes_per_block(sizes):
    w = _workload(sizes, 150, 8)                                  # (64 members have blocks of four)
    _check_against_fp32(w, _population(w, sum(sizes)))


@pytest.mark.parametrize("sizes,episodes", [((28, 160, 8), 4), ((28, 192, 140, 8), 8), ((28, 150, 130, 190, 8), 4), ((28, 129, 60, 80, 180, 8), 8),
                                            ((5, 192, 1), 4), ((5, 140, 150, 160, 1), 8)])
def test_the_same_of_more_than_128_units(sizes, episodes):
    w = _workload(sizes, 64, episodes)
    _check_against_fp32(w, _population(w, sum(sizes)))


@pytest.mark.parametrize("sizes,pop,episodes", [((28, 180, 180, 180, 8), 8, 4), ((28, 150, 130, 190, 8), 4, 8), ((28, 150, 130, 190, 8), 160, 8),
                                                ((28, 128, 163, 128, 143, 8), 4, 4), ((5, 192, 192, 192, 1), 4, 3), ((5, 133, 120, 117, 132, 1), 160, 8)])
def test_above_128_units_policies_that_do_not_fit_the_shared_memory_keep_fp32_arithmetic(sizes, pop, episodes):
    """Split products would be the faster ones, but the fitness is then further from the oracle's (1.1 to 1.5 times in the mean)."""
    w = _workload(sizes, pop, episodes).with_(horizon=20)
    theta, fit = _population(w, 3), []
    for kernel in (ROLLOUT_AUTO, ROLLOUT_GENERIC):
        s = Solver(w, rollout_kernel=kernel)
        rows = s.padded_rows(pop)
        rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
        fit.append(s.rollout(rows).cpu().numpy())
        assert s.sync_status() == 0
        s.close()
    assert np.array_equal(fit[0], fit[1])


@pytest.mark.parametrize("sizes,pop,episodes", [
    ((28, 64, 64, 8), 64, 4), ((28, 128, 128, 8), 300, 4), ((28, 64, 64, 64, 8), 64, 8), ((5, 16, 16, 1), 64, 4),
    ((5, 64, 64, 1), 64, 8), ((5, 128, 90, 1), 300, 4), ((5, 40, 40, 40, 1), 64, 4),
    ((28, 128, 8), 64, 8), ((28, 128, 128, 128, 8), 64, 4), ((28, 100, 128, 70, 128, 8), 64, 8), ((5, 128, 100, 128, 1), 64, 8)])
def test_a_huge_weight_takes_nothing_from_the_others(sizes, pop, episodes):
    """One weight or bias beyond the fp16 range per member, from 2e4 to 1e30, anywhere in the policy."""
    w = _workload(sizes, pop, episodes)
    theta = _population(w, 1 + sum(sizes))
    rng = np.random.default_rng(pop)
    for m in range(pop):
        theta[m, rng.integers(w.param_dim)] = rng.choice((-1.0, 1.0)) * rng.choice((2.0e4, 1.0e7, 1.0e12, 1.0e30))
    _check_against_fp32(w, theta)


def _launches(w):
    s = Solver(w)
    s.ask()
    before = s.launch_count()
    s.rollout()
    n = s.launch_count() - before
    s.close()
    return n


def _huge_weights(w, theta, seed):
    rng = np.random.default_rng(seed)
    for m in range(w.pop_size):
        theta[m, rng.integers(w.param_dim)] = rng.choice((-1.0, 1.0)) * rng.choice((2.0e4, 1.0e7, 1.0e12, 1.0e30))


@pytest.mark.parametrize("huge", [False, True])
@pytest.mark.parametrize("sizes,pop", [
    # weights in registers, in one row tile a warp and (300 members) two, in both layers or one
    ((28, 64, 64, 8), 150), ((28, 128, 128, 8), 150), ((5, 64, 64, 1), 150), ((28, 128, 128, 8), 300), ((5, 128, 90, 1), 300),
    ((28, 90, 40, 8), 300), ((28, 40, 90, 8), 300), ((5, 120, 60, 1), 300), ((5, 40, 110, 1), 300),
    # one, three and four hidden layers
    ((28, 128, 8), 76), ((28, 64, 64, 64, 8), 76), ((28, 100, 128, 70, 128, 8), 76), ((5, 128, 100, 128, 1), 76), ((5, 50, 64, 49, 64, 1), 76),
    # above 128 units
    ((28, 160, 8), 76), ((28, 192, 140, 8), 76), ((28, 150, 130, 100, 8), 76), ((28, 192, 100, 64, 192, 8), 76), ((28, 129, 64, 65, 130, 8), 76),
    ((5, 160, 1), 76), ((5, 190, 180, 1), 76), ((5, 140, 90, 120, 1), 76), ((5, 160, 48, 49, 160, 1), 76),
    # weights in shared memory
    ((28, 200, 8), 76), ((28, 32, 32, 32, 32, 32, 8), 76), ((5, 200, 12, 1), 76)])
def test_blocks_of_eight_episodes(sizes, pop, huge):
    """Every kernel with blocks of eight episodes, with weights in the fp16 range and beyond."""
    w = _workload(sizes, pop, 8)
    assert _launches(w) == 1                                      # (blocks of four, or the runtime-shape kernel, need a second one)
    theta = _population(w, 2 + sum(sizes))
    if huge:
        _huge_weights(w, theta, pop)
    _check_against_fp32(w, theta)


@pytest.mark.parametrize("huge", [False, True])
@pytest.mark.parametrize("sizes", [(28, 90, 40, 8), (28, 40, 90, 8), (28, 115, 51, 8), (5, 120, 60, 1), (5, 40, 110, 1)])
def test_two_row_tiles_a_warp_in_one_layer(sizes, huge):
    w = _workload(sizes, 300, 4)
    theta = _population(w, 3 + sum(sizes))
    if huge:
        _huge_weights(w, theta, 300)
    _check_against_fp32(w, theta)


@pytest.mark.parametrize("sizes", [(28, 160, 8), (28, 150, 130, 100, 8), (28, 192, 100, 64, 192, 8), (5, 160, 1), (5, 140, 90, 120, 1), (5, 160, 48, 49, 160, 1)])
def test_a_huge_weight_above_128_units(sizes):
    w = _workload(sizes, 64, 4)
    theta = _population(w, 4 + sum(sizes))
    _huge_weights(w, theta, 64)
    _check_against_fp32(w, theta)


@pytest.mark.parametrize("sizes", [(28, 24, 40, 8), (28, 24, 24, 24, 8), (5, 16, 16, 1), (5, 30, 40, 1), (5, 16, 16, 16, 1)])
def test_infinite_weights_saturate(sizes):
    w = _workload(sizes, 64, 4).with_(pop_size=8, horizon=3)
    theta = _population(w, 9)[:8]
    second = sizes[0] * sizes[1] + sizes[1]
    theta[0, 3], theta[1, second + 1], theta[2, second + sizes[1] * sizes[2]] = np.inf, -np.inf, np.inf      # both layers, a bias
    theta[3, second + 1], theta[3, second + 2] = np.inf, np.nan
    fit = {}
    for kernel in (ROLLOUT_AUTO, ROLLOUT_GENERIC):
        s = Solver(w, rollout_kernel=kernel)
        rows = s.padded_rows(8)
        rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
        fit[kernel] = s.rollout(rows).cpu().numpy()
        s.close()
    np.testing.assert_allclose(fit[ROLLOUT_AUTO], fit[ROLLOUT_GENERIC], rtol=1e-5)
    assert np.isnan(fit[ROLLOUT_AUTO]).tolist() == [False] * 3 + [True] + [False] * 4


@pytest.mark.parametrize("sizes,pop,episodes", [
    ((28, 150, 60, 8), 8, 4), ((28, 150, 60, 8), 8, 8), ((28, 129, 64, 65, 130, 8), 8, 4), ((28, 129, 64, 65, 130, 8), 8, 8), ((5, 160, 48, 49, 160, 1), 8, 4),
    ((5, 160, 48, 49, 160, 1), 8, 8), ((28, 90, 40, 8), 300, 4), ((5, 40, 110, 1), 300, 4), ((28, 90, 40, 8), 300, 8), ((28, 24, 40, 8), 8, 8), ((5, 16, 16, 16, 1), 8, 8)])
def test_infinite_weights_saturate_in_every_kernel(sizes, pop, episodes):
    """As above: above 128 units, with one row tile a warp in one layer and two in the other, with blocks of eight episodes."""
    w = _workload(sizes, pop, episodes).with_(horizon=3)
    theta = _population(w, 9)
    second = sizes[0] * sizes[1] + sizes[1]
    theta[0, 3], theta[1, second + 1], theta[2, second + sizes[1] * sizes[2]] = np.inf, -np.inf, np.inf
    theta[3, second + 1], theta[3, second + 2] = np.inf, np.nan
    fit = {}
    for kernel in (ROLLOUT_AUTO, ROLLOUT_GENERIC):
        s = Solver(w, rollout_kernel=kernel)
        rows = s.padded_rows(pop)
        rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
        fit[kernel] = s.rollout(rows).cpu().numpy()
        s.close()
    np.testing.assert_allclose(fit[ROLLOUT_AUTO], fit[ROLLOUT_GENERIC], rtol=1e-5)
    assert np.flatnonzero(np.isnan(fit[ROLLOUT_AUTO])).tolist() == [3]


@pytest.mark.parametrize("sizes,pop", [((28, 24, 40, 8), 64), ((28, 128, 100, 8), 300), ((28, 24, 24, 24, 8), 64)])
@pytest.mark.parametrize("scale", [-1.0e3, 3.0e3, 1.0e6, 1.0e15])
def test_large_action_scales(sizes, pop, scale):
    """Actions that saturate the dynamics: a state near a sign change is either sign's in any arithmetic, so most members agree with
    the oracle to fp32 rounding and every one is finite."""
    w = _workload(sizes, pop, 4).with_(horizon=8, action_scale=scale)
    theta = _population(w, 5)
    s = Solver(w)
    rows = s.padded_rows(pop)
    rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    fit = s.rollout(rows).cpu().numpy()
    assert s.sync_status() == 0 and np.isfinite(fit).all()
    want, _ = oracle_fitness(w, theta[:64], 0, 8)
    err = np.abs(fit[:64] - want) / np.abs(want)
    assert np.median(err) < 1e-5, np.sort(err)
    s.close()
