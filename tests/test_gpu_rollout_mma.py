"""Control roll-outs on warp-level tensor-core products against the oracle, at the shapes where the tiling can go
wrong: widths at and around multiples of 16, one layer to five, layers of fewer and of more units than a
block has warps for, episode counts around the 4 and 8 that a block takes."""
import numpy as np
import pytest
import torch

from helpers import rel_err, oracle_fitness, cartpole_features
from paper_2202_05008_b200 import Solver, workloads as W

pytestmark = pytest.mark.gpu

# the bounds of the control roll-outs: state 1e-4 of a component's RMS, fitness 1e-3
STATE_TOL, FIT_TOL = 1e-4, 1e-3


def check(sizes, episodes, T, pop=4, scale=0.25, theta=None, generation=0):
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=pop, episodes=episodes, horizon=T, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    s = Solver(w, trace_steps=T)
    if theta is None:
        theta = W.random_parameters(sum(sizes), pop, w.param_dim, scale=scale)
    if generation:
        s.set_state(generation=generation)
    arg = s.padded_rows(pop)
    arg[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    trace = torch.zeros(pop, episodes, T, 4 if sizes[0] == 5 else 28, device="cuda")
    fit = s.rollout(arg, trace=trace)
    again = s.rollout(arg).clone()
    assert s.sync_status() == 0
    assert torch.equal(fit, again)
    fit_o, traces_o = oracle_fitness(w, theta, generation, T, want_trace=True)
    assert rel_err(fit.cpu().numpy(), fit_o, floor=1.0) < FIT_TOL
    for m in range(pop):
        got, want = trace[m].cpu().numpy().astype(np.float64), traces_o[m]
        if sizes[0] == 5:
            got, want = cartpole_features(got), cartpole_features(want)
        for i in range(got.shape[-1]):
            assert rel_err(got[..., i], want[..., i]) < STATE_TOL, (m, i)
    s.close()


@pytest.mark.parametrize("sizes", [(28, 8), (28, 17, 8), (28, 16, 15, 8), (28, 64, 64, 64, 8), (28, 130, 5, 33, 16, 8),
                                   (28, 200, 8), (28, 129, 129, 8)])
@pytest.mark.parametrize("episodes", [1, 4, 5, 9])
def test_tanh_linear_shapes(sizes, episodes):
    check(sizes, episodes, 40, scale=0.05)


@pytest.mark.parametrize("sizes", [(5, 1), (5, 33, 1), (5, 16, 16, 16, 1), (5, 200, 12, 1), (5, 129, 7, 3, 31, 1)])
@pytest.mark.parametrize("episodes", [1, 4, 5, 17])
def test_cartpole_shapes(sizes, episodes):
    check(sizes, episodes, 60)


def test_a_nan_parameter_reaches_the_fitness():
    sizes = (28, 24, 24, 24, 8)
    w = W.CFG4.with_(pop_size=4, episodes=4, horizon=5, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    s = Solver(w)
    arg = s.padded_rows(4)
    arg[1, 3] = float("nan")                               # a first-layer weight
    arg[2, 24 * 28 + 24 + 24 * 24] = float("nan")          # a second-layer bias
    fit = s.rollout(arg)
    assert torch.isnan(fit).tolist() == [False, True, True, False] and s.sync_status() == 0
    s.close()


@pytest.mark.parametrize("sizes", [(28, 1, 1, 8), (28, 16, 17, 8), (28, 33, 48, 8), (28, 64, 65, 8), (28, 65, 3, 8), (28, 128, 127, 8),
                                   (5, 17, 16, 1), (5, 48, 49, 1), (5, 64, 64, 1), (5, 127, 65, 1), (5, 5, 128, 1)])
@pytest.mark.parametrize("episodes", [3, 8, 11])
def test_two_hidden_layers_with_the_weights_in_registers(sizes, episodes):
    check(sizes, episodes, 40, scale=0.05 if sizes[0] == 28 else 0.25)


@pytest.mark.parametrize("sizes", [(28, 128, 128, 8), (28, 90, 70, 8), (28, 20, 128, 8), (5, 128, 65, 1), (5, 81, 96, 1)])
@pytest.mark.parametrize("episodes", [4, 5])
def test_two_row_tiles_per_warp(sizes, episodes):
    """More than two blocks per SM: the wide policies run with the low parts of the second layer in shared memory."""
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=300, episodes=episodes, horizon=12, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes), sigma=0.05)
    s = Solver(w)
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    members = [0, 1, 147, 148, 298, 299]
    fit_o, _ = oracle_fitness(w, theta[members], 0, 12)
    assert rel_err(fit[members], fit_o, floor=1.0) < FIT_TOL
    s.close()


@pytest.mark.parametrize("sizes", [(28, 8), (28, 17, 8), (28, 130, 8), (28, 16, 15, 8), (28, 64, 64, 8), (28, 128, 127, 8), (28, 90, 33, 8), (28, 192, 140, 8),
                                   (28, 64, 17, 49, 8), (28, 128, 65, 16, 8), (28, 129, 144, 60, 8), (28, 64, 33, 64, 49, 8), (28, 20, 60, 9, 100, 8),
                                   (28, 250, 8), (5, 1), (5, 33, 1), (5, 128, 1), (5, 64, 64, 1), (5, 127, 65, 1), (5, 40, 110, 1), (5, 16, 16, 16, 1),
                                   (5, 65, 128, 3, 1), (5, 16, 17, 150, 1), (5, 16, 65, 64, 128, 1), (5, 200, 12, 1)])
@pytest.mark.parametrize("episodes", [5, 8, 11])
def test_eight_episodes_per_block(sizes, episodes):
    """What populations too large for blocks of four episodes take: states and fitness of a few of 150 members (300 and more blocks of four)."""
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    T, members = 20, [0, 1, 147, 149]
    w = base.with_(pop_size=150, episodes=episodes, horizon=T, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    theta = W.random_parameters(sum(sizes), 150, w.param_dim, scale=0.05 if sizes[0] == 28 else 0.25)
    s = Solver(w, trace_steps=T)
    arg = s.padded_rows(150)
    arg[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    trace = torch.zeros(150, episodes, T, 4 if sizes[0] == 5 else 28, device="cuda")
    fit = s.rollout(arg, trace=trace).cpu().numpy()
    assert s.sync_status() == 0
    fit_o, traces_o = oracle_fitness(w, theta[members], 0, T, want_trace=True)
    assert rel_err(fit[members], fit_o, floor=1.0) < FIT_TOL
    for m, want in zip(members, traces_o):
        got = trace[m].cpu().numpy().astype(np.float64)
        if sizes[0] == 5:
            got, want = cartpole_features(got), cartpole_features(want)
        for i in range(got.shape[-1]):
            assert rel_err(got[..., i], want[..., i]) < STATE_TOL, (m, i)
    s.close()


@pytest.mark.parametrize("sizes,steps,launches", [((5, 64, 64, 1), 20, 1), ((5, 20, 30, 1), 79, 1), ((5, 20, 30, 1), 80, 2), ((28, 20, 8), 49, 1),
                                                  ((28, 64, 64, 64, 8), 20, 2), ((5, 16, 16, 1), 20, 2)])
def test_short_roll_outs_of_eight_episodes_are_one_launch(sizes, steps, launches):
    """A block of eight episodes writes the fitness itself; the sums of blocks of four need a second launch.  (5-16-16-1 has a warp for four in any case.)"""
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=74, episodes=8, horizon=steps, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes), sigma=0.05)
    s = Solver(w)
    theta = s.ask().cpu().numpy()
    before = s.launch_count()
    fit = s.rollout().cpu().numpy()
    assert s.launch_count() - before == launches
    assert s.sync_status() == 0
    fit_o, _ = oracle_fitness(w, theta[[0, 73]], 0, steps)
    assert rel_err(fit[[0, 73]], fit_o, floor=1.0) < FIT_TOL
    s.close()


@pytest.mark.parametrize("sizes", [(28, 128, 64, 8), (28, 90, 33, 8), (28, 96, 5, 8), (28, 48, 81, 8), (28, 64, 113, 8), (28, 17, 65, 8),
                                   (5, 128, 50, 1), (5, 70, 48, 1), (5, 64, 128, 1), (5, 3, 90, 1)])
@pytest.mark.parametrize("episodes", [4, 5])
def test_two_row_tiles_per_warp_in_one_layer(sizes, episodes):
    """As above where the other layer has at most half as many tiles, one per warp."""
    test_two_row_tiles_per_warp(sizes, episodes)


@pytest.mark.parametrize("sizes,pop", [((28, 128, 128, 8), 4), ((28, 128, 128, 8), 300), ((5, 64, 64, 1), 4), ((5, 16, 16, 1), 4),
                                       ((28, 32, 32, 32, 8), 4)])
def test_weights_far_beyond_the_fp16_range(sizes, pop):
    """The unit with a weight of 1e7 keeps its other weights to 22 bits of that one, every other unit keeps its own as they are, so
    the fitness agrees with the oracle, which uses every weight as it is."""
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=pop, episodes=4, horizon=20, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    theta = W.random_parameters(5, pop, w.param_dim, scale=0.05)
    theta[0, 3] = 1.0e7
    theta[1, sizes[0] * sizes[1] + sizes[1] + 2] = -1.0e5
    s = Solver(w)
    arg = s.padded_rows(pop)
    arg[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    fit = s.rollout(arg).cpu().numpy()
    assert s.sync_status() == 0 and np.isfinite(fit).all()
    fit_o, _ = oracle_fitness(w, theta[:4], 0, 20)
    assert rel_err(fit[:4], fit_o, floor=1.0) < FIT_TOL
    s.close()


@pytest.mark.parametrize("sizes,episodes", [((28, 384, 96, 8), 4), ((5, 112, 384, 1), 8), ((5, 256, 192, 1), 4)])
def test_policies_that_just_fit_the_shared_memory(sizes, episodes):
    """221 to 222 KB of operand tiles, biases and exponents; with a larger one the runtime-shape kernel would run."""
    check(sizes, episodes, 12, scale=0.02 if sizes[0] == 28 else 0.1)


def test_eight_episodes_a_block_at_the_limit_of_the_shared_memory():
    """222 KB with the operands of eight episodes; 76 members, so that blocks of four would not find an SM each."""
    sizes = (5, 112, 384, 1)
    w = W.CFG2.with_(pop_size=76, episodes=8, horizon=24, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes), sigma=0.1)
    s = Solver(w)
    theta = s.ask().cpu().numpy()
    before = s.launch_count()
    fit = s.rollout().cpu().numpy()
    assert s.launch_count() - before == 1
    assert s.sync_status() == 0
    members = [0, 1, 74, 75]
    fit_o, _ = oracle_fitness(w, theta[members], 0, 24)
    assert rel_err(fit[members], fit_o, floor=1.0) < FIT_TOL
    s.close()


@pytest.mark.parametrize("sizes", [(28, 128, 8), (28, 3, 8), (28, 64, 17, 49, 8), (28, 128, 128, 128, 8), (28, 65, 16, 100, 8), (28, 5, 128, 64, 8),
                                   (28, 64, 33, 64, 49, 8), (28, 128, 64, 65, 128, 8),
                                   (5, 128, 1), (5, 64, 64, 64, 1), (5, 65, 128, 3, 1), (5, 50, 64, 49, 64, 1), (5, 16, 65, 64, 128, 1)])
@pytest.mark.parametrize("episodes", [3, 8, 11])
def test_one_three_and_four_hidden_layers_with_the_weights_in_registers(sizes, episodes):
    check(sizes, episodes, 40, scale=0.05 if sizes[0] == 28 else 0.25)


@pytest.mark.parametrize("sizes", [(28, 129, 8), (28, 192, 8), (28, 192, 192, 8), (28, 192, 176, 180, 8), (28, 144, 145, 129, 8), (28, 20, 190, 5, 8),
                                   (28, 129, 64, 65, 130, 8), (28, 192, 100, 64, 192, 8), (5, 130, 1), (5, 190, 180, 1), (5, 16, 17, 192, 1),
                                   (5, 192, 192, 192, 1), (5, 160, 48, 49, 160, 1), (5, 3, 176, 128, 64, 1)])
@pytest.mark.parametrize("episodes", [3, 11])
def test_up_to_192_units_with_the_weights_in_registers(sizes, episodes):
    check(sizes, episodes, 30, scale=0.04 if sizes[0] == 28 else 0.2)


@pytest.mark.parametrize("sizes", [(28, 128, 8), (28, 64, 64, 64, 8), (28, 128, 100, 128, 8), (28, 64, 40, 64, 30, 8), (28, 128, 128, 128, 128, 8),
                                   (5, 60, 1), (5, 64, 64, 64, 1), (5, 128, 30, 100, 64, 1)])
@pytest.mark.parametrize("episodes", [4, 5])
def test_weights_far_beyond_the_fp16_range_in_every_layer(sizes, episodes):
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=len(sizes) // 2 * 2, episodes=episodes, horizon=20, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    theta = W.random_parameters(7, w.pop_size, w.param_dim, scale=0.05)
    at = 0
    for m, (a, b) in enumerate(zip(sizes[:-1], sizes[1:])):      # member m: the last unit of layer m has one
        theta[m % w.pop_size, at + a * b - 1] = 1.0e6
        at += (a + 1) * b
    s = Solver(w)
    arg = s.padded_rows(w.pop_size)
    arg[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    fit = s.rollout(arg).cpu().numpy()
    assert s.sync_status() == 0 and np.isfinite(fit).all()
    fit_o, _ = oracle_fitness(w, theta, 0, 20)
    assert rel_err(fit, fit_o, floor=1.0) < FIT_TOL
    s.close()


@pytest.mark.parametrize("sizes,pop,episodes", [((28, 120, 20, 10, 8), 300, 4), ((28, 100, 30, 100, 8), 300, 8), ((5, 90, 20, 20, 20, 1), 150, 16)])
def test_deep_wide_policies_of_more_blocks_than_the_gpu_holds(sizes, pop, episodes):
    """Either side of the line between weights in registers and in shared memory."""
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=pop, episodes=episodes, horizon=12, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes), sigma=0.05)
    s = Solver(w)
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    members = [0, 1, 147, 148, pop - 1]
    fit_o, _ = oracle_fitness(w, theta[members], 0, 12)
    assert rel_err(fit[members], fit_o, floor=1.0) < FIT_TOL
    s.close()
