"""A caller's own parameter matrix: evo_rollout asks for its pitch and alignment only, so whatever lies in the padding columns
behind the parameters must not reach a result."""
import pytest
import torch

from paper_2202_05008_b200 import Solver, workloads as W
from paper_2202_05008_b200.binding import ROLLOUT_AUTO, ROLLOUT_GENERIC, ROLLOUT_TILED

pytestmark = pytest.mark.gpu


def _fitness(s, w, theta, fill):
    rows = torch.full((w.pop_size, s.ldD), fill, device="cuda")
    rows[:, :w.param_dim] = theta
    fit = s.rollout(rows).clone()
    assert s.sync_status() == 0
    return fit


@pytest.mark.parametrize("sizes,pop,episodes,kernel", [
    ((5, 16, 16, 1), 16, 5, ROLLOUT_AUTO), ((5, 64, 64, 1), 8, 9, ROLLOUT_AUTO), ((28, 64, 64, 8), 8, 4, ROLLOUT_AUTO),
    ((28, 128, 128, 8), 300, 4, ROLLOUT_AUTO), ((5, 127, 90, 1), 300, 4, ROLLOUT_AUTO), ((28, 33, 33, 33, 8), 8, 4, ROLLOUT_AUTO),
    ((5, 11, 1), 8, 4, ROLLOUT_AUTO), ((5, 64, 64, 1), 8, 9, ROLLOUT_TILED), ((28, 128, 128, 8), 8, 4, ROLLOUT_TILED),
    ((5, 64, 64, 1), 8, 9, ROLLOUT_GENERIC)])
def test_control_rollouts_ignore_the_padding_columns(sizes, pop, episodes, kernel):
    base = W.CFG2 if sizes[0] == 5 else W.CFG4
    w = base.with_(pop_size=pop, episodes=episodes, horizon=30, layer_sizes=sizes, param_dim=W.mlp_param_count(sizes))
    s = Solver(w, rollout_kernel=kernel)
    assert s.ldD > w.param_dim
    theta = torch.tensor(W.random_parameters(3, pop, w.param_dim, scale=0.1), device="cuda")
    want = _fitness(s, w, theta, 0.0)
    for fill in (1.0e20, float("inf"), float("nan")):
        assert torch.equal(_fitness(s, w, theta, fill), want), fill
    s.close()
