"""tell where its kernel's tiles and splits are not full: columns around 256 (64 quads), pairs around the 32 of a split, populations
ranked inside the gradient kernel and by a kernel of their own (more than 2,048 members, or many columns), ties across the
128 entries that a warp compares at a time.  Ranks exact; centre, moments and gradient to 1e-5 of their RMS, as
everywhere (fp64 sums)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import rel_err
from paper_2202_05008_b200 import Solver, workloads as W

pytestmark = pytest.mark.gpu
F32 = lambda x: float(np.float32(x))


@pytest.mark.parametrize("P,D", [(2, 1), (64, 255), (66, 256), (62, 257), (130, 1025), (2046, 300), (2048, 33), (2050, 33), (4098, 70),
                                 (8200, 40), (16386, 9), (1024, 70000)])
@pytest.mark.parametrize("noise_mode", [W.NOISE_STORED, W.NOISE_REGENERATED])
@pytest.mark.parametrize("clipup", [False, True])
def test_tell_shapes(P, D, noise_mode, clipup):
    w = W.Workload("tell", P, D, seed=P + D, sigma=0.1, optimizer=W.OPT_CLIPUP if clipup else W.OPT_ADAM)
    s = Solver(w, noise_mode=noise_mode)
    rng = np.random.default_rng(P)
    for gen in range(2):
        c0 = s.center().cpu().numpy()
        m0, v0 = (x.cpu().numpy().astype(np.float64) for x in s.moments())
        s.ask()
        f = np.round(rng.standard_normal(P) * 20).astype(np.float32)          # plenty of ties
        f[rng.integers(0, P, 3)] = [np.inf, -np.inf, -0.0]
        s.tell(torch.tensor(f, device="cuda"))
        assert s.sync_status() == 0
        rank, u = (x.cpu().numpy() for x in s.ranks())
        rank_o, u_o, _ = oracle.centered_rank(f)
        assert (rank == rank_o).all() and (u == u_o).all()
        _, eps_o = oracle.ask(w.seed, gen, P, D, c0, w.sigma)
        g_o = oracle.gradient(u_o, eps_o, F32(w.sigma))
        assert rel_err(s.gradient().cpu().numpy(), g_o) < 1e-5
        if not clipup:
            c_o, m_o, v_o = oracle.adam(c0.astype(np.float64), m0, v0, g_o, gen + 1, F32(w.lr), F32(0.9), F32(0.999), F32(1e-8))
            keep = np.abs(g_o) >= 1e-6 * np.sqrt(np.mean(g_o ** 2))
            assert rel_err(s.center().cpu().numpy()[keep], c_o[keep]) < 1e-5
            assert rel_err(s.moments()[0].cpu().numpy(), m_o) < 1e-5 and rel_err(s.moments()[1].cpu().numpy(), v_o) < 1e-5
        else:
            vel = 0.9 * m0 + F32(w.lr) * g_o / np.sqrt(np.sum(g_o ** 2))
            n, most = np.sqrt(np.sum(vel ** 2)), 2 * F32(w.lr)
            vel = vel * (most / n if n > most else 1.0)
            assert rel_err(s.moments()[0].cpu().numpy(), vel) < 1e-5
            assert rel_err(s.center().cpu().numpy(), c0 + vel) < 1e-5
    assert s.counters() == (2, 2)
    s.close()


@pytest.mark.parametrize("P,D", [(64, 257), (1024, 600), (4098, 70), (1024, 70000)])      # ranks inside and outside, one and several splits
@pytest.mark.parametrize("noise_mode", [W.NOISE_STORED, W.NOISE_REGENERATED])
@pytest.mark.parametrize("clipup,adapt", [(False, False), (True, False), (False, True), (True, True)])
def test_a_nan_between_two_good_tells_changes_nothing(P, D, noise_mode, clipup, adapt):
    """Centre, moments and sigma keep their bits over a tell with a NaN fitness, which is reported; the next good tell is that of a
    solver which never saw one (same state, same generation)."""
    w = W.Workload("nan", P, D, seed=P, sigma=0.1, optimizer=W.OPT_CLIPUP if clipup else W.OPT_ADAM,
                   sigma_mode=W.SIGMA_PGPE if adapt else W.SIGMA_CONSTANT)
    rng = np.random.default_rng(D)
    good = [torch.tensor(rng.standard_normal(P).astype(np.float32), device="cuda") for _ in range(2)]
    state = lambda s: [x.clone() for x in (s.center(), *s.moments(), s.sigma())]
    s = Solver(w, noise_mode=noise_mode)
    s.ask(); s.tell(good[0])
    before = state(s)
    bad = good[1].clone()
    bad[int(rng.integers(P))] = float("nan")
    s.ask(); s.tell(bad)
    for a, b in zip(before, state(s)):
        assert torch.equal(a, b)
    assert s.sync_status() == 5 and s.sync_status() == 0                       # EVO_ERR_NONFINITE, then cleared
    assert s.counters() == (2, 1)
    s.ask(); s.tell(good[1])
    assert s.sync_status() == 0
    t = Solver(w, noise_mode=noise_mode)
    t.set_state(center=before[0], m=before[1], v=before[2], generation=2, adam_step=1)
    t.set_sigma(before[3])
    t.ask(); t.tell(good[1])
    for a, b in zip(state(s), state(t)):
        assert torch.equal(a, b)
    assert not torch.equal(before[0], s.center()) and s.counters() == t.counters() == (3, 2)
    s.close(); t.close()


@pytest.mark.parametrize("P,D,launches", [(16, 385, 1), (64, 5994, 1), (200, 6000, 1), (300, 6000, 2), (2048, 8000, 2), (2048, 600, 2)])
def test_a_tell_ranks_inside_the_gradient_kernel_only_while_that_is_cheaper(P, D, launches):
    s = Solver(W.Workload("tell", P, D, seed=1, sigma=0.1))
    s.ask()
    before = s.launch_count()
    s.tell(torch.randn(P, device="cuda"))
    assert s.launch_count() - before == launches and s.sync_status() == 0
    s.close()


@pytest.mark.parametrize("D,launches", [(12288, 1), (12320, 2)])
def test_clipup_moves_many_columns_in_a_kernel_of_its_own(D, launches):
    s = Solver(W.Workload("tell", 8, D, seed=1, sigma=0.1, optimizer=W.OPT_CLIPUP))
    s.ask()
    before = s.launch_count()
    s.tell(torch.randn(8, device="cuda"))
    assert s.launch_count() - before == launches and s.sync_status() == 0
    s.close()


@pytest.mark.parametrize("P,D", [(300, 40256), (202, 60001), (1000, 20000)])
@pytest.mark.parametrize("noise_mode", [W.NOISE_STORED, W.NOISE_REGENERATED])
def test_tells_of_fewer_splits_than_there_is_room_for(P, D, noise_mode):
    """Column blocks times splits just above a wave or two of blocks: the launch takes fewer, longer splits."""
    test_tell_shapes(P, D, noise_mode, clipup=False)
