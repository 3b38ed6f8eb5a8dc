"""Parity of the seq2seq roll-out (paper Section 3, "Seq2Seq Learning") with the oracle, through the
C-ABI: the CUDA-core kernel (any hidden width, logits visible) and the tcgen05 kernel (h = 128)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2202_05008_b200 import Solver, workloads as W
from paper_2202_05008_b200.binding import ROLLOUT_AUTO, ROLLOUT_GENERIC, ROLLOUT_TILED

pytestmark = pytest.mark.gpu

# Both sides round the operands of the contractions to bf16 at the same points; what is left is
# fp32 accumulation order and the rare hidden-state element that rounds to the neighbouring bf16
# value (2^-9 relative) because the kernel's fp32 activation differs from the oracle's fp64 one in
# the last bits.  Averaged over the batch that stays well below 1e-3 on the fitness.
FIT_TOL = 1e-3


def _workload(h, nd, B, P, sigma=0.3, seed=11):
    return W.SEQ2SEQ.with_(pop_size=P, param_dim=W.seq2seq_param_count(h), layer_sizes=(h,), batch=B,
                           task_param=(float(nd),), sigma=sigma, seed=seed)


def _oracle_fits(w, theta, generation, want_logits=False):
    h, nd = w.layer_sizes[0], int(w.task_param[0])
    enc, dec, tgt = oracle.seq2seq_queries(w.seed, generation, w.batch, nd)
    return [oracle.seq2seq_fitness(row, h, nd, enc, dec, tgt, True, want_logits=want_logits) for row in theta]


@pytest.mark.parametrize("h,nd,B", [(32, 2, 20), (64, 1, 16), (128, 3, 9)])
def test_cuda_core_kernel_matches_oracle_with_logits(h, nd, B):
    w = _workload(h, nd, B, P=4)
    s = Solver(w, rollout_kernel=ROLLOUT_GENERIC, trace_steps=1)
    theta = s.ask().cpu().numpy()
    logits = torch.zeros(w.pop_size, B, nd + 1, 12, device="cuda")
    fit = s.rollout(trace=logits).cpu().numpy()
    want = _oracle_fits(w, theta, 0, want_logits=True)
    assert s.sync_status() == 0
    for m in range(w.pop_size):
        assert np.max(np.abs(logits[m].cpu().numpy() - want[m][2])) < 2e-2
        assert abs(fit[m] - want[m][0]) < FIT_TOL
    # the typical element agrees far better than the worst one
    assert np.median(np.abs(logits[0].cpu().numpy() - want[0][2])) < 1e-4


@pytest.mark.parametrize("B", [128, 100, 200])
def test_tensor_core_kernel_matches_oracle(B):
    w = _workload(128, 3, B, P=6, sigma=0.1)
    s = Solver(w, rollout_kernel=ROLLOUT_TILED)
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    want = _oracle_fits(w, theta, 0)
    for m in range(w.pop_size):
        assert abs(fit[m] - want[m][0]) < FIT_TOL, (m, fit[m], want[m][0])
    assert np.std(fit) > 1e-3                                    # members really differ


@pytest.mark.parametrize("P", [2, 148])                          # (two members: more items than 128 queries would ask for)
@pytest.mark.parametrize("B", [1, 8, 9, 16, 17, 65, 111, 113, 127, 129, 257])
def test_batches_that_do_not_fill_an_item(B, P):
    """Items of one half and of two, eights of queries that hold one or none, chunks of unequal size."""
    w = _workload(128, 1, B, P, sigma=0.1)
    s = Solver(w, rollout_kernel=ROLLOUT_TILED)
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    members = [0, P - 1]
    for m, want in zip(members, _oracle_fits(w, theta[members], 0)):
        assert abs(fit[m] - want[0]) < FIT_TOL, (m, fit[m], want[0])


@pytest.mark.parametrize("kernel", [ROLLOUT_AUTO, ROLLOUT_GENERIC])
@pytest.mark.parametrize("h,B", [(128, 9), (128, 40), (128, 100), (128, 128), (64, 40)])
def test_an_infinite_recurrent_weight_meets_the_zero_state(h, B, kernel):
    """Infinity times the start state is not a number, in the oracle and in every kernel, however many queries an item has."""
    w = _workload(h, 2, B, P=4, sigma=0.1)
    s = Solver(w, rollout_kernel=kernel)
    rows = s.ask().cpu().numpy()
    at = 4 * h * 12                                              # the encoder's recurrent weights
    rows[0, at], rows[1, at + 2 * h * h + 5], rows[3, at + 4 * h * h - 1] = np.inf, -np.inf, np.inf
    theta = s.padded_rows(4)
    theta[:, :w.param_dim] = torch.tensor(rows, device="cuda")
    fit = s.rollout(theta).cpu().numpy()
    assert s.sync_status() == 0
    want = np.array([f[0] for f in _oracle_fits(w, rows, 0)])
    assert np.isnan(want).tolist() == [True, True, False, True]
    assert np.isnan(fit).tolist() == np.isnan(want).tolist()
    assert abs(fit[2] - want[2]) < FIT_TOL


def _saturated_fitness(P, batch):
    """Gates and cells saturated by their biases: every hidden state is +-bf16(tanh 1) = +-195/256 exactly, whatever the query.  Only the
    logit of '=' (never an answer) has weights, all of its terms positive: the loss of every position is that logit (28 and
    more, so that the others add nothing to the exponentials), a sum of 128 products that fp32 holds exactly.  Fitness and products."""
    h = 128
    w = _workload(h, 1, batch, P=P)
    rng = np.random.default_rng(2)
    sign = rng.choice((-1.0, 1.0), (P, h)).astype(np.float32)
    weights = (np.exp2(rng.uniform(-10.0, 2.0, (P, h))).astype(np.float32).view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)
    theta = np.zeros((P, w.param_dim), np.float32)
    cell = 4 * h * 12 + 4 * h * h + 4 * h
    for at in (cell - 4 * h, 2 * cell - 4 * h):                  # the biases: input 1, forget 0, cell +-1, output 1
        theta[:, at:at + h], theta[:, at + h:at + 2 * h] = 64.0, -64.0
        theta[:, at + 2 * h:at + 3 * h], theta[:, at + 3 * h:at + 4 * h] = 64.0 * sign, 64.0
    theta[:, 2 * cell + 11 * h:2 * cell + 12 * h] = weights * sign
    s = Solver(w)
    rows = s.padded_rows(P)
    rows[:, :w.param_dim] = torch.tensor(theta, device="cuda")
    fit = s.rollout(rows).cpu().numpy()
    assert s.sync_status() == 0
    s.close()
    return fit, weights * np.float32(195.0 / 256.0)


def test_the_read_out_is_as_exact_as_a_chain_of_fp32_additions():
    """Its error may be no larger than that of two chains of 64 rounded additions (RMS; 1,024 members scatter by 2 %), and without their
    rounding's bias: a mean within 4 of its standard errors."""
    P = 1024
    fit, terms = _saturated_fitness(P, 1)
    chains = np.zeros((P, 2), np.float32)
    for k in range(0, 128, 2):
        chains = chains + terms[:, k:k + 2]
    exact = terms.astype(np.float64).sum(1)
    chain_err, err = (chains[:, 0] + chains[:, 1]) / exact - 1.0, -fit.astype(np.float64) / exact - 1.0
    rms = lambda x: float(np.sqrt((x * x).mean()))
    assert rms(err) <= 1.05 * rms(chain_err), (rms(err), rms(chain_err))
    assert abs(err.mean()) <= 4.0 * err.std() / math.sqrt(P), (err.mean(), err.std())


def test_chunks_of_128_queries_are_summed_in_order():
    """All chunks have the same sum, which the fitness of one chunk gives exactly (a division by 256)."""
    chunk = _saturated_fitness(256, 128)[0] * np.float32(-256.0)
    total = np.zeros(256, np.float32)
    for _ in range(5):
        total = total + chunk
    want = -total * (np.float32(1.0) / (np.float32(640.0) * np.float32(2.0)))
    assert np.array_equal(_saturated_fitness(256, 640)[0], want)


@pytest.mark.parametrize("kernel", [ROLLOUT_TILED, ROLLOUT_GENERIC])
def test_kernels_against_the_unrounded_oracle(kernel):
    """Against the fp64 oracle with NO bf16 rounding (the mode pinned to torch.nn.LSTM): bound =
    the kernel's 1e-3 plus the gap between the two oracle modes pinned on the CPU
    (tests/test_oracle_bf16_gap.py), so the rounding points are not only checked against an oracle
    that rounds at the same places."""
    w = _workload(128, 3, 128, P=4, sigma=0.1)
    s = Solver(w, rollout_kernel=kernel)
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    enc, dec, tgt = oracle.seq2seq_queries(w.seed, 0, w.batch, 3)
    for m in range(w.pop_size):
        want = oracle.seq2seq_fitness(theta[m], 128, 3, enc, dec, tgt, False)[0]
        assert abs(fit[m] - want) / max(abs(want), 1.0) < 2e-3, (m, fit[m], want)


def test_tensor_core_and_cuda_core_kernels_agree_and_repeat():
    w = _workload(128, 3, 128, P=150, sigma=0.05)                # more items than SMs: blocks loop
    a = Solver(w, rollout_kernel=ROLLOUT_TILED)
    b = Solver(w, rollout_kernel=ROLLOUT_GENERIC)
    a.ask(); b.ask()
    fa = a.rollout().clone(); fa2 = a.rollout().clone(); fb = b.rollout().clone()
    assert torch.equal(fa, fa2)
    assert float((fa - fb).abs().max()) < FIT_TOL
    assert a.sync_status() == 0 and b.sync_status() == 0


def test_bench_size_workload_sampled_members():
    """The workload bench.py times (P = 1024, 128 queries, h = 128) in its launch configuration:
    members sampled across the population (first, last, and the block-loop boundaries at multiples
    of the SM count) against the oracle one by one; every fitness finite and below zero."""
    w = W.SEQ2SEQ
    s = Solver(w)
    theta = s.ask()
    fit = s.rollout().cpu().numpy()
    assert s.sync_status() == 0
    assert np.all(np.isfinite(fit)) and np.all(fit < 0.0)
    h, nd = w.layer_sizes[0], int(w.task_param[0])
    enc, dec, tgt = oracle.seq2seq_queries(w.seed, 0, w.batch, nd)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    for m in sorted({0, 1, sm - 1, sm, 2 * sm + 1, w.pop_size // 2, w.pop_size - 1}):
        row = theta[m].cpu().numpy()
        want = oracle.seq2seq_fitness(row, h, nd, enc, dec, tgt, True)[0]
        assert abs(fit[m] - want) < FIT_TOL, (m, fit[m], want)


def test_zero_parameters_and_generation_dependence():
    w = _workload(128, 3, 128, P=2, sigma=0.1)
    s = Solver(w)
    s.ask()
    zero = s.padded_rows(2); zero.zero_()
    fit = s.rollout(theta=zero).cpu().numpy()
    assert np.max(np.abs(fit + math.log(12))) < 1e-6
    f0 = s.rollout().clone()
    s.tell(f0)
    s.ask()
    f1 = s.rollout().clone()
    assert not torch.equal(f0, f1)                               # new centre and new queries
    assert s.sync_status() == 0


def test_second_generation_uses_that_generations_queries():
    w = _workload(128, 2, 64, P=4, sigma=0.1)
    s = Solver(w)
    s.ask(); s.tell(s.rollout())
    theta = s.ask().cpu().numpy()
    fit = s.rollout().cpu().numpy()
    want = _oracle_fits(w, theta, 1)
    for m in range(w.pop_size):
        assert abs(fit[m] - want[m][0]) < FIT_TOL


def test_config_errors():
    from paper_2202_05008_b200 import EvoError
    with pytest.raises(EvoError):
        Solver(_workload(128, 3, 128, P=2).with_(param_dim=1000))
    with pytest.raises(EvoError):
        Solver(_workload(48, 3, 128, P=2))                        # width not a multiple of 32
    with pytest.raises(EvoError):
        Solver(_workload(128, 5, 128, P=2))                       # more digits than supported
    s = Solver(_workload(64, 3, 128, P=2), rollout_kernel=ROLLOUT_TILED)
    s.ask()
    with pytest.raises(EvoError):
        s.rollout()                                               # the tensor-core kernel needs h = 128


@pytest.mark.parametrize("h", [32, 64, 96])
@pytest.mark.parametrize("nd,B,P", [(1, 1, 2), (3, 7, 6), (2, 64, 4), (2, 65, 300), (4, 129, 6)])
def test_narrow_cells_on_tensor_cores_match_oracle(h, nd, B, P):
    """n-tiles of 8 queries and blocks of up to 8 of them, full and not; against the bf16 oracle and the CUDA-core kernel
    (both round the same operands; left are accumulation order and gates to about 3e-7)."""
    w = _workload(h, nd, B, P=P, sigma=0.2)
    a, b = Solver(w), Solver(w, rollout_kernel=ROLLOUT_GENERIC)
    theta = a.ask().cpu().numpy(); b.ask()
    fa = a.rollout().clone(); again = a.rollout(); fb = b.rollout()
    assert a.sync_status() == 0 and b.sync_status() == 0
    assert torch.equal(fa, again)
    assert torch.max(torch.abs(fa - fb)) < FIT_TOL
    members = [0, P - 1]
    want = _oracle_fits(w, theta[members], 0)
    for i, m in enumerate(members):
        assert abs(float(fa[m]) - want[i][0]) < FIT_TOL


@pytest.mark.parametrize("h", [32, 64, 96])
@pytest.mark.parametrize("nd,B,P", [(1, 100, 300), (1, 400, 60), (1, 112, 296), (1, 9, 750), (2, 400, 250), (3, 133, 302)])
def test_runs_of_tiles_that_begin_and_end_inside_a_member(h, nd, B, P):
    """The blocks' runs of n-tiles: of several members, of a part of one, in one piece and several (of one member too: 133 and 400 queries);
    every member against the CUDA-core kernel.  Both round the same operands; left are accumulation order, gates to about 3e-7 and, by these,
    a hidden state here and there that rounds to the neighbouring bf16 value: 5e-3 of one position's loss at most were seen,
    where a position lost or taken from another query changes its loss by 0.1 and more."""
    w = _workload(h, nd, B, P=P, sigma=0.2)
    a, b = Solver(w), Solver(w, rollout_kernel=ROLLOUT_GENERIC)
    a.ask(); b.ask()
    fa = a.rollout().clone(); again = a.rollout(); fb = b.rollout()
    assert a.sync_status() == 0 and b.sync_status() == 0
    assert torch.equal(fa, again)
    assert torch.max(torch.abs(fa - fb)) < FIT_TOL
    assert torch.max(torch.abs(fa - fb)) < 2e-2 / (B * (nd + 1))
    a.close(); b.close()
