"""Performance cases: one generation (ask -> rollout -> tell) through ``Solver``, as a training loop
drives it, over the range of tasks, policies and sizes that the library is used with.

Every solver starts in the middle of a training run (a centre that has moved, filled optimiser
moments), which is where nearly all generations of a run are, and where the update depends smoothly
on the fitness.
"""
import math

import torch

from paper_2202_05008_b200 import Solver
from paper_2202_05008_b200 import workloads as W

ADAM_STEP = 40          # generations done before the first timed one

CARTPOLE = (1.0, 0.1, 0.5, 9.8, 0.01, 0.2)


def _control(task, sizes, pop, episodes, horizon, **kw):
    return dict({"family": "control", "task": task, "sizes": "-".join(map(str, sizes)), "pop": pop, "episodes": episodes,
                 "horizon": horizon, "regenerated": False, "clipup": False, "adapt_sigma": False}, **kw)


def listed():
    return [
        # the smallest control problem: a few thousand parameters in all, launches and latency only
        _control("cartpole", (5, 16, 16, 1), 16, 1, 200, name="cartpole_small"),
        # the ordinary one: a swing-up population that does not fill the GPU evenly, full episodes
        _control("cartpole", (5, 64, 64, 1), 256, 16, 1000, name="cartpole_medium"),
        # the largest control problem: thousands of members, long episodes
        _control("tanh_linear", (28, 128, 128, 8), 4096, 4, 1000, name="tanh_linear_large"),
        # uneven layers, population and episodes; noise recomputed to save its memory, sigma adapted
        _control("tanh_linear", (28, 96, 40, 8), 250, 3, 500, name="tanh_linear_ragged", regenerated=True, adapt_sigma=True),
        # a policy with another number of layers than two hidden ones
        _control("tanh_linear", (28, 64, 64, 64, 8), 512, 4, 200, name="mlp_deep"),
        # supervised: the ordinary population and batch
        {"name": "cnn", "family": "cnn", "pop": 64, "batch": 1024, "regenerated": False, "clipup": False, "adapt_sigma": False},
        # supervised: many members, a batch that is no multiple of a tile
        {"name": "cnn_large", "family": "cnn", "pop": 500, "batch": 1000, "regenerated": False, "clipup": True, "adapt_sigma": False},
        # recurrent encoder-decoder: the ordinary width
        {"name": "seq2seq", "family": "seq2seq", "hidden": 128, "digits": 3, "pop": 1024, "batch": 128,
         "regenerated": False, "clipup": False, "adapt_sigma": False},
        # recurrent, a narrower cell, odd population and batch
        {"name": "seq2seq_narrow", "family": "seq2seq", "hidden": 64, "digits": 2, "pop": 300, "batch": 100,
         "regenerated": False, "clipup": True, "adapt_sigma": False},
        # the solver on its own: triangles painted over a target image
        {"name": "paint", "family": "paint", "triangles": 64, "width": 128, "height": 128, "pop": 1024,
         "regenerated": False, "clipup": False, "adapt_sigma": False},
        # ask and tell only (the caller evaluates): the largest population, noise kept
        {"name": "update_stored", "family": "update", "dim": 131072, "pop": 16384, "regenerated": False, "clipup": False,
         "adapt_sigma": False},
        # ask and tell only: the most parameters, no multiple of anything; noise recomputed, ClipUp, sigma adapted
        {"name": "update_regenerated", "family": "update", "dim": 1000003, "pop": 2000, "regenerated": True, "clipup": True,
         "adapt_sigma": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pop(rng, lo, hi):
    return max(2, _log_int(rng, lo, hi) // 2 * 2)


def _macs(sizes):
    return sum(a * b for a, b in zip(sizes[:-1], sizes[1:]))


def draw(rng):
    opt = {"regenerated": rng.random() < 0.25, "clipup": rng.random() < 0.3, "adapt_sigma": rng.random() < 0.3}
    kind = rng.choice(["cartpole", "tanh_linear", "mlp", "cnn", "seq2seq", "paint", "update"])
    if kind == "cartpole":
        sizes = (5, rng.randint(8, 128), rng.randint(8, 128), 1)
        pop, episodes = _pop(rng, 16, 600), rng.randint(1, 24)
        horizon = max(20, min(_log_int(rng, 50, 1000), 8000000000 // (pop * episodes * (_macs(sizes) + 352))))
        return _control("cartpole", sizes, pop, episodes, horizon, **opt)
    if kind == "tanh_linear":
        sizes = (28, rng.randint(16, 128), rng.randint(16, 128), 8)
        pop, episodes = _pop(rng, 16, 4096), rng.randint(1, 12)
        horizon = max(20, min(_log_int(rng, 50, 1000), 4000000 // (pop * ((episodes + 3) // 4))))
        return _control("tanh_linear", sizes, pop, episodes, horizon, **opt)
    if kind == "mlp":
        task = rng.choice(["cartpole", "tanh_linear"])
        inner = tuple(_log_int(rng, 8, 192) for _ in range(rng.choice([1, 3, 3, 4])))
        sizes = (5,) + inner + (1,) if task == "cartpole" else (28,) + inner + (8,)
        pop, episodes = _pop(rng, 16, 512), rng.randint(1, 16)
        horizon = max(20, min(_log_int(rng, 50, 200), 5000000000 // (pop * episodes * (_macs(sizes) + 1000))))
        return _control(task, sizes, pop, episodes, horizon, **opt)
    if kind == "cnn":
        pop = _pop(rng, 16, 512)
        return dict({"family": "cnn", "pop": pop, "batch": min(_log_int(rng, 50, 2048), 500000 // pop)}, **opt)
    if kind == "seq2seq":
        pop = _pop(rng, 16, 1024)
        return dict({"family": "seq2seq", "hidden": rng.choice([32, 64, 96, 128, 128]), "digits": rng.randint(1, 4), "pop": pop,
                     "batch": min(_log_int(rng, 16, 400), 100000 // pop)}, **opt)
    if kind == "paint":
        pop, width, height = _pop(rng, 32, 1024), rng.randint(32, 200), rng.randint(32, 200)
        return dict({"family": "paint", "triangles": max(4, min(_log_int(rng, 8, 200), 1000000000 // (pop * width * height))),
                     "width": width, "height": height, "pop": pop}, **opt)
    pop = _pop(rng, 64, 16384)
    return dict({"family": "update", "dim": min(_log_int(rng, 5000, 2000000), 2000000000 // pop), "pop": pop}, **opt)


def _sizes(case):
    return tuple(int(x) for x in case["sizes"].split("-"))


def _workload(case, seed):
    kw = dict(name="case", pop_size=case["pop"], seed=seed,
              noise_mode=W.NOISE_REGENERATED if case["regenerated"] else W.NOISE_STORED,
              optimizer=W.OPT_CLIPUP if case["clipup"] else W.OPT_ADAM,
              sigma_mode=W.SIGMA_PGPE if case["adapt_sigma"] else W.SIGMA_CONSTANT)
    f = case["family"]
    if f == "control":
        sizes, cart = _sizes(case), case["task"] == "cartpole"
        return W.Workload(param_dim=W.mlp_param_count(sizes), policy_kind=W.POLICY_MLP, layer_sizes=sizes,
                          action_scale=10.0 if cart else 1.0, task_kind=W.TASK_CARTPOLE if cart else W.TASK_TANH_LINEAR,
                          episodes=case["episodes"], horizon=case["horizon"], task_param=CARTPOLE if cart else (), **kw)
    if f == "cnn":
        return W.Workload(param_dim=W.CNN_PARAMS, policy_kind=W.POLICY_CNN_28, task_kind=W.TASK_SUPERVISED,
                          batch=case["batch"], **kw)
    if f == "seq2seq":
        return W.Workload(param_dim=W.seq2seq_param_count(case["hidden"]), policy_kind=W.POLICY_LSTM_SEQ2SEQ,
                          layer_sizes=(case["hidden"],), task_kind=W.TASK_SEQ2SEQ_ADD, batch=case["batch"],
                          task_param=(float(case["digits"]),), **kw)
    if f == "paint":
        return W.Workload(param_dim=10 * case["triangles"], task_kind=W.TASK_PAINT, lr=0.02,
                          task_param=(float(case["width"]), float(case["height"]), 0.0), **kw)
    return W.Workload(param_dim=case["dim"], sigma=0.02, **kw)


def prepare(case, seed):
    w = _workload(case, seed)
    s = Solver(w, device="cuda:0")
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(seed)
    D, P = w.param_dim, w.pop_size
    z = torch.randn(3, D, device="cuda:0", generator=gen)
    if case["family"] == "paint":
        # a painting on its way: triangles of some size spread over the canvas, half transparent
        at = torch.rand(case["triangles"], 2, device="cuda:0", generator=gen) * 1.6 - 0.8
        tri = z[0].view(-1, 10) * 0.6
        tri[:, :6] += at.repeat(1, 3)
        tri[:, 6:] = torch.rand(case["triangles"], 4, device="cuda:0", generator=gen) * 1.6 - 0.8
        centre = tri.reshape(-1)
    else:
        centre = 0.05 * z[0]
    # gradients of such a run are about this large; the moments hold what Adam (or ClipUp's velocity in
    # the first of them) has gathered of them
    g = w.sigma * 0.41 / math.sqrt(2.0 * P)
    if case["clipup"]:
        m, v = z[1] * (w.lr / math.sqrt(D)), torch.zeros(D, device="cuda:0")
    else:
        m, v = z[1] * (0.23 * g), (g * g * (1.0 - 0.999 ** ADAM_STEP)) * (0.5 + z[2].square() * 0.5)
    s.set_state(center=centre.contiguous(), m=m.contiguous(), v=v.contiguous(), generation=ADAM_STEP + seed % 1000,
                adam_step=ADAM_STEP)
    state = {"solver": s, "family": case["family"], "fitness": torch.empty(P, dtype=torch.float32, device="cuda:0")}
    if case["family"] == "cnn":
        images, labels = W.image_batch(seed, 0, w.batch)
        state["images"] = torch.tensor(images, device="cuda:0")
        state["labels"] = torch.tensor(labels, device="cuda:0")
    elif case["family"] == "paint":
        s.set_target(torch.tensor(W.paint_target(seed, case["width"], case["height"]), device="cuda:0"))
    elif case["family"] == "update":
        state["fitness"] = torch.randn(P, device="cuda:0", generator=gen)       # what the caller's evaluation gave
    # the search distribution that every generation updates in place
    state["out"] = {"fitness": state["fitness"], "center": s.center(), "sigma": s.sigma(), "m": s.moments()[0], "v": s.moments()[1]}
    return state


def run(state):
    s, out = state["solver"], dict(state["out"])
    out["theta"] = s.ask()
    if state["family"] != "update":                     # else the caller evaluates theta
        if state["family"] == "cnn":
            s.set_batch(state["images"], state["labels"])
        s.rollout(fitness=state["fitness"])
    s.tell(state["fitness"])
    return out


def work(case):
    w = _workload(case, 0)
    P, D = w.pop_size, w.param_dim
    # theta written once, the centre and the moments read and written; a normal per (pair, dimension)
    # (about 25 operations), two members and one term of the gradient made of it
    bytes_ = 4.0 * P * D + 4.0 * 7 * D + 8.0 * P
    flops = (P / 2.0) * D * (25.0 + 4.0 + 2.0)
    f = case["family"]
    if f == "control":
        # per environment step: the layers, and the dynamics (28 x 36, or four Runge-Kutta stages)
        macs = _macs(_sizes(case)) + (1008 if case["task"] == "tanh_linear" else 0)
        flops += P * w.episodes * w.horizon * (2.0 * macs + (200.0 if case["task"] == "cartpole" else 0.0))
    elif f == "cnn":
        bytes_ += 4.0 * 784 * w.batch
        flops += 645120.0 * P * w.batch
    elif f == "seq2seq":
        h, nd = case["hidden"], case["digits"]
        flops += P * w.batch * ((3 * nd + 2) * 2.0 * 4 * h * (h + 13) + (nd + 1) * 2.0 * 12 * h)
    elif f == "paint":
        # the pixels that a triangle covers: about a fifteenth of the canvas each, 6 operations
        flops += P * case["width"] * case["height"] * (case["triangles"] * 0.4 + 9.0)
        bytes_ += 12.0 * case["width"] * case["height"]
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # The fitness itself agrees to about 1e-5 between the kernels of a task (and to 2e-4 over a population with a
    # few chaotic members); what shows is that two members whose fitness agrees to that may change ranks,
    # which moves the gradient.  Largest seen over the kernels of a task, and with every fitness off by 1e-6
    # at random: rel 1.3e-3 (the first moment), max 8.9e-3 (the fitness of a chaotic member).
    if case["family"] == "update":
        return {"rel": 1e-5, "max": 1e-4}               # ranks and noise are exact, sums are 32 and 64 bits
    return {"rel": 5e-3, "max": 3.6e-2}
