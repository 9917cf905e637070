"""Performance cases of the AET-SGD library: what its users run, through its public entry points.

A case names one training job (a model, the number of clients, the round schedule, the delays and options) and the
way a program drives it:

  run     a handle that stays open over data already loaded: reset, run all rounds, read the model(s) back
  loop    the same handle driven a few rounds at a time, the model read after every call (a program that evaluates
          as it trains)
  job     everything from pinned host buffers: create, prepare, load, run, model and event log back, destroy
  round   one round-task from the caller's own device buffers, with nothing allocated (aet_round_no_alloc)

Data follow the recipe of workloads.py (dark ten-class images, one label in ten redrawn), made on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_13935_b200 import api, workloads

LR, MLP, CONV = 0, 1, 2
NEVER = -1          # "lag": the checkpoint never blocks


def _case(name, **over):
    """Every field of a case, so that a case is complete by itself."""
    c = dict(how="run", model=LR, dims="784-10", bf16=False, batch=1, clients=16, rounds=5, chunk=0, a=10, b=10,
             base=0, lag=1, lr=0.01, beta=0.0, l2=0.0, uniform=False, net=0.5, stragglers=0, slow=1.0, ring=False,
             split=False, rows=20000, skew=0.0, ahead=False)
    assert set(over) <= set(c), over
    c.update(over)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One client's round for a caller that may not allocate: the smallest call there is (50 samples).
        _case("one_round", how="round", clients=4, rounds=5, a=10, b=10, l2=1e-4, rows=2000),
        # Four clients and 600 samples in all: a quick look at a setting, bound by launches and the chain of steps.
        _case("lr_4_clients_l2", clients=4, rounds=5, l2=1e-4, rows=8000),
        # A short job start to end from host memory: set-up, schedule, copies, run, results.
        _case("lr_job_64_clients", how="job", clients=64, rounds=10, a=8, b=8, lr=0.02 / 64, rows=12800, ahead=True),
        # 16 label-skewed clients, two of them ten times slower, rounds up to 600 samples: few long chains.
        _case("lr_16_skewed", clients=16, rounds=30, a=20, b=20, lr=0.002, stragglers=2, slow=10.0, rows=60000, skew=0.5),
        # Training with a look at the model after every second round; an odd number of clients and odd round sizes.
        _case("lr_loop_101_clients", how="loop", clients=101, rounds=12, chunk=2, a=7, b=9, lr=0.02 / 101, rows=40400),
        # 1,024 clients, short rounds: the crowded case, ten thousand round-tasks.
        _case("lr_1024_clients", clients=1024, rounds=10, a=8, b=8, lr=0.02 / 1024, rows=1024 * 1024),
        # The paper's own setting: a ring of five nodes, s_i = 10 i for 110 rounds, diminishing step, uniform delays.
        _case("lr_ring_paper", clients=5, rounds=110, a=10, b=0, base=1, beta=0.01, uniform=True, ring=True, rows=60000),
        # fp32 multi-layer perceptron on the 28x28 set, minibatch 32.
        _case("mlp_32_clients", model=MLP, dims="784-128-10", batch=32, clients=32, rounds=40, a=64, b=64, lr=0.001, net=1.0,
              rows=60000),
        # The same kind of job at widths and a minibatch nobody tuned for.
        _case("mlp_ragged", model=MLP, dims="784-100-37-10", batch=20, clients=12, rounds=10, a=40, b=60, lr=0.004, l2=1e-4,
              net=1.0, rows=9000),
        # The wide bf16 perceptron on the 32x32x3 set: 64 skewed clients, eight of them twenty times slower.
        _case("mlp_bf16_64_clients", model=MLP, dims="3072-256-128-10", bf16=True, batch=64, clients=64, rounds=30, a=128, b=128,
              lr=0.0005, stragglers=8, slow=20.0, rows=50000, skew=0.3),
        # A narrower bf16 perceptron with few clients.
        _case("mlp_bf16_narrow", model=MLP, dims="3072-128-32-10", bf16=True, batch=64, clients=12, rounds=10, a=128, b=64,
              lr=0.002, rows=12000),
        # The convolutional classifier of the LeNet shape.
        _case("conv_16_clients", model=CONV, dims="28-1-6-16-120-84-10", batch=16, clients=16, rounds=12, a=32, b=32, lr=0.005,
              net=1.0, rows=60000),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _rounds_for(chain, a, b, base, most):
    """Rounds that take a client's chain to about `chain` samples."""
    r, done = 0, 0
    while r < most and (r < 2 or done < chain):
        done += a * (base + r) + b
        r += 1
    return r


def draw(rng):
    kind = rng.choice(["lr", "lr", "lr_crowd", "lr_loop", "job", "round", "mlp", "mlp_ragged", "bf16", "bf16_narrow", "conv"])
    if kind in ("lr", "lr_crowd", "lr_loop", "job"):
        n = _log_int(rng, 2, 128) if kind == "lr" else _log_int(rng, 149, 1024) if kind == "lr_crowd" else _log_int(rng, 4, 200)
        base = rng.choice([0, 1])
        a = _log_int(rng, 3, 24)
        b = _log_int(rng, 1, 40) if base == 0 else rng.choice([0, _log_int(rng, 1, 40)])
        chain = _log_int(rng, 200, 20000) if kind == "lr" else _log_int(rng, 100, 900)
        rounds = _rounds_for(chain, a, b, base, 110)
        c = dict(clients=n, base=base, a=a, b=b, rounds=rounds, lr=0.02 / max(2, n) * rng.choice([0.5, 1.0]),
                 l2=rng.choice([0.0, 0.0, 1e-4]), beta=rng.choice([0.0, 0.01]), uniform=rng.random() < 0.3,
                 rows=n * _log_int(rng, 100, 1000))
        if kind == "lr":
            c.update(ring=rng.random() < 0.3, stragglers=rng.choice([0, n // 8]), slow=10.0, lag=rng.choice([0, 1, 1, 3, NEVER]))
            if not c["ring"] and rng.random() < 0.2:      # Algorithm 2's coin flips share a global round size
                c.update(split=True, a=a * n, b=(b + 1) * n)
        elif kind == "lr_crowd":
            c.update(net=rng.choice([0.1, 0.5, 5.0]), lag=rng.choice([1, 1, NEVER]))
        elif kind == "lr_loop":
            c.update(how="loop", chunk=rng.choice([1, 2, 3]), rounds=min(rounds, 16))
        else:
            c.update(how="job", rounds=min(rounds, 16), rows=n * _log_int(rng, 50, 400), ahead=True)
        return _case(None, **c)
    if kind == "round":
        a, b, rounds = _log_int(rng, 3, 24), _log_int(rng, 1, 40), _log_int(rng, 2, 20)
        return _case(None, how="round", clients=_log_int(rng, 2, 64), rounds=rounds, a=a, b=b, l2=rng.choice([0.0, 1e-4]),
                     lr=rng.choice([0.01, 0.005]), rows=64 * 200)
    if kind == "conv":
        batch = rng.choice([8, 12, 16, 16, 24, 32])
        n = _log_int(rng, 3, 32)
        return _case(None, model=CONV, dims="28-1-6-16-120-84-10", batch=batch, clients=n, rounds=rng.randint(3, 12),
                     a=batch * rng.choice([1, 2]), b=batch * rng.choice([1, 2]), lr=0.08 / max(16, n), net=1.0,
                     l2=rng.choice([0.0, 0.0, 1e-4]), rows=n * rng.randint(100, 1500))
    if kind == "mlp":
        n = _log_int(rng, 4, 64)
        return _case(None, model=MLP, dims="784-128-10", batch=32, clients=n, rounds=rng.randint(4, 30), a=32 * rng.choice([1, 2]),
                     b=32 * rng.choice([1, 2]), lr=0.032 / max(16, n), l2=rng.choice([0.0, 0.0, 1e-4]), net=1.0,
                     rows=n * rng.randint(200, 1500))
    if kind == "mlp_ragged":
        n, batch = _log_int(rng, 4, 32), rng.choice([8, 16, 20, 32, 50])
        hidden = rng.choice(["%d" % rng.randint(24, 128), "%d-%d" % (rng.randint(24, 128), rng.randint(12, 64))])
        return _case(None, model=MLP, dims="784-%s-10" % hidden, batch=batch, clients=n, rounds=rng.randint(4, 12),
                     a=batch * rng.choice([1, 2]), b=batch * rng.choice([1, 3]), lr=0.048 / max(16, n),
                     l2=rng.choice([0.0, 1e-4]), net=1.0, rows=n * rng.randint(200, 1000))
    if kind == "bf16":
        n = _log_int(rng, 4, 64)
        return _case(None, model=MLP, dims="%d-256-128-10" % rng.choice([1024, 2048, 3072, 3072]), bf16=True, batch=64, clients=n,
                     rounds=rng.randint(4, 16), a=64 * rng.choice([1, 2]), b=64 * rng.choice([1, 2]), lr=0.032 / max(16, n),
                     l2=rng.choice([0.0, 0.0, 1e-4]), stragglers=rng.choice([0, n // 8]), slow=20.0, rows=n * rng.randint(200, 800))
    n, batch = _log_int(rng, 4, 32), rng.choice([32, 64])
    return _case(None, model=MLP, dims="3072-%s-10" % rng.choice(["128-32", "128", "128-64", "256"]), bf16=True, batch=batch, clients=n,
                 rounds=rng.randint(4, 10), a=batch * rng.choice([1, 2]), b=batch * rng.choice([1, 2]), lr=0.024 / max(16, n),
                 rows=n * rng.randint(200, 800))


# ---- the job a case describes -----------------------------------------------------------------------------------

def _dims(case):
    return [int(v) for v in case["dims"].split("-")]


def _row_values(case):
    d = _dims(case)
    return d[0] * d[0] * d[1] if case["model"] == CONV else d[0]


def _config(case, seed):
    return dict(n_clients=case["clients"], model=case["model"], dims=_dims(case), precision=1 if case["bf16"] else 0,
                batch=case["batch"], sched_a=case["a"], sched_b=case["b"], round_base=case["base"],
                max_lag_d=workloads.NEVER_WAIT if case["lag"] == NEVER else case["lag"], lr=case["lr"], lr_beta=case["beta"],
                l2=case["l2"], seed=seed, delay_dist=1 if case["uniform"] else 0, compute_delay_mean=1.0,
                network_delay_mean=case["net"], compute_delay_lo=0.1, compute_delay_hi=1.0, network_delay_lo=0.1,
                network_delay_hi=1.5, straggler_factor=case["slow"], n_stragglers=case["stragglers"],
                split_mode=1 if case["split"] else 0, topology=1 if case["ring"] else 0, n_rounds=case["rounds"])


def _client_data(case, seed):
    """Per-client (x, y) on the GPU: the recipe of workloads.make_pool, split evenly (ragged) or with label skew."""
    n, rows, dim = case["clients"], case["rows"], _row_values(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    mu = torch.rand((workloads.N_CLASSES, dim), generator=g, device="cuda") * 2.5 - 2.0
    y = torch.randint(0, workloads.N_CLASSES, (rows,), generator=g, device="cuda", dtype=torch.int32)
    x = torch.empty((rows, dim), device="cuda")
    step = max(1, (1 << 28) // dim)
    for s in range(0, rows, step):
        part = x[s:s + step]
        part.normal_(generator=g)
        part.mul_(0.25).add_(mu[y[s:s + step].long()]).clamp_(0.0, 1.0)
    again = torch.rand((rows,), generator=g, device="cuda") < workloads.LABEL_NOISE
    other = torch.randint(0, workloads.N_CLASSES, (rows,), generator=g, device="cuda", dtype=torch.int32)
    y = torch.where(again, other, y).contiguous()
    if case["skew"]:
        parts = workloads.split_dirichlet(y.cpu().numpy(), n, case["skew"], seed + 1000, max(case["batch"], 8))
        return [(x[i].contiguous(), y[i].contiguous()) for i in (torch.from_numpy(p).cuda() for p in parts)]
    cuts = [rows * c // n for c in range(n + 1)]
    return [(x[lo:hi], y[lo:hi]) for lo, hi in zip(cuts, cuts[1:])]


class _State:
    """What a program holds between passes; the library's handle is closed with it."""

    def __init__(self, case, seed):
        self.case, self.cfg, self.session = case, _config(case, seed), None

    def __del__(self):
        if self.session is not None:
            self.session.close()


def prepare(case, seed):
    s = _State(case, seed)
    data = _client_data(case, seed)
    w0 = workloads.make_start_model(s.cfg)
    if case["how"] == "round":
        s.client, s.round = seed % case["clients"], case["base"] + case["rounds"] - 1
        s.x, s.y = (t.contiguous() for t in data[s.client])
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        s.w = torch.randn((w0.size,), generator=g, device="cuda") * 0.01
        s.U, s.w_end = torch.empty_like(s.w), torch.empty_like(s.w)
        s.conf = api.make_config(s.cfg)
    elif case["how"] == "job":
        s.data = [(x.cpu().pin_memory(), y.cpu().pin_memory()) for x, y in data]
        s.w0 = torch.from_numpy(w0).pin_memory()
        s.out = torch.empty(w0.size, dtype=torch.float32).pin_memory()
    else:
        s.session = api.Session(s.cfg, data, torch.from_numpy(w0).cuda())
    return s


def run(state):
    case, cfg = state.case, state.cfg
    if case["how"] == "round":
        api.aet_round_no_alloc(state.conf, state.client, state.round, state.x, state.y, state.w, state.U, state.w_end)
        return {"U": state.U, "w": state.w_end}
    if case["how"] == "job":
        h = api.aet_create(cfg)
        try:
            if case["ahead"]:
                api.aet_prepare_rounds(h, case["rounds"])
            api.aet_set_global_model(h, state.w0)
            for c, (x, y) in enumerate(state.data):
                api.aet_load_client_data(h, c, x, y)
            api.aet_run_rounds(h, case["rounds"])
            api.aet_get_global_model(h, state.out)
            log, summary = api.aet_get_event_log(h, raw=True)
        finally:
            api.aet_destroy(h)
        return {"w": state.out, "log": np.frombuffer(log, dtype=np.int32), "summary": summary}
    sess = state.session
    sess.reset()
    if case["how"] == "loop":
        seen = []
        for first in range(0, case["rounds"], case["chunk"]):
            sess.run(min(case["chunk"], case["rounds"] - first))
            seen.append(sess.model())
        return {"models": np.stack(seen)}
    sess.run(case["rounds"])
    if case["ring"]:
        return {"models": np.stack([api.aet_get_node_model(sess.h, c) for c in range(case["clients"])])}
    return {"w": sess.model()}


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def _samples(case):
    per_round = [case["a"] * (case["base"] + i) + case["b"] for i in range(case["rounds"])]
    if case["how"] == "round":
        return per_round[-1]
    return sum(per_round) * (1 if case["split"] else case["clients"])


def _flops_per_sample(case):
    d = _dims(case)
    if case["model"] == CONV:
        side, c_in, c1, c2, f1, f2, ncls = d
        s1 = side - workloads.CONV_K + 1
        s2 = s1 // 2 - workloads.CONV_K + 1
        k2 = workloads.CONV_K ** 2
        dense = c2 * (s2 // 2) ** 2 * f1 + f1 * f2 + f2 * ncls
        return 2 * (2 * c1 * c_in * k2 * s1 * s1 + 3 * c2 * c1 * k2 * s2 * s2 + 3 * dense)
    return sum(4 * d[k] * d[k + 1] for k in range(len(d) - 1)) + sum(2 * d[k] * d[k + 1] for k in range(1, len(d) - 1))


def work(case):
    """Forward and gradient products of every sample; the rows drawn (a row at most once), the models in and out."""
    samples = _samples(case)
    params = workloads.model_n_params(dict(model=case["model"], dims=_dims(case)))
    rows = min(samples, case["rows"])
    models = 2
    if case["how"] == "round":
        models = 3
    elif case["how"] == "loop":
        models = 1 + -(-case["rounds"] // case["chunk"])
    elif case["ring"]:
        models = 1 + case["clients"]
    if case["how"] == "job":
        rows = case["rows"]          # the whole data set crosses from the host
    value = 2 if case["bf16"] else 4
    return {"bytes": rows * (value * _row_values(case) + 4) + models * 4 * params, "flops": samples * _flops_per_sample(case)}


def tolerance(case):
    """fp32 sums in another order, carried through a chain of dependent steps."""
    if case["bf16"]:
        return {"rel": 1e-2}
    if case["model"] == LR:
        return {"rel": 1e-5}
    return {"rel": 1e-4, "max": 1e-2}
