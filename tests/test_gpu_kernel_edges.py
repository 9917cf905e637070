"""Every round kernel and aggregation shape at the edges of its tiles, blocks and launch rules, against the CPU checker.

A client's first round starts from w_0 on both sides, so its update sum is held to the per-round bar; which kernel and
cluster width runs it is set by how many clients the launch holds.  Later rounds start from models that differ by
round-off and are held to the end-to-end bars."""
import threading

import numpy as np
import pytest
import torch

from oracle import sim
from paper_2112_13935_b200 import api, workloads
from gpu_helpers import U_TOL, check_against_oracle, make, rel_err, run_gpu, to_device

pytestmark = pytest.mark.gpu

BF16_TOL, BF16_FLIP_FRAC, BF16_FLIP_TOL = 3e-4, 1e-2, 3e-2   # a bf16 rounding or a ReLU mask may fall the other way


def check(cfg, w_tol=2e-5, bf16=False):
    data, w0 = make(cfg)
    ref = sim.run(cfg, data, w0)
    gpu = run_gpu(cfg, data, w0)
    check_against_oracle(cfg, data, w0, gpu, ref)
    assert rel_err(gpu["w"], ref["w"]) <= (1e-3 if bf16 else w_tol)
    for e in ref["events"]:
        k = e["seq"]
        want = np.asarray(ref["U"][k])
        d = np.abs(gpu["U"][k] - want) / max(np.abs(want).max(), 1e-300)
        if not bf16:
            assert d.max() <= (U_TOL if e["round"] == 0 else 1e-4), (e["client"], e["round"], d.max())
        elif e["round"] == 0:
            assert (d > BF16_TOL).mean() <= BF16_FLIP_FRAC and d.max() <= BF16_FLIP_TOL, (e["client"], d.max())


@pytest.mark.parametrize("l2", [0.0, 1e-3])
@pytest.mark.parametrize("n_clients", [3, 33, 74, 100, 200])    # clusters of eight, four, two (the most of the last two); one CTA; two CTAs per SM
@pytest.mark.parametrize("first", [1, 7, 15, 31])           # rounds of first, first + 1, first + 2 samples: around blocks of 8 and 16
def test_regression_rounds_around_whole_blocks(n_clients, first, l2):
    check(workloads.get_config("cfg5", n_clients=n_clients, n_rounds=3, sched_a=1, sched_b=first, l2=l2, lr=0.002 if n_clients < 10 else 1e-4,
                               data=dict(per_client=40)))


# Clusters of eight (up to 15 round-tasks on this part), of six (up to 22, rounds above 64 samples) and of four (shorter ones); blocks of
# sixteen, rings of three and four blocks.
@pytest.mark.parametrize("n_clients,first,l2", [(1, 16, 0.0), (15, 33, 1e-3), (16, 1, 1e-3), (16, 48, 0.0), (22, 17, 1e-3), (22, 79, 0.0),
                                                (16, 65, 1e-3), (16, 80, 0.0), (22, 81, 1e-3), (19, 128, 1e-3)])
def test_regression_rounds_of_few_clients(n_clients, first, l2):
    check(workloads.get_config("cfg5", n_clients=n_clients, n_rounds=3, sched_a=15, sched_b=first, l2=l2, lr=0.03 / n_clients, data=dict(per_client=40)))


# Hand-overs inside the kernels on clusters: a race between the warps that add up couplings gave a few of such runs other bits.
@pytest.mark.parametrize("over", [
    dict(n_clients=95, n_rounds=22, sched_a=6, sched_b=28, l2=0.0), dict(n_clients=41, n_rounds=10, sched_a=7, sched_b=9, l2=1e-4),
    dict(n_clients=44, n_rounds=51, sched_a=5, sched_b=11, l2=0.0, topology=1), dict(n_clients=16, n_rounds=32, sched_a=4, sched_b=9, l2=1e-4, topology=1),
])
def test_regression_runs_repeat_bit_for_bit(over):
    cfg = workloads.get_config("cfg5", lr=0.02 / over["n_clients"], data=dict(per_client=100), **over)
    data, w0 = make(cfg)
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        seen = set()
        for _ in range(40):
            s.reset()
            s.run()
            seen.add(b"".join(api.aet_get_node_model(s.h, c).tobytes() for c in range(cfg["n_clients"])) if cfg.get("topology") else s.model().tobytes())
    assert len(seen) == 1, len(seen)


# A step moves a sample's own logits by eta (|x|^2 + 1), 16 eta and more here: 33 samples carry corrections far beyond the exponential's
# range, which the walk has to shift out.  The bar: one fp32 rounding (2^-24) per step, each amplified by no more than the softmax's
# 1/2 x 16 eta per later step that shares its class.
@pytest.mark.parametrize("n_clients,lr,samples", [(3, 0.2, 33), (3, 2.0, 33), (18, 2.0, 33),    # (from 20 on the checker's own loss overflows)
                                                  (18, 0.2, 66)])                                # clusters of six
def test_regression_rounds_with_steps_that_swing(n_clients, lr, samples):
    check(workloads.get_config("cfg5", n_clients=n_clients, n_rounds=1, sched_a=1, sched_b=samples, lr=lr, data=dict(per_client=40)))


def round_rms(cfg, w0, clients):
    """rms error of the first round's update sums over the rms of the sums, all parameters of `clients` together."""
    data = workloads.make_client_data(cfg)
    got = run_gpu(cfg, data, w0)
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        s.run()
        seq = {e["client"]: e["seq"] for e in s.log()[0]}
    err = ref = 0.0
    for c in clients:
        want, _ = sim.run_task(cfg, data[c], c, 0, w0.astype(np.float64))
        err += ((got["U"][seq[c]] - want) ** 2).sum()
        ref += (want ** 2).sum()
    return float(np.sqrt(err / ref))


# What sums of fp32 FMAs in this order leave: 0.42e-7 at 5 samples, 0.67e-7 at 50, 2.0e-7 at 600 (measured against fp64); operands of
# 22 bits instead of 24 would show at 50 (1.5e-7).  Crowded launches (200 clients): the kernels before left 1.5e-7 at 12 samples, 1.25e-7
# with l2; cut operands 1.6e-7 and 1.5e-7.
@pytest.mark.parametrize("n_clients,samples,l2,bar", [
    # clusters of eight, four (of six from 65 samples on), four, two; one CTA
    *[(n, s, 0.0, bar) for n in (3, 20, 33, 50, 100) for s, bar in ((5, 0.46e-7), (50, 0.9e-7), (600, 2.2e-7))],
    (200, 12, 0.0, 1.1e-7), (200, 12, 1e-4, 1.0e-7), (200, 50, 0.0, 1.1e-7),
])
def test_regression_rounds_are_as_good_as_fp32_sums(n_clients, samples, l2, bar):
    cfg = workloads.get_config("cfg5", n_clients=n_clients, n_rounds=1, sched_a=1, sched_b=samples, l2=l2, lr=0.002, data=dict(per_client=64))
    w0 = np.random.default_rng(0).normal(0, 0.05, workloads.n_params(cfg["dims"])).astype(np.float32)
    assert round_rms(cfg, w0, range(3)) <= bar


@pytest.mark.parametrize("dims,batch,n_clients", [
    ([784, 128, 10], 32, 4), ([784, 128, 10], 32, 20), ([784, 128, 10], 32, 40), ([784, 128, 10], 32, 80),   # clusters of 8, 4, 2, 1
    ([784, 128, 32], 64, 4),          # most samples and classes
    ([50, 17, 10], 7, 3),             # one hidden tile and a bit, minibatch inside a tile, rows not a multiple of 16 bytes
    ([100, 16, 10], 9, 3), ([100, 112, 33, 12], 17, 3), ([272, 20, 20, 20, 15], 33, 3), ([64, 100, 10], 41, 3), ([64, 30, 10], 50, 3),
    ([784, 112, 12, 10], 50, 3), ([783, 100, 10], 50, 3), ([784, 112, 10], 56, 20),   # one buffer for the rows
])
def test_fp32_mlp_rounds(dims, batch, n_clients):
    check(workloads.get_config("cfg3", n_clients=n_clients, n_rounds=2, dims=dims, batch=batch, sched_a=batch, sched_b=2 * batch, l2=1e-3,
                               data=dict(total=70 * n_clients, dim=dims[0])))


# Clusters of seven, six, five and three: units of inputs, and groups of hidden rows, that do not come out even.
@pytest.mark.parametrize("dims,batch,n_clients,bf16", [
    ([784, 112, 10], 24, 12, False), ([784, 128, 10], 32, 20, False), ([770, 17, 10], 8, 24, False), ([784, 128, 10], 16, 44, False),
    ([200, 100, 10], 32, 12, True), ([112, 64, 10], 32, 24, True), ([784, 128, 10], 32, 44, True),
])
def test_mlp_rounds_on_clusters_that_are_no_powers_of_two(dims, batch, n_clients, bf16):
    check(workloads.get_config("cfg4" if bf16 else "cfg3", n_clients=n_clients, n_rounds=2, dims=dims, batch=batch, sched_a=batch, sched_b=batch, l2=1e-3,
                               n_stragglers=0, data=dict(kind="iid", total=70 * n_clients, dim=dims[0])), bf16=bf16)


@pytest.mark.parametrize("dims,batch,n_clients", [
    ([512, 256, 10], 16, 4), ([520, 100, 30, 10], 48, 4), ([200, 17, 10], 33, 20), ([1024, 64, 16], 64, 80),   # first layer on the chip
    ([1024, 256, 128, 10], 64, 4), ([512, 256, 128, 10], 64, 20), ([512, 256, 128, 10], 64, 50), ([160, 256, 128, 16], 64, 90),
    ([1024, 256, 128, 10], 32, 50), ([1024, 256, 128, 10], 64, 16), ([1024, 256, 10], 64, 4), ([512, 256, 10], 32, 50), ([128, 256, 11], 64, 90),   # ... streamed: clusters of 8, 4, 2, 1
])
def test_bf16_mlp_rounds(dims, batch, n_clients):
    check(workloads.get_config("cfg4", n_clients=n_clients, n_rounds=2, dims=dims, batch=batch, sched_a=batch, sched_b=2 * batch, l2=1e-3,
                               n_stragglers=0, data=dict(kind="iid", total=70 * n_clients, dim=dims[0])), bf16=True)


# Sums of fp32 FMAs leave 0.7e-7 to 1.0e-7 after two iterations (measured against fp64); operands of 22 bits instead of 24, or
# long sums cut by the tensor cores, would show as 1.4e-7 to 3e-7.
@pytest.mark.parametrize("dims,batch,n_clients", [
    ([784, 128, 10], 32, 4), ([784, 128, 10], 32, 20), ([784, 128, 10], 32, 40), ([784, 128, 10], 32, 80), ([784, 100, 37, 10], 20, 12),
    ([50, 17, 10], 7, 3), ([272, 20, 20, 20, 15], 33, 3), ([784, 64, 10], 16, 8), ([784, 112, 12, 10], 50, 3), ([300, 12], 9, 3),
])
def test_fp32_mlp_rounds_are_as_good_as_fp32_sums(dims, batch, n_clients):
    cfg = workloads.get_config("cfg3", n_clients=n_clients, n_rounds=1, dims=dims, batch=batch, sched_a=batch, sched_b=2 * batch, l2=1e-4,
                               lr=0.004, data=dict(total=80 * n_clients, dim=dims[0]))
    assert round_rms(cfg, make(cfg)[1], range(3)) <= 1.15e-7


# One iteration from the start model: a sum holds W_0's gradient to fp32 rounding (1e-7 of its rms); a bf16 rounding of an
# activation that falls the other way moves dZ, and with it W_0's gradient, by at most some 1e-5; (W_start - W_end) / eta would be
# off by 2^-25 |w| / eta, 2e-4 and more of the gradient's rms at this step size.
@pytest.mark.parametrize("dims,batch,n_clients,layers", [
    ([784, 100, 10], 32, 8, (0, 1)), ([200, 17, 10], 33, 20, (0, 1)), ([520, 100, 30, 10], 48, 4, (0, 1, 2)), ([1024, 64, 16], 64, 80, (0, 1)),
    ([512, 256, 10], 64, 4, (0,)), ([160, 256, 128, 16], 64, 4, (0, 1)), ([784, 128, 10], 32, 40, (0, 1)),
    ([1024, 256, 128, 10], 32, 50, (1,)),    # W_0 streams, W_1's sum is kept
])
def test_bf16_update_sums_are_sums(dims, batch, n_clients, layers):
    cfg = workloads.get_config("cfg4", n_clients=n_clients, n_rounds=1, dims=dims, batch=batch, sched_a=batch, sched_b=batch, n_stragglers=0,
                               lr=0.0005, data=dict(kind="iid", total=70 * n_clients, dim=dims[0]))
    data, w0 = make(cfg)
    gpu = run_gpu(cfg, data, w0)
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        s.run()
        events, _ = s.log()
    for k in (0, len(events) - 1):
        want, _ = sim.run_task(cfg, data[events[k]["client"]], events[k]["client"], 0, w0.astype(np.float64))
        at = 0
        for l in range(len(dims) - 1):
            n = dims[l] * dims[l + 1]
            d, ref = gpu["U"][k][at:at + n] - want[at:at + n], want[at:at + n]
            if l in layers:
                assert np.sqrt((d * d).mean() / (ref * ref).mean()) <= 2e-5, (events[k]["client"], l)
            at += n + dims[l + 1]


@pytest.mark.parametrize("batch,n_clients", [(1, 3), (8, 3), (9, 3), (16, 20), (17, 3), (24, 3), (24, 20), (25, 3)])   # (the last two: the general kernel)
def test_conv_rounds(batch, n_clients):
    check(workloads.get_config("cfg7", n_clients=n_clients, n_rounds=2, batch=batch, sched_a=batch, sched_b=batch, l2=1e-3,
                               data=dict(total=60 * n_clients)))


# Sums of fp32 FMAs leave 0.9e-7 to 1.06e-7 (measured against fp64, one iteration); operands of 22 bits 1.2e-7 to 1.5e-7.
@pytest.mark.parametrize("batch,n_clients", [(8, 3), (16, 3), (16, 20), (24, 3)])   # clusters of eight and four
def test_conv_rounds_are_as_good_as_fp32_sums(batch, n_clients):
    cfg = workloads.get_config("cfg7", n_clients=n_clients, n_rounds=1, batch=batch, sched_a=batch, sched_b=batch, l2=1e-4,
                               data=dict(total=60 * n_clients))
    assert round_rms(cfg, make(cfg)[1], range(3)) <= 1.1e-7


@pytest.mark.parametrize("n_clients", [1, 64, 65, 3100])   # updates between two waves: one, around a sub-range, more than a cluster holds at once
def test_aggregation_of_short_and_long_ranges(n_clients):
    cfg = workloads.get_config("cfg5", n_clients=n_clients, n_rounds=2, sched_a=0, sched_b=1, lr=1e-4, data=dict(per_client=4))
    data, w0 = make(cfg)
    ref = sim.run(cfg, data, w0)
    gpu = run_gpu(cfg, data, w0)
    check_against_oracle(cfg, data, w0, gpu, ref)
    acc = w0.astype(np.float64)
    for e in ref["events"]:
        acc -= sim.step_size(cfg, e["round"]) * gpu["U"][e["seq"]].astype(np.float64)
    assert np.abs(acc - gpu["w"]).max() <= 2e-6 * max(1.0, np.abs(acc).max())


def wave_us(cfg):
    """Device time of one wave: the median over passes of a one-round run."""
    data, w0 = make(cfg)
    times = []
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        for _ in range(15):
            s.reset()
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            begin.record()
            s.run()
            end.record()
            torch.cuda.synchronize()
            times.append(begin.elapsed_time(end))
    return float(np.median(times[3:]))


# A wave on clusters of which the device runs too few at once is two waves; on narrower ones it is one.  So a few clients more on
# the next narrower cluster never make the wave shorter (two waves took 1.15 to 1.45 times as long as those).
@pytest.mark.parametrize("name,over,fewer,more", [
    ("cfg4", dict(n_stragglers=0, sched_a=64, sched_b=1280, data=dict(kind="per_client", per_client=64)), 16, 17),
    ("cfg4", dict(n_stragglers=0, sched_a=64, sched_b=1280, data=dict(kind="per_client", per_client=64)), 35, 38),
    ("cfg7", dict(sched_a=16, sched_b=320, data=dict(kind="per_client", per_client=64)), 16, 17),
    ("cfg5", dict(sched_a=1, sched_b=400, lr=1e-4, data=dict(per_client=64)), 70, 75),
])
def test_fewer_clients_never_take_longer(name, over, fewer, more):
    t = [wave_us(workloads.get_config(name, n_clients=n, n_rounds=1, **over)) for n in (fewer, more)]
    assert t[0] <= 1.08 * t[1], t


def test_handles_of_several_threads_share_released_memory():
    cfgs = [workloads.get_config("cfg5", n_clients=n, n_rounds=3, data=dict(per_client=32)) for n in (5, 70, 170)]
    made = [make(c) for c in cfgs]
    want = [run_gpu(c, d, w, want_U=False)["w"].tobytes() for c, (d, w) in zip(cfgs, made)]
    got = [[] for _ in range(4)]

    def work(i):
        for j in range(6):
            k = (i + j) % 3
            got[i].append((k, run_gpu(cfgs[k], *made[k], want_U=False)["w"].tobytes()))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(len(g) == 6 and all(w == want[k] for k, w in g) for g in got)


@pytest.mark.parametrize("shift", [0, 1])   # floats off a 16-byte boundary: the specialised kernel, the general one
def test_one_round_without_allocation_on_any_alignment(shift):
    cfg = workloads.get_config("cfg1", data=dict(per_client=100))
    data, w0 = make(cfg)
    buf = torch.zeros(3, w0.size + 4, dtype=torch.float32, device="cuda")
    w, U, w_end = (buf.view(-1)[i * (w0.size + 4 - (w0.size % 4)) + shift:][:w0.size] for i in range(3))
    w.copy_(torch.from_numpy(w0))
    x, y = to_device(data)[1]
    api.aet_round_no_alloc(cfg, 1, 2, x, y, w, U, w_end)
    torch.cuda.synchronize()
    U_ref, w_ref = sim.run_task(cfg, data[1], 1, 2, w0.astype(np.float64))
    assert rel_err(U.cpu().numpy(), U_ref) <= U_TOL and rel_err(w_end.cpu().numpy(), w_ref) <= U_TOL


# The end model leaves through the buffers the update sum left through: the sum is, bit for bit, that of a run, which asks for no end model.
@pytest.mark.parametrize("samples,l2", [(1, 0.0), (17, 1e-3), (50, 0.0), (160, 1e-3)])
def test_update_sums_beside_end_models(samples, l2):
    cfg = workloads.get_config("cfg5", n_clients=15, n_rounds=1, sched_a=1, sched_b=samples, l2=l2, lr=0.002, data=dict(per_client=64))
    w0 = np.random.default_rng(1).normal(0, 0.05, workloads.n_params(cfg["dims"])).astype(np.float32)
    data = workloads.make_client_data(cfg)
    gpu = run_gpu(cfg, data, w0)
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        s.run()
        seq = {e["client"]: e["seq"] for e in s.log()[0]}
        w, U, w_end = torch.from_numpy(w0).cuda(), torch.empty(w0.size, device="cuda"), torch.empty(w0.size, device="cuda")
        for c, (x, y) in enumerate(to_device(data)):
            for _ in range(4):
                api.aet_round_no_alloc(cfg, c, 0, x, y, w, U, w_end)
                assert U.cpu().numpy().tobytes() == gpu["U"][seq[c]].tobytes(), c
            assert rel_err(w_end.cpu().numpy(), sim.run_task(cfg, data[c], c, 0, w0.astype(np.float64))[1]) <= U_TOL


# A round restarted on its own runs the kernel and the cluster width that ran it among all the others: the same bits.
@pytest.mark.parametrize("n_clients,samples,l2", [(15, 40, 0.0), (16, 40, 0.0), (16, 70, 1e-3), (22, 70, 0.0), (33, 70, 1e-3), (34, 40, 0.0),
                                                  (74, 70, 0.0), (75, 40, 0.0), (150, 40, 1e-3)])
def test_restarted_regression_rounds_run_the_kernel_of_the_wave(n_clients, samples, l2):
    cfg = workloads.get_config("cfg5", n_clients=n_clients, n_rounds=1, sched_a=1, sched_b=samples, l2=l2, lr=0.001, data=dict(per_client=40))
    data, w0 = make(cfg)
    gpu = run_gpu(cfg, data, w0)
    with api.Session(cfg, to_device(data), torch.from_numpy(w0).cuda()) as s:
        s.run()
        for e in s.log()[0][::max(1, n_clients // 5)]:
            U, w_end = api.aet_debug_run_client_round(s.h, e["client"], 0, w0)
            assert U.tobytes() == gpu["U"][e["seq"]].tobytes(), e["client"]
            assert rel_err(w_end, sim.run_task(cfg, data[e["client"]], e["client"], 0, w0.astype(np.float64))[1]) <= U_TOL


@pytest.mark.parametrize("name,over", [
    ("cfg5", dict(n_clients=5, data=dict(per_client=1))), ("cfg5", dict(n_clients=3, data=dict(per_client=668))),
    ("cfg5", dict(n_clients=3, data=dict(per_client=669))),                       # the last size fetched by a kernel, the first copied
    ("cfg3", dict(n_clients=3, dims=[50, 17, 10], data=dict(total=301, dim=50))),   # rows that are not whole 16-byte pieces
    ("cfg4", dict(n_clients=3, n_stragglers=0, dims=[200, 64, 10], data=dict(kind="iid", total=500, dim=200))),   # bf16
])
def test_client_data_from_page_locked_pageable_and_device_memory(name, over):
    cfg = workloads.get_config(name, n_rounds=2, **over)
    data, w0 = make(cfg)
    cpu = [(torch.from_numpy(x), torch.from_numpy(y)) for x, y in data]
    got = []
    for place in (lambda t: t, lambda t: t.pin_memory(), lambda t: t.cuda()):
        with api.Session(cfg, [(place(x), place(y)) for x, y in cpu], torch.from_numpy(w0).cuda()) as s:
            s.run()
            got.append(s.model().tobytes())
    assert got[0] == got[1] == got[2]
