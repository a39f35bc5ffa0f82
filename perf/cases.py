"""The work a training program has this library do, as a set of timed cases.

A case names one operator of the population library, a population (number of models, tensor
table, layout, element types) and the operator's options; `run` is one call of the public entry
points as a training loop makes it.  Sizes are the repository's own workloads (ResNet-18 and
ResNet-50 tensor tables, flat vectors) and generic flat vectors of odd lengths.

  op         "shuffle"    wash_shuffle / wash_shuffle_both, counters kept
             "consensus"  wash_shuffle_consensus over the quarters of the tensor table
             "ema"        papa_ema          "average"  population_average
             "papa_all"   papa_all
             "exchange"   plan, send, receive of one worker of the one-model-per-device form
             "host"       wash_step_host: the shuffling step over pinned host buffers
  table      tensor table (workloads.table_from_spec)
  dtype      parameters, opt: momentum beside them ("none": absent), out: the average's type
  schedule   per-layer probabilities ("none": uniform p)
  mode       "stream" (the default of a new context) or "auto" (what the README's loop sets)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_17517_b200 import binding as B
from paper_2405_17517_b200 import workloads as W

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
_CODE = {"f32": B.WASH_F32, "bf16": B.WASH_BF16}
_BYTES = {"f32": 4, "bf16": 2, "none": 0}
_MODE = {"stream": B.WASH_MODE_STREAM, "auto": B.WASH_MODE_AUTO}
_LARGEST_STACK = 1 << 32      # bytes of both stacks of a drawn case (the largest listed: 32 models of 2^25 fp32)
_LARGEST_HOST = 450_000_000   # the same for the step over host buffers (listed: 449 MB)
ALPHA = 0.99


def _case(op, N, table, p=0.0, dtype="f32", opt="none", layout="np", schedule="none", mode="stream", out="f32", **name):
    return dict(name, op=op, N=N, table=table, p=p, dtype=dtype, opt=opt, layout=layout, schedule=schedule, mode=mode, out=out)


def listed():
    return [
        # a step of a small model (or of one layer that is shuffled by itself): launch and host time count
        _case("shuffle", 3, "flat:1048576", 0.01, name="flat_n3"),
        # the training loop of the README on the small-image network: weights and momentum, rarely selected
        _case("shuffle", 5, "resnet18:100", 0.001, opt="f32", mode="auto", name="resnet18_n5_opt"),
        # the large network with per-layer probabilities, streamed whole: the benchmark's own workload
        _case("shuffle", 10, "resnet50:1000", 0.01, opt="f32", schedule="decreasing", name="resnet50_n10_opt"),
        # bf16 weights with fp32 momentum
        _case("shuffle", 8, "resnet50:1000", 0.005, dtype="bf16", opt="f32", mode="auto", name="resnet50_n8_bf16_opt"),
        # the paper's ImageNet setting: five models, p = 0.05 falling to 0 at the last layer, weights only
        _case("shuffle", 5, "resnet50:1000", 0.05, schedule="decreasing", mode="auto", name="resnet50_n5_p0.05"),
        # a pair of large models: little data per coordinate
        _case("shuffle", 2, "flat:134217728", 0.01, name="flat_n2_large"),
        # a large population, coordinate-major, a tenth of the coordinates selected
        _case("shuffle", 32, "flat:33554432", 0.1, layout="pn", name="flat_n32_pn"),
        # the shuffle that also reports the distance to the consensus, per quarter of the network
        _case("consensus", 5, "resnet18:100", 0.001, opt="f32", name="resnet18_n5_consensus"),
        # PAPA's pull toward the mean
        _case("ema", 8, "resnet50:1000", dtype="bf16", name="resnet50_n8_bf16_ema"),
        # the averaged model at the end of a run of the paper's largest population
        _case("average", 20, "resnet18:100", name="resnet18_n20_average"),
        # one model per device: this worker's part of a step
        _case("exchange", 5, "resnet50:1000", 0.01, opt="f32", schedule="decreasing", name="resnet50_n5_worker"),
        # stacks kept in pinned host memory between steps
        _case("host", 5, "resnet18:100", 0.001, opt="f32", name="resnet18_n5_host"),
    ]


def draw(rng):
    op = rng.choices(["shuffle", "consensus", "ema", "average", "papa_all", "exchange", "host"], [10, 2, 2, 2, 1, 2, 1])[0]
    # the population sizes of the configurations and of the paper, and any size in between
    N = rng.choice([2, 3, 4, 5, 8, 10, 16, 20, 32]) if rng.random() < 0.6 else rng.randint(2, 32)
    dtype = "bf16" if rng.random() < 0.3 else "f32"
    opt = "f32" if op in ("shuffle", "consensus", "exchange", "host") and rng.random() < 0.5 else "none"
    largest = _LARGEST_HOST if op == "host" else _LARGEST_STACK
    most = min(1 << 27, largest // (N * (_BYTES[dtype] + _BYTES[opt])))     # coordinates per model
    table = rng.choice(["resnet18:%d" % rng.choice([10, 100]), "resnet50:1000", "flat"])
    if table == "flat" or int(W.numels(W.table_from_spec(table)).sum()) > 0.99 * most:
        table = "flat:%d" % int(math.exp(rng.uniform(math.log(1 << 17), math.log(most))))
    return _case(op, N, table, p=round(10.0 ** rng.uniform(-4.0, 0.0), 6) if opt != "none" or op in ("shuffle", "consensus", "exchange", "host") else 0.0,
                 dtype=dtype, opt=opt, layout=rng.choice(["np", "np", "pn"]),
                 schedule="decreasing" if rng.random() < 0.4 and not table.startswith("flat") else "none",
                 mode=rng.choice(["stream", "auto"]), out=rng.choice(["f32", dtype]))


def _numel(case):
    return W.numels(W.table_from_spec(case["table"]))


def _p_layer(case, L):
    return B.wash_layer_probs(L, case["p"], B.WASH_SCHEDULE_DECREASING) if case["schedule"] == "decreasing" else None


def _selected(case, numel):
    """Expected number of selected coordinates of a step."""
    L = len(numel)
    share = case["p"] * (1.0 - np.arange(L) / max(L - 1, 1)) if case["schedule"] == "decreasing" and L > 1 else np.full(L, case["p"])
    return float((share * numel).sum())


def _stack(N, padded_P, layout, dtype, scale, drift, gen):
    """N models a small drift apart from a common point, on the device."""
    common = torch.randn(padded_P, device="cuda", generator=gen).mul_(scale)
    shape = (N, padded_P) if layout == "np" else (padded_P, N)
    stack = torch.randn(shape, device="cuda", generator=gen).mul_(drift)
    stack.add_(common if layout == "np" else common[:, None])
    return stack.reshape(-1).to(_TORCH[dtype])


def prepare(case, seed):
    N, numel = case["N"], _numel(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = dict(case=case, seed=seed, step=0, p=case["p"], p_layer=_p_layer(case, len(numel)),
             stats=torch.zeros(2, dtype=torch.int64, device="cuda"))
    layout = {"np": B.WASH_LAYOUT_NP, "pn": B.WASH_LAYOUT_PN}[case["layout"]]
    pop = s["pop"] = B.Population(N, numel, layout, 0)
    P = pop.padded_P
    if case["op"] == "exchange":
        _prepare_worker(s, case, numel, gen)
        return s
    stacks = [_stack(N, P, case["layout"], case["dtype"], 0.05, 0.005, gen)]
    if case["opt"] != "none":
        stacks.append(_stack(N, P, case["layout"], case["opt"], 0.0, 1e-3, gen))
    s["stacks"] = stacks
    for role, stack in zip((B.WASH_STACK_PARAMS, B.WASH_STACK_OPT), stacks):
        pop.bind(role, stack)
    B.wash_set_mode(pop.ctx, _MODE[case["mode"]])
    L = len(numel)
    if case["op"] == "consensus":
        s["bounds"] = [0, L // 4, L // 2, 3 * L // 4, L] if L >= 4 else [0, L]
        s["sq"] = torch.zeros((len(s["bounds"]) - 1) * N, dtype=torch.float64, device="cuda")
    elif case["op"] == "average":
        s["average"] = torch.zeros(P, dtype=_TORCH[case["out"]], device="cuda")
    elif case["op"] == "host":
        s["host"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in stacks]
    return s


def _prepare_worker(s, case, numel, gen):
    """One worker of the form with one model per device, its peers' buffers on this device: rows,
    staging buffers with room for a step, its own holding what the peers have sent."""
    N, pop = case["N"], s["pop"]
    s["self"] = me = N // 2
    need = _selected(case, numel)
    capacity = (int(need + 8.0 * math.sqrt(need)) // 64 + 2) * 64
    s["rows"], s["staging"] = [], []
    for role, dtype, scale in ((B.WASH_STACK_PARAMS, case["dtype"], 0.05), (B.WASH_STACK_OPT, case["opt"], 1e-3)):
        if dtype == "none":
            continue
        row = torch.randn(pop.padded_P, device="cuda", generator=gen).mul_(scale).to(_TORCH[dtype])
        B.wash_exchange_bind(pop.ctx, me, role, _CODE[dtype], row, row.numel())
        buffers = torch.zeros((N, capacity), dtype=_TORCH[dtype], device="cuda")
        buffers[me].copy_(torch.randn(capacity, device="cuda", generator=gen).mul_(scale))
        B.wash_exchange_staging(pop.ctx, role, 0, list(buffers), capacity)
        s["rows"].append(row)
        s["staging"].append(buffers)


def run(s):
    case, ctx = s["case"], s["pop"].ctx
    op, step = case["op"], s["step"]
    s["step"] = step + 1
    if op == "shuffle":
        shuffle = B.wash_shuffle_both if case["opt"] != "none" else B.wash_shuffle
        shuffle(ctx, step, s["p"], s["p_layer"], s["seed"], stats=s["stats"])
        return s["stacks"], s["stats"]
    if op == "consensus":
        which = B.WASH_STACK_BOTH if case["opt"] != "none" else B.WASH_STACK_PARAMS
        s["sq"].zero_()
        B.wash_shuffle_consensus(ctx, which, step, s["p"], s["p_layer"], s["seed"], None, s["stats"], s["bounds"], s["sq"])
        return s["stacks"], s["stats"], s["sq"]
    if op == "ema":
        B.papa_ema(ctx, B.WASH_STACK_PARAMS, ALPHA)
        return s["stacks"]
    if op == "papa_all":
        B.papa_all(ctx, B.WASH_STACK_PARAMS)
        return s["stacks"]
    if op == "average":
        B.population_average(ctx, B.WASH_STACK_PARAMS, s["average"], _CODE[case["out"]])
        return s["average"]
    if op == "exchange":
        B.wash_exchange_plan(ctx, step, s["p"], s["p_layer"], s["seed"])
        B.wash_exchange_send(ctx)
        B.wash_exchange_receive(ctx, stats=s["stats"])
        return s["rows"], s["staging"], s["stats"]
    counters = B.wash_step_host(ctx, B.WASH_OP_SHUFFLE, s["host"][0], s["host"][1] if len(s["host"]) > 1 else None, None,
                                step, s["p"], s["p_layer"], s["seed"])
    return s["host"], counters


def work(case):
    """Bytes only (no operator here is a contraction).  A shuffle of the streaming mode reads the
    stacks and writes the selected values; the automatic mode need only touch the selected values."""
    N, numel = case["N"], _numel(case)
    P, selected = float(numel.sum()), _selected(case, numel)
    E, both = _BYTES[case["dtype"]], _BYTES[case["dtype"]] + _BYTES[case["opt"]]
    op = case["op"]
    if op in ("ema", "papa_all"):
        n = 2.0 * N * P * E
    elif op == "average":
        n = N * P * E + P * _BYTES[case["out"]]
    elif op == "exchange":      # values out to the peers, values in from the own buffer: each read and written
        n = 4.0 * selected * (N - 1) / N * both
    elif op == "host":          # every value crosses to the device and back
        n = 2.0 * N * P * both
    elif op == "shuffle" and case["mode"] == "auto":
        n = 2.0 * selected * N * both
    else:
        n = (P + selected) * N * both
    return {"bytes": n, "flops": 0}


def tolerance(case):
    """Everything is defined bit for bit (a shuffle moves bits; the mean's order of summation and
    roundings are part of the interface) except the consensus distances, binary64 sums whose terms
    arrive in any order: on 11M coordinates they differ by 3e-16 from the same sums in torch's order,
    and the difference grows with the root of the length (1e-15 at 2^27 coordinates)."""
    return {"rel": 4e-15} if case["op"] == "consensus" else "exact"
