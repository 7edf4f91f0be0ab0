"""Performance cases of the DAT outer-minimisation path: what users of this package run, through its public calls.

A case is a dict of plain values:
    call      which public entry points one pass takes (see run())
    model     a workload of synth.config() whose tensor shapes are used, or "flat": `layers` sizes, log-uniform,
              odd ones among them, that sum to `total`
    M, bits, rng_bits, scale, dist, seed_sizes, ranks
              workers, code width b (32: no quantisation), resolution of the uniform number, "shared" or
              "per_worker" norms, distribution of the gradients, seed of the flat sizes, ranks of a sharded step

Calls:
    step        dat_step: Steps 7, 9 and 12 on M gradient buffers of one GPU
    lamb        dat_step_lamb: the same with LAMB as the outer-minimisation oracle (the ImageNet setting)
    two_sided   dat_step_two_sided: the server quantizes the aggregate once more
    message     dat_quantize -> dat_aggregate -> dat_lalr_step: the packed messages are wanted as well
    server      dat_aggregate -> dat_requantize -> dat_lamb_step: a parameter server that has received M messages
    rank        one rank's device work in a step sharded over `ranks` GPUs (ShardedStep, "pull" form)
    host        dat_step_host: parameters, momentum and gradients live in pinned host memory

Every pass is the next training step: the step counter (the key of the random streams) advances, parameters and
momentum carry over.
"""
import weakref

import numpy as np
import torch

from paper_2206_06257_b200 import api, sharded, synth

HP = (0.1, 0.9, 5e-4, 0.0, 10.0)                       # lr, momentum, weight decay, c_l, c_u: the workloads' own
LAMB_HP = (0.1, 0.9, 0.999, 1e-6, 1e-4, 0.0, 10.0)     # the ImageNet settings of bench.py


def _case(name, call, model, M, bits, rng_bits=16, scale="shared", dist="normal", total=0, layers=0, seed_sizes=0, ranks=0):
    c = dict(call=call, model=model, M=M, bits=bits, rng_bits=rng_bits, scale=scale, dist=dist, total=total, layers=layers,
             seed_sizes=seed_sizes, ranks=ranks)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model (235 thousand parameters): launches, synchronisation and host work are what it costs
        _case("step_tiny_mlp", "step", "tiny_mlp", M=4, bits=8),
        # CIFAR-10 training: the ordinary small convolutional network, 6 workers
        _case("step_resnet18", "step", "resnet18", M=6, bits=8),
        # ImageNet training, the configuration that bench.py measures by default
        _case("step_resnet50", "step", "resnet50", M=8, bits=8),
        # ImageNet in the large-batch regime: many workers, few bits, heavy-tailed gradients, a zero layer
        _case("step_resnet50_m32", "step", "resnet50_m32", M=32, bits=4, dist="student_t3"),
        # the largest: a billion parameters in 400 tensors of 64 to 16M elements, sizes not multiples of 4
        _case("step_flat1b", "step", "flat1b", M=8, bits=8),
        # the unquantised baseline runs (32 bits) that every comparison of the method needs
        _case("step_resnet50_b32", "step", "resnet50", M=8, bits=32),
        # LAMB as the outer-minimisation oracle, with its second moment
        _case("lamb_resnet50", "lamb", "resnet50", M=8, bits=8),
        # two-sided quantisation with the equations as written (every worker's own norm), 23-bit uniform numbers, odd sizes
        _case("two_sided_flat_small", "two_sided", "flat_small", M=3, bits=4, rng_bits=23, scale="per_worker"),
        # encode, decode and update as separate calls: the messages themselves are kept (sent, logged, checked)
        _case("message_resnet50", "message", "resnet50", M=8, bits=8),
        # a parameter server: decodes 16 workers' 4-bit messages, re-encodes the aggregate, updates with LAMB
        _case("server_resnet18", "server", "resnet18", M=16, bits=4),
        # one of eight GPUs of a sharded ImageNet step: encodes its own worker for every owner, decodes and updates its range
        _case("rank_resnet50", "rank", "resnet50", M=8, bits=8, ranks=8),
        # state and gradients in pinned host memory (an offloaded optimizer): the copies are part of the call
        _case("host_resnet18", "host", "resnet18", M=6, bits=8),
    ]


CALLS = ["step"] * 6 + ["lamb"] * 2 + ["two_sided"] * 2 + ["message"] * 3 + ["server"] + ["rank"] * 2 + ["host"]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    call = rng.choice(CALLS)
    bits = rng.choice([1, 2, 2, 4, 4, 4, 8, 8, 8, 8, 16])
    if call == "step" and rng.random() < 0.15:
        bits = 32
    ranks = rng.choice([2, 4, 8]) if call == "rank" else 0
    M = ranks * rng.choice([1, 1, 2, 4]) if call == "rank" else _log_int(rng, 1, 64)
    scale = "per_worker" if call in ("step", "lamb", "two_sided", "message", "server") and bits != 32 and rng.random() < 0.2 else "shared"
    rng_bits = 23 if rng.random() < 0.25 else 16
    dist = "student_t3" if rng.random() < 0.25 else "normal"
    model = rng.choice(["flat", "flat", "flat", "tiny_mlp", "resnet18", "resnet50"])
    room = {"host": 1.5e9}.get(call, 12e9)              # bytes of one state, about
    total = layers = seed_sizes = 0
    if model == "flat":
        total = _log_int(rng, 20_000, int(min(4e8, room / (4 * (M + 6)))))
        layers = _log_int(rng, max(4, ranks, total // 8_000_000), max(8, min(400, total // 500)))
        seed_sizes = rng.randrange(1 << 20)
    elif 4 * (M + 6) * synth.config(model).d > room:
        model = "tiny_mlp"
    return _case("", call, model, M=M, bits=bits, rng_bits=rng_bits, scale=scale, dist=dist, total=total, layers=layers,
                 seed_sizes=seed_sizes, ranks=min(ranks, 2) if model == "tiny_mlp" else ranks)


def _config(case, seed=0):
    if case["model"] == "flat":
        t = synth.flat_tensors(total=case["total"], num_layers=case["layers"], lo=5, hi=16 * 1024 * 1024, seed=case["seed_sizes"])
        cfg = synth.Config("flat", t, M=1, bits=8, log10_sigma=(-5.0, -1.0), theta_init="normal:0.02", mom_std=1e-3)
    else:
        cfg = synth.config(case["model"])
    cfg.M, cfg.bits, cfg.rng_bits, cfg.grad_dist, cfg.seed = case["M"], case["bits"], case["rng_bits"], case["dist"], int(seed)
    return cfg


class State:
    """What a training program holds: a plan, the model's state, the step counter."""

    def __init__(self, **kw):
        self.__dict__.update(kw)


def _plan(state, cfg, case):
    state.plan = api.dat_plan_create(cfg.offsets, cfg.M, cfg.bits, rng_bits=cfg.rng_bits,
                                     scale_mode=api.DAT_SCALE_PER_WORKER if case["scale"] == "per_worker" else api.DAT_SCALE_SHARED_MAX)
    weakref.finalize(state, api.dat_plan_destroy, state.plan)


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    cfg = _config(case, seed)
    dev = torch.device("cuda")
    s = State(call=case["call"], seed=int(seed), step=0)
    s.theta, s.mom = synth.make_params(cfg, device=dev)
    grads = synth.make_grads(cfg, 0, device=dev)
    if s.call == "rank":
        _prepare_rank(s, cfg, case, grads)
        return s
    _plan(s, cfg, case)
    if s.call == "host":
        s.theta, s.mom, s.grads = s.theta.cpu().pin_memory(), s.mom.cpu().pin_memory(), [g.cpu().pin_memory() for g in grads]
        return s
    s.grads = grads
    if s.call in ("lamb", "server"):
        s.var = torch.rand(cfg.d, generator=torch.Generator(device=dev).manual_seed(int(seed) + 77), device=dev) * 1e-6
    if s.call in ("two_sided", "message", "server"):
        s.g_hat = torch.empty(cfg.d, device=dev)
    if s.call in ("message", "server"):
        lb, sb, ns, _ = api.dat_plan_sizes(s.plan)
        s.levels, s.signs, s.scales = _bytes(cfg.M * lb), _bytes(cfg.M * sb), torch.empty(ns, device=dev)
    if s.call == "server":                              # the messages as they have arrived
        api.dat_quantize(s.plan, s.grads, s.seed, 0, s.levels, s.signs, s.scales)
        s.grads = None
        s.out_levels, s.out_signs, s.out_scales = _bytes(lb), _bytes(sb), torch.empty(cfg.h, device=dev)
    return s


def _prepare_rank(s, cfg, case, grads):
    """Rank 0 of `ranks`: its own workers' gradients, and for its range the planes that the other ranks have published."""
    G, M_loc = case["ranks"], cfg.M // case["ranks"]
    ops = sharded.CudaOps(api, cfg.offsets, cfg.M, M_loc, 0, G, cfg.bits, cfg.rng_bits)
    weakref.finalize(s, ops.close)
    s.sharded = sharded.ShardedStep(ops, cfg.offsets, cfg.M, 0, G)
    own = s.sharded.own
    s.grads = grads[:M_loc]
    s.nu_others = torch.zeros(cfg.h, device=s.theta.device)
    for r in range(1, G):
        other = sharded.CudaOps(api, cfg.offsets, cfg.M, M_loc, r, G, cfg.bits, cfg.rng_bits)
        s.nu_others = torch.maximum(s.nu_others, other.worker_norms(grads[r * M_loc:(r + 1) * M_loc]).max(dim=0).values)
        other.close()
    nu = torch.maximum(s.sharded.local_norms(s.grads), s.nu_others)
    s.others = []
    for r in range(1, G):
        other = sharded.CudaOps(api, cfg.offsets, cfg.M, M_loc, r, G, cfg.bits, cfg.rng_bits)
        s.others.append(other.quantize_range(0, own, grads[r * M_loc:(r + 1) * M_loc], own.scales(nu), s.seed, 0))
        other.close()
    s.mom = s.mom[own.a8:own.b].clone()
    s.sharded.quantize(nu, s.grads, s.seed, 0)          # the rank's plans exist from the first step on
    s.sharded.ops.plane_bytes(own)


def run(s):
    step, s.step = s.step, s.step + 1
    if s.call == "step":
        api.dat_step(s.plan, s.theta, s.mom, s.grads, s.seed, step, HP)
        return s.theta, s.mom
    if s.call == "lamb":
        api.dat_step_lamb(s.plan, s.theta, s.mom, s.var, s.grads, s.seed, step, LAMB_HP, step + 1)
        return s.theta, s.mom, s.var
    if s.call == "two_sided":
        api.dat_step_two_sided(s.plan, s.theta, s.mom, s.grads, s.seed, step, HP, s.g_hat)
        return s.theta, s.mom, s.g_hat
    if s.call == "message":
        api.dat_quantize(s.plan, s.grads, s.seed, step, s.levels, s.signs, s.scales)
        api.dat_aggregate(s.plan, s.levels, s.signs, s.scales, None, s.g_hat)
        api.dat_lalr_step(s.plan, s.theta, s.mom, s.g_hat, HP)
        return s.levels, s.signs, s.scales, s.g_hat, s.theta, s.mom
    if s.call == "server":
        api.dat_aggregate(s.plan, s.levels, s.signs, s.scales, None, s.g_hat)
        api.dat_requantize(s.plan, s.g_hat, s.seed, step, s.out_levels, s.out_signs, s.out_scales)
        api.dat_lamb_step(s.plan, s.theta, s.mom, s.var, s.g_hat, LAMB_HP, step + 1)
        return s.out_levels, s.out_signs, s.out_scales, s.g_hat, s.theta, s.mom, s.var
    if s.call == "rank":
        nu = torch.maximum(s.sharded.local_norms(s.grads), s.nu_others)      # stands for the all-reduce of h floats
        mine = s.sharded.quantize(nu, s.grads, s.seed, step)
        s.sharded.update_pull(nu, [mine[0]] + s.others, s.theta, s.mom, HP)
        return nu, mine, s.theta, s.mom
    api.dat_step_host(s.plan, s.theta, s.mom, s.grads, s.seed, step, HP)
    return s.theta, s.mom


def work(case):
    """Each input read once, each output written once.  Operations: a square per worker-element for the norm, about
    five for a level and its place in the sum; a dozen per element for the update and its norms."""
    cfg = _config(case)
    d, M, b = cfg.d, case["M"], case["bits"]
    plane = 0.0 if b == 32 else (b + 1) / 8.0
    flops = M * d * (1 if b == 32 else 7) + 12 * d
    if case["call"] == "rank":
        G, own = case["ranks"], d / case["ranks"]
        return {"bytes": 4 * d * M / G + plane * d * M / G + plane * own * (M - M / G) + 16 * own, "flops": 7 * d * M / G + own * (M + 12)}
    n = {"step": 4 * M + 16, "host": 4 * M + 16, "lamb": 4 * M + 24, "two_sided": 4 * M + 20,
         "message": 4 * M + plane * M + 20, "server": plane * M + plane + 28}[case["call"]]
    return {"bytes": n * d, "flops": d * (M + 24) if case["call"] == "server" else flops}


def tolerance(case):
    """Codes and planes are whole numbers drawn from fixed random streams and stay as they are.  The norms are 64-bit
    sums of exact squares, rounded once; the rest is single precision with the operations in a stated order."""
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
