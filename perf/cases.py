"""The calls that users of the round library make, as timed cases.

A case is a simulated network (graph, worker count, model or bare parameter matrix), an entry point, and the options
a program sets on its handle.  `kind` names the call:

  round     one iteration of Algorithm 1: threshold rule where the backup counts are dynamic, then `Dbw.round`
            (mini-batch gradients, or an external gradient matrix, or none for the consensus-only tail)
  host      the same iteration through `Dbw.round_host`: times and batches in pinned host memory, results read back
  grad      the mini-batch gradients alone (`Dbw.grad`), for callers that bring their own update
  mix       the weighted mix alone (`Dbw.mix`) on a given kept mask
  schedule  the threshold rule and the selection alone: a study of iteration times without a model

Parameters are chained from pass to pass the way a simulation chains its rounds: in place where the library allows it,
else between two buffers, and with parameter tracking on.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2102_06280_b200 as dbw
from workloads import configs

ROUNDS = 16  # rounds of arrival times, backup counts and batches that a state holds; passes walk through them in turn


# ------------------------------------------------------------------------------------------ the cases
def _case(name, kind, workers, graph, degree, d=0, layers="", batch=0, samples=0, precision="fp32", backups="dtur",
          weights="metropolis", order="local_then_mix", gradients=True, times="exp"):
    case = dict(kind=kind, workers=workers, graph=graph, degree=degree, d=d, layers=layers, batch=batch, samples=samples,
                precision=precision, backups=backups, weights=weights, order=order, gradients=gradients, times=times)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # The smallest training round: softmax regression on a ring with one backup worker each.  Latency only.
        _case("ring8_softmax", "round", 8, "ring", 2, layers="784-10", batch=32, samples=600, backups="fixed1"),
        # A small fp32 network, threshold rule before every round; its inputs on the device ...
        _case("reg32_mlp200", "round", 32, "regular", 4, layers="784-200-10", batch=64, samples=2000, times="rates"),
        # ... and in host memory with the results read back every round, as a driver program that logs losses does.
        _case("reg32_mlp200_host", "host", 32, "regular", 4, layers="784-200-10", batch=64, samples=2000, times="rates"),
        # The paper's own experiment: ten workers, the 256-256-10 network, batch 1024; here its baseline that waits for
        # every neighbour.
        _case("er10_2nn_batch1024_full", "round", 10, "er", 4, layers="256-256-256-10", batch=1024, samples=6000, backups="fixed0", times="straggler"),
        # The ordinary tensor-core round: CIFAR-shaped data, dynamic backups, slow workers; and the largest training round.
        _case("er64_mlp512_bf16", "round", 64, "er", 13, layers="3072-512-256-10", batch=128, samples=5000, precision="bf16", times="slow"),
        _case("reg128_mlp1024_bf16", "round", 128, "regular", 8, layers="3072-1024-1024-10", batch=256, samples=5000, precision="bf16", times="lognormal"),
        # Gradients alone, widths and batch that fill no tile: forward and backward through three layers.
        _case("grad_ragged_bf16", "grad", 24, "regular", 4, layers="1000-328-136-10", batch=104, samples=700, precision="bf16", backups="fixed0"),
        # Mixing alone with Eq. 3's order on an odd number of columns: a caller that computes its own gradients.
        _case("mix_reg96_odd", "mix", 96, "regular", 6, d=300_007, backups="uniform", order="mix_then_correct"),
        # Mix-only rounds with many kept neighbours (the paper's weights, and uniform weights at the largest size) ...
        _case("reg1024_deg32_metropolis", "round", 1024, "regular", 32, d=1 << 18, backups="uniform"),
        _case("reg1024_deg32_uniform", "round", 1024, "regular", 32, d=1 << 20, backups="uniform", weights="uniform"),
        # ... and more workers than one SM's shared memory has room for: the mix, and the iteration times alone.
        _case("reg4096_deg8", "round", 4096, "regular", 8, d=1 << 16, backups="uniform"),
        _case("schedule_reg4096", "schedule", 4096, "regular", 8, d=4),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph(rng, workers, most=32):
    if workers >= 8 and workers <= 128 and rng.random() < 0.3:
        return "er", rng.randint(4, min(16, workers // 2))
    degree = 2 * rng.randint(1, max(1, min(most, workers // 2) // 2))
    return ("ring", 2) if degree == 2 else ("regular", degree)


def draw(rng):
    kind = rng.choice(["round", "round", "round", "mixround", "mixround", "mix", "grad", "host", "schedule"])
    backups = rng.choice(["dtur", "dtur", "uniform", "fixed0", "fixed1"])
    weights = rng.choice(["metropolis", "metropolis", "uniform"])
    order = rng.choice(["local_then_mix", "local_then_mix", "mix_then_correct"])
    times = rng.choice(["exp", "rates", "slow", "straggler", "lognormal"])
    if kind == "schedule":
        workers = _spread(rng, 64, 4096)
        graph, degree = _graph(rng, workers, 16)
        return _case("", kind, workers, graph, degree, d=4, times=times)
    if kind in ("mix", "mixround"):
        workers = _spread(rng, 8, 4096)
        graph, degree = _graph(rng, workers, 32 if workers <= 1024 else 8)
        most = (1 << 28) if workers <= 1024 else (1 << 27)
        d = _spread(rng, 1 << 10, most // workers)
        return _case("", "mix" if kind == "mix" else "round", workers, graph, degree, d=d, backups=backups, weights=weights, order=order,
                     gradients=rng.random() < 0.8, times=times)
    if rng.random() < 0.5:  # fp32: any widths
        dims = [rng.choice([64, 256, 784, rng.randint(30, 900)])] + [_spread(rng, 16, 320) for _ in range(rng.randint(0, 2))] + [10]
        batch, workers, precision = _spread(rng, 16, 512), _spread(rng, 4, 64), "fp32"
        flops = 6.0 * batch * sum(a * b for a, b in zip(dims, dims[1:]))
        workers = max(4, min(workers, int(2e10 / flops)))
    else:  # tensor cores: widths and batch are multiples of eight
        dims = [rng.choice([256, 784, 1024, 3072])] + [8 * _spread(rng, 8, 128) for _ in range(rng.randint(1, 2))] + [10]
        batch, workers, precision = 8 * rng.randint(4, 40), _spread(rng, 4, 128), "bf16"
    graph, degree = _graph(rng, workers, 8)
    return _case("", kind, workers, graph, degree, layers="-".join(map(str, dims)), batch=batch, samples=3 * batch + rng.randint(0, 500),
                 precision=precision, backups=backups, weights=weights, order=order, times=times)


# ------------------------------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=4)
def _csr(graph, workers, degree):
    if graph == "ring":
        return configs.ring(workers)
    if graph == "regular":
        return configs.random_regular(workers, degree, 5001)
    return configs.erdos_renyi_connected(workers, degree / (workers - 1), 3)


def _arrival_times(kind, workers, gen):
    t = 1.0 + torch.empty(ROUNDS, workers, dtype=torch.float64, device="cuda").exponential_(1.0, generator=gen)
    if kind == "rates":        # worker j's exponential part has a rate from U[0.5, 2]
        t = 1.0 + (t - 1.0) / (0.5 + 1.5 * torch.rand(workers, dtype=torch.float64, device="cuda", generator=gen))
    elif kind == "slow":       # one worker in ten is five times as slow
        slow = torch.randperm(workers, device="cuda", generator=gen)[: round(0.1 * workers)]
        t[:, slow] = 1.0 + (t[:, slow] - 1.0) * 5.0
    elif kind == "straggler":  # one random worker per round takes five times as long
        late = torch.randint(0, workers, (ROUNDS,), device="cuda", generator=gen)
        t[torch.arange(ROUNDS, device="cuda"), late] *= 5.0
    elif kind == "lognormal":
        t = torch.randn(ROUNDS, workers, dtype=torch.float64, device="cuda", generator=gen).exp()
    return t


def _backups(kind, deg, gen):
    if kind == "uniform":      # up to a quarter of the degree
        b = torch.floor(torch.rand(ROUNDS, deg.numel(), device="cuda", generator=gen) * (deg // 4 + 1)).int()
    else:
        b = torch.full((ROUNDS, deg.numel()), 1 if kind == "fixed1" else 0, dtype=torch.int32, device="cuda")
    return torch.minimum(b, deg.int())


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, kind = case["workers"], case["kind"]
    rowptr, col = _csr(case["graph"], n, case["degree"])
    flags = ((dbw.WEIGHT_UNIFORM if case["weights"] == "uniform" else 0) | (dbw.GEMM_BF16 if case["precision"] == "bf16" else 0)
             | (dbw.ORDER_MIX_THEN_CORRECT if case["order"] == "mix_then_correct" else 0))
    st = {"kind": kind, "dynamic": case["backups"] == "dtur", "k": 0, "X": None, "G": None, "idx": None, "loss": None}
    if case["layers"]:
        dims = [int(v) for v in case["layers"].split("-")]
        batch, samples = case["batch"], case["samples"]
        m = dbw.model_layout(dims, batch)
        h = dbw.Dbw(rowptr, col, d=m.d, model=m, flags=flags)
        # Gaussian mixture with ten class means; the MNIST-shaped features lie in [0, 1]
        noise, clip = (0.5, True) if dims[0] < 1000 else (0.3, False)
        means = torch.randn(dims[-1], dims[0], device="cuda", generator=gen)
        labels = torch.randint(0, dims[-1], (n, samples), dtype=torch.int32, device="cuda", generator=gen)
        feat = torch.empty(n, samples, dims[0], device="cuda")
        for i in range(n):
            feat[i].normal_(0.0, noise, generator=gen).add_(means[labels[i].long()])
            if clip:
                feat[i].clamp_(0.0, 1.0)
        h.set_dataset(feat, labels, samples)
        X = torch.zeros(n, m.ld, device="cuda")
        for l, (a, b) in enumerate(zip(dims, dims[1:])):
            X[:, m.w_off[l]: m.w_off[l] + a * b].normal_(0.0, math.sqrt(2.0 / a), generator=gen)
        idx = torch.stack([torch.rand(n, samples, device="cuda", generator=gen).argsort(dim=1)[:, :batch] for _ in range(ROUNDS)]).int()
        st.update(idx=list(idx.unbind()), loss=torch.zeros(n, device="cuda"))
        if kind == "grad":
            st["G"] = torch.zeros(n, m.ld, device="cuda")
    else:
        h = dbw.Dbw(rowptr, col, d=case["d"], flags=flags)
        if kind != "schedule":
            X = torch.zeros(n, h.ld, device="cuda")
            X[:, : case["d"]].normal_(0.0, 1.0, generator=gen)
            if case["gradients"]:
                st["G"] = torch.zeros(n, h.ld, device="cuda")
                st["G"][:, : case["d"]].normal_(0.0, 0.01, generator=gen)
    if kind != "schedule":
        st.update(X=X, X_out=X if kind == "grad" or h.mix_in_place_ok() else torch.zeros_like(X))
        h.set_param_tracking(kind in ("round", "host") and bool(case["layers"]))
    deg = torch.from_numpy(np.diff(rowptr)).cuda()
    t, b = _arrival_times(case["times"], n, gen), _backups(case["backups"], deg, gen)
    st.update(h=h, t=list(t.unbind()), b=list(b.unbind()), b_dyn=torch.zeros(n, dtype=torch.int32, device="cuda"),
              kept=torch.zeros(len(col), dtype=torch.uint8, device="cuda"), T_worker=torch.zeros(n, dtype=torch.float64, device="cuda"),
              T_round=torch.zeros(1, dtype=torch.float64, device="cuda"))
    if kind == "mix":          # the masks of the rounds to come
        st["masks"] = [torch.zeros_like(st["kept"]) for _ in range(ROUNDS)]
        for k in range(ROUNDS):
            if st["dynamic"]:
                h.update_backups(st["t"][k], st["b"][k])
            h.select(st["t"][k], st["b"][k], st["masks"][k])
    if kind == "host":
        pin = lambda x: x.cpu().pin_memory()  # noqa: E731
        st.update(t=list(pin(t).unbind()), b=list(pin(b).unbind()), idx=list(pin(idx).unbind()), b_dyn=pin(st["b_dyn"]), kept=pin(st["kept"]),
                  T_worker=pin(st["T_worker"]), T_round=pin(st["T_round"]), loss=pin(st["loss"]))
    return st


# ------------------------------------------------------------------------------------------ one pass
def run(st):
    h, k, kind = st["h"], st["k"] % ROUNDS, st["kind"]
    st["k"] += 1
    t, b, lr = st["t"][k], st["b"][k], 0.05
    if kind == "grad":
        h.grad(st["X"], st["idx"][k], st["G"], st["loss"])
        return {"G": st["G"], "loss": st["loss"]}
    X, out = st["X"], st.get("X_out")
    if kind == "mix":
        h.mix(X, st["G"], st["masks"][k], b, lr, out)
        st["X"], st["X_out"] = out, X
        return {"X": out}
    if kind == "host":
        h.round_host(X, t, None if st["dynamic"] else b, lr, out, h_batch_idx=st["idx"][k], h_kept=st["kept"], h_T_worker=st["T_worker"],
                     h_T_round=st["T_round"], h_loss=st["loss"], h_b_out=st["b_dyn"] if st["dynamic"] else None)
        torch.cuda.current_stream().synchronize()  # the program reads the round's results
    else:
        if st["dynamic"]:
            b = st["b_dyn"]
            h.update_backups(t, b)
        if kind == "schedule":
            h.select(t, b, st["kept"], st["T_worker"], T_round=st["T_round"])
            return {"b": b, "kept": st["kept"], "T_worker": st["T_worker"], "T_round": st["T_round"]}
        h.round(X, t, b, lr, out, st["kept"], batch_idx=None if st["idx"] is None else st["idx"][k], G_ext=st["G"],
                T_worker=st["T_worker"], T_round=st["T_round"], loss=st["loss"])
    st["X"], st["X_out"] = out, X
    got = {"X": out, "b": st["b_dyn"] if st["dynamic"] else b, "kept": st["kept"], "T_worker": st["T_worker"], "T_round": st["T_round"]}
    if st["loss"] is not None:
        got["loss"] = st["loss"]
    return got


# ------------------------------------------------------------------------------------------ what a pass cannot do without
def work(case):
    n = case["workers"]
    nnz = len(_csr(case["graph"], n, case["degree"])[1])
    # times in and out, backup counts, graph and mask: read or written once
    plan = n * (8 + 8 + 4 + 4) + nnz * (4 + 1)
    if case["kind"] == "schedule":
        return {"bytes": plan, "flops": 0}
    if not case["layers"]:
        kept = nnz / n * {"dtur": 0.25, "uniform": 0.875}.get(case["backups"], 1.0)
        return {"bytes": (12.0 if case["gradients"] else 8.0) * n * case["d"] + plan, "flops": 2.0 * n * case["d"] * (kept + 2.0)}
    dims = [int(v) for v in case["layers"].split("-")]
    pairs = [a * b for a, b in zip(dims, dims[1:])]
    d = sum(pairs) + sum(dims[1:])
    # parameters in, parameters (or gradients) out, the mini-batch's features, labels and indices
    size = 8.0 * n * d + n * case["batch"] * (4.0 * dims[0] + 8.0) + plan
    return {"bytes": size, "flops": n * case["batch"] * (6.0 * sum(pairs) - 2.0 * pairs[0])}


def tolerance(case):
    """About four times the largest difference seen against a recomputation of the pass in double precision (with bf16:
    rounded where the library rounds), over the listed cases and a hundred drawn ones.

    Sums in fp32 alone: 1.9e-7 (largest element 2.1e-6 of the rms).  A model adds ReLU units whose pre-activation is zero
    up to rounding and may land on either side, which moves a row of a weight gradient by one sample's share: gradients
    3.8e-4 (largest element 0.033 of the rms) in fp32 and 7.2e-4 (0.29) with bf16 operands, parameters after the step 4.1e-6
    (1.5e-4) and 2.1e-5 (8.8e-3).  Masks, backup counts and times are compared without an allowance.
    """
    if case["kind"] == "schedule":
        return "exact"
    if not case["layers"]:
        return {"rel": 1e-6, "max": 1e-5}
    if case["kind"] == "grad":
        return {"rel": 3e-3, "max": 0.9} if case["precision"] == "bf16" else {"rel": 1.5e-3, "max": 0.13}
    return {"rel": 8e-5, "max": 0.035} if case["precision"] == "bf16" else {"rel": 1.6e-5, "max": 6e-4}
