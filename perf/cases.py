"""The work that programs give this library, as cases that can be timed and compared.

Two kinds of program use it.  A trainer holds a HierAvg handle: it runs whole rounds
(``round``, or ``round_host`` when the data set stays in host memory), or writes its own
loop of ``step`` and ``local_average``.  A trainer with an optimiser of its own only
averages its replica matrix (``local_average_buffer`` and its two siblings).

A case is a dict of plain values:
  kind       round | round_host | loop | local | global | local_global
  handle:    dims ("3072-512-10"), precision, P, S, K1, K2, B, N, lr, G (local steps per
             global average, 0: K1 * K2); ``loop`` runs K1 steps and a local average
  averages:  P, S, D, ld (row stride in floats; D: a plain contiguous matrix)
Notation: P learners, clusters of S, K1 local steps per local average, K2 local averages
per global average, B samples per learner and step, N samples per learner.
"""
from __future__ import annotations

import math

import torch

from paper_1903_05133_gb300 import hier_avg
from paper_1903_05133_gb300.hier_avg import HierAvg

AVERAGES = ("local", "global", "local_global")


def _handle(name, kind, dims, precision, P, S, K1, K2, B, N, lr, G=0):
    return {"name": name, "kind": kind, "dims": dims, "precision": precision, "P": P, "S": S,
            "K1": K1, "K2": K2, "B": B, "N": N, "lr": lr, "G": G}


def _average(name, kind, P, S, D, ld=0):
    return {"name": name, "kind": kind, "P": P, "S": S, "D": D, "ld": ld or D}


def listed():
    return [
        # Softmax regression in full fp32 precision, the smallest model: a few
        # microseconds of arithmetic per step, so launches and latency are its cost.
        _handle("softmax_round_fp32", "round", "3072-10", "fp32", 4, 2, 2, 2, 16, 512, 0.05),
        # A small net with odd widths and an odd batch in fp32 (tabular data).
        _handle("odd_mlp_round_fp32", "round", "100-37-10", "fp32", 4, 2, 2, 2, 7, 40, 0.05),
        # The CIFAR-shaped net in fp32: what a user runs who may not round operands.
        _handle("cifar_mlp_round_fp32", "round", "3072-512-10", "fp32", 16, 4, 4, 2, 32, 1024, 0.05),
        # The same net with bf16 operands: parameters that fit in L2, ordinary size.
        _handle("cifar_mlp_round_bf16", "round", "3072-512-10", "bf16", 16, 4, 4, 4, 32, 1024, 0.05),
        # The same round fed from pinned host memory, loss read back: the end-to-end call.
        # (The device data set holds the previous copy of the same rows.)
        _handle("cifar_mlp_round_host_bf16", "round_host", "3072-512-10", "bf16", 16, 4, 4, 4, 32, 1024,
                0.05),
        # A wider CIFAR-shaped net on 64 learners, 64-row batches: parameters (2.7 GB)
        # stream from HBM in every step.
        _handle("cifar_wide_round_bf16", "round", "3072-2048-2048-10", "bf16", 64, 8, 8, 4, 64, 2048, 0.02),
        # The ImageNet-shaped net (71M parameters per learner): the largest workload.
        _handle("imagenet_mlp_round_bf16", "round", "12288-4096-4096-1000", "bf16", 32, 8, 4, 8, 32, 1024,
                0.01),
        # Hundreds of classes and a small batch: logits beyond one output tile.
        _handle("classes300_round_bf16", "round", "1024-1152-300", "bf16", 32, 8, 2, 2, 16, 64, 0.05),
        # A program's own loop of single steps and local averages on a ragged net; the
        # batch does not divide the data set, so some batches wrap around its end.
        _handle("ragged_loop_bf16", "loop", "264-136-200-13", "bf16", 6, 3, 4, 1, 20, 50, 0.05),
        # Local average of 128 replicas of an 11.2M-parameter model (ResNet-18 size).
        _average("local_avg_11M", "local", 128, 8, 11_200_000),
        # Global average of 128 replicas of a 1M-parameter model: short rows.
        _average("global_avg_1M", "global", 128, 1, 1_000_000),
        # Replicas as a user's own contiguous [P, D] matrix: the learner count is no power
        # of two and the row length is odd, so rows do not start on 16-byte boundaries.
        _average("odd_local_global_avg", "local_global", 12, 6, 1_000_003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _divisor(rng, n):
    return rng.choice([d for d in range(1, n + 1) if n % d == 0])


def _weights(dims):
    return sum(i * o for i, o in zip(dims[:-1], dims[1:]))


def _draw_average(rng):
    kind = rng.choice(AVERAGES)
    P = rng.choice([2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 128])
    D = min(_log_int(rng, 1000, 32_000_000), 1_400_000_000 // P)
    ld = rng.choice([D, D, (D + 63) // 64 * 64])
    return {"kind": kind, "P": P, "S": 1 if kind == "global" else _divisor(rng, P), "D": D, "ld": ld}


def _draw_handle(rng):
    precision = rng.choice(["fp32", "bf16", "bf16"])
    bf16 = precision == "bf16"
    step = 8 if bf16 else 1                      # bf16 takes input widths that are multiples of 8
    classes = rng.choice([10, _log_int(rng, 2, 1000)])
    n_hidden = rng.choice([0, 1, 1, 2, 2])
    while True:
        width = lambda lo, hi: max(step, _log_int(rng, lo, hi) // step * step)
        dims = [rng.choice([784, 3072, width(64, 12288)])]
        dims += [rng.choice([512, width(32, 4096)]) for _ in range(n_hidden)]
        dims.append(classes)
        P = rng.choice([1, 2, 4, 6, 8, 12, 16, 24, 32, 64])
        B = rng.choice([16, 32, 64, rng.randint(1, 64)])
        K1, K2 = rng.randint(1, 8), rng.randint(1, 4)
        G = rng.choice([0, 0, 0, rng.randint(1, K1 * K2 + 3)])
        steps = G or K1 * K2
        w = P * _weights(dims)
        # no drawn case costs more than the largest listed one
        if w <= 600_000_000 and (w * steps <= 12_000_000_000 if bf16 else w * B * steps <= 12_000_000_000):
            break
    kind = rng.choice(["round", "round", "round", "loop", "round_host"])
    N = max(B, rng.choice([B * steps, B * steps, B * max(1, steps // 2) + rng.randint(0, B)]))
    most = 256_000_000 if kind == "round_host" else 1_000_000_000   # bytes of samples
    N = min(N, max(B, most // (P * dims[0] * (2 if bf16 else 4))))
    return {"kind": kind, "dims": "-".join(map(str, dims)), "precision": precision, "P": P,
            "S": _divisor(rng, P), "K1": K1, "K2": K2, "B": B, "N": N, "lr": 0.02, "G": G}


def draw(rng):
    return _draw_average(rng) if rng.random() < 0.35 else _draw_handle(rng)


# ------------------------------------------------------------------ inputs
def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _replicas(case, seed):
    """[P, D] fp32 replicas of one model that have drifted apart, row stride ld."""
    g = _generator(seed)
    P, D = case["P"], case["D"]
    w = torch.zeros(P, case["ld"], device="cuda")[:, :D]
    base = torch.randn(D, generator=g, device="cuda") * 0.05
    for j in range(P):
        w[j] = torch.randn(D, generator=g, device="cuda").mul_(0.01).add_(base)
    return w


def _training_inputs(case, seed):
    """(layers, X, y): He-normal weights and zero biases shared by all learners; samples
    of a Gaussian mixture with one mean per class (CIFAR- or ImageNet-shaped), per learner."""
    g = _generator(seed)
    dims, P, N = _dims(case), case["P"], case["N"]
    layers = [(torch.randn(o, i, generator=g, device="cuda").mul_(math.sqrt(2.0 / i)),
               torch.zeros(o, device="cuda")) for i, o in zip(dims[:-1], dims[1:])]
    mu = torch.randn(dims[-1], dims[0], generator=g, device="cuda").mul_(0.1)
    y = torch.randint(0, dims[-1], (P, N), generator=g, device="cuda", dtype=torch.int32)
    X = torch.empty(P, N, dims[0], device="cuda",
                    dtype=torch.bfloat16 if case["precision"] == "bf16" else torch.float32)
    for j in range(P):
        X[j] = torch.randn(N, dims[0], generator=g, device="cuda").add_(mu[y[j].long()])
    return layers, X, y


def prepare(case, seed):
    if case["kind"] in AVERAGES:
        return {"case": case, "w": _replicas(case, seed)}
    layers, X, y = _training_inputs(case, seed)
    ha = HierAvg(case["P"], case["S"], case["K1"], case["K2"], case["lr"], case["B"], _dims(case),
                 case["precision"])
    state = {"case": case, "ha": ha}
    if case["kind"] == "round_host":
        state["X"], state["y"] = X.cpu().pin_memory(), y.cpu().pin_memory()
        state["loss"] = torch.empty(case["P"], pin_memory=True)
    ha.bind(ha.pack(layers), X, y)
    if case["G"]:
        ha.set_global_steps(case["G"])
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "local":
        hier_avg.local_average_buffer(state["w"], case["S"])
    elif kind == "global":
        hier_avg.global_average_buffer(state["w"])
    elif kind == "local_global":
        hier_avg.local_global_average_buffer(state["w"], case["S"])
    if kind in AVERAGES:
        return state["w"]
    ha = state["ha"]
    if kind == "round":
        ha.round()
    elif kind == "round_host":
        ha.round_host(state["X"], state["y"], state["loss"])
        return {"params": ha.params, "loss": state["loss"]}
    else:
        for _ in range(case["K1"]):
            ha.step()
        ha.local_average()
    return {"params": ha.params}


# ------------------------------------------------------------------ what is to be expected
def _steps(case):
    return case["K1"] if case["kind"] == "loop" else case["G"] or case["K1"] * case["K2"]


def work(case):
    P = case["P"]
    if case["kind"] in AVERAGES:
        n = P * case["D"]                       # every value read once and written once
        return {"bytes": 8 * n, "flops": n}
    dims, rows = _dims(case), P * case["B"] * _steps(case)
    D = _weights(dims) + sum(dims[1:])
    # parameters in and out once, every sample and label read once; a local step has a
    # forward and a dW product per layer, and a dX product for every layer but the first
    return {"bytes": 8 * P * D + rows * (dims[0] * (2 if case["precision"] == "bf16" else 4) + 4),
            "flops": 2 * rows * (3 * _weights(dims) - dims[0] * dims[1])}


def tolerance(case):
    if case["kind"] in AVERAGES:
        return "exact"      # the library promises one summation order, bit for bit
    if case["precision"] == "fp32":
        # Measured against 64 bits: 1.2e-7 at 3072-10.  With hidden layers 5e-8 (100-37-10)
        # until a pre-activation within rounding of zero takes the other ReLU branch (a few
        # in the millions of a round), which moves one row: 2.3e-5 at 3072-512-10, 16 steps.
        return {"rel": 1e-6 if len(_dims(case)) == 2 else 1e-4}
    # bf16 operands against 64 bits without rounding, measured: 5.5e-4 at 264-136-200-13,
    # 5.1e-4 at 3072-512-10 (16 steps; its loss 3.2e-4), 9e-5 at 1024-1152-300.
    return {"rel": 2e-3}


def _softmax_ce(Z, y):
    """dZ (mean over the batch) and the mean loss of logits [P, B, C], labels [P, B]."""
    logp = torch.log_softmax(Z, dim=2)
    hot = torch.nn.functional.one_hot(y, Z.shape[2]).to(Z.dtype)
    return (logp.exp() - hot) / Z.shape[1], -(logp * hot).sum(2).mean(1)


def _group_mean(w, n):
    P = w.shape[0]
    return w.reshape(P // n, n, *w.shape[1:]).mean(1).repeat_interleave(n, dim=0)


def exact(case, seed):
    if case["kind"] in AVERAGES:
        w = _replicas(case, seed)
        out = torch.empty(w.shape, device="cuda", dtype=torch.float64)
        for c in range(0, w.shape[1], 1 << 20):
            v = w[:, c:c + (1 << 20)].double()
            if case["kind"] != "global":
                v = _group_mean(v, case["S"])
            out[:, c:c + (1 << 20)] = v if case["kind"] == "local" else _group_mean(v, case["P"])
        return out
    if work(case)["flops"] > 8e12:
        return None                              # over 20 seconds in 64 bits
    layers, X, y = _training_inputs(case, seed)
    P, B, N, dims, steps = case["P"], case["B"], case["N"], _dims(case), _steps(case)
    Ws = [W.double().expand(P, *W.shape).contiguous() for W, _ in layers]
    bs = [b.double().expand(P, *b.shape).contiguous() for _, b in layers]
    L, lr, loss = len(Ws), float(torch.tensor(case["lr"], dtype=torch.float32)), None
    for t in range(steps):
        rows = (torch.arange(B, device="cuda") + t * B) % N
        H = [X[:, rows].double()]
        for l in range(L):
            Z = torch.baddbmm(bs[l][:, None], H[l], Ws[l].transpose(1, 2))
            H.append(Z.relu() if l + 1 < L else Z)
        dZ, loss = _softmax_ce(H[L], y[:, rows].long())
        for l in range(L - 1, -1, -1):
            dH = torch.bmm(dZ, Ws[l]) * (H[l] > 0) if l else None
            Ws[l].baddbmm_(dZ.transpose(1, 2), H[l], alpha=-lr)
            bs[l] -= lr * dZ.sum(1)
            dZ = dH
        if (t + 1) % case["K1"] == 0:
            Ws, bs = [_group_mean(W, case["S"]) for W in Ws], [_group_mean(b, case["S"]) for b in bs]
    if case["kind"] != "loop":
        Ws, bs = [_group_mean(W, P) for W in Ws], [_group_mean(b, P) for b in bs]
    pad = lambda n: (n + 63) // 64 * 64          # every segment of a row starts on a 64-float boundary
    parts = []
    for W, b in zip(Ws, bs):
        for v in (W.reshape(P, -1), b):
            parts += [v, v.new_zeros(P, pad(v.shape[1]) - v.shape[1])]
    out = {"params": torch.cat(parts, dim=1)}
    if case["kind"] == "round_host":
        out["loss"] = loss
    return out
