"""What a user of this framework has it do, as cases to be measured.

A user's program creates a run (``PGC``), loads the partitions once and then
takes training steps in a loop: one pass here is one such step through the
public binding, with the straggler mask of that step, returning the decoded
gradient and the new parameters.  The runs are past their warm-up step, as a
training loop is for all but its first call; GC mode evaluates every partition
each step, which is also what a warm-up step does.

A case is a dict:
  mode     "pgc", "is_sgd", "gc" or "naive_cr"; scheme "FR" or "CR"
  n, s     workers and stragglers; loss, dtype, d, K as PGC takes them
  m        rows per partition; ragged: partitions of unequal size, up to m
  out      "device": outputs are device tensors, steps follow one another;
           "host": outputs are pinned host tensors, each call waits for them
  monitor  the program also asks for the training loss after the step
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_20739_gb300 import binding as B

LR = {"logistic": 0.1, "lsq": 0.05, "softmax": 0.1}
UNIFORM_LR = 1e-3           # few-class softmax on non-negative, image-like features


def _case(name, mode, scheme, n, s, loss, dtype, d, K, m, ragged=False, out="device", monitor=False):
    return {"name": name, "mode": mode, "scheme": scheme, "n": n, "s": s, "loss": loss, "dtype": dtype, "d": d,
            "K": K, "m": m, "ragged": ragged, "out": out, "monitor": monitor}


def listed():
    return [
        # the smallest run: a few hundred rows of a small model, where a step is
        # a launch and its latency
        _case("fr4_logistic_d64", "pgc", "FR", 4, 1, "logistic", "f32", 64, 1, 256),
        # an ordinary logistic regression, rows of a round length, bound by reading them
        _case("cr8_logistic_d1024", "pgc", "CR", 8, 2, "logistic", "f32", 1024, 1, 8192),
        # tabular data as it comes: an odd number of features, partitions of
        # unequal size, twelve workers with six copies each, results on the host
        _case("cr12_logistic_d3001", "pgc", "CR", 12, 5, "logistic", "f32", 3001, 1, 3000, ragged=True, out="host"),
        # the baseline that ignores stragglers, half-precision features
        _case("issgd16_lsq_bf16_d2000", "is_sgd", "CR", 16, 3, "lsq", "bf16", 2000, 1, 4096),
        # the largest streaming run: long rows, 8.6 GB of features a step
        _case("cr64_lsq_d16384", "pgc", "CR", 64, 4, "lsq", "f32", 16384, 1, 2048),
        # the naive pipelined construction, whose decode weights are solved for each mask
        _case("naive8_logistic_d1024", "naive_cr", "CR", 8, 2, "logistic", "f32", 1024, 1, 8192),
        # small images in single precision, ten classes
        _case("cr8_softmax_f32_k10_d784", "pgc", "CR", 8, 2, "softmax", "f32", 784, 10, 4096),
        # colour images in half precision, ten classes
        _case("fr32_softmax_bf16_k10_d3072", "pgc", "FR", 32, 3, "softmax", "bf16", 3072, 10, 4096),
        # gradient coding: all partitions each step (so is every run's warm-up step)
        _case("gc16_softmax_bf16_k10_d1000", "gc", "FR", 16, 3, "softmax", "bf16", 1000, 10, 1000, ragged=True),
        # colour images, a hundred classes
        _case("cr12_softmax_bf16_k100_d3072", "pgc", "CR", 12, 3, "softmax", "bf16", 3072, 100, 4096),
        # the largest matrix work: a thousand classes, 128 workers
        _case("cr128_softmax_bf16_k1000_d4096", "pgc", "CR", 128, 7, "softmax", "bf16", 4096, 1000, 1024),
        # a small many-class model trained with its loss printed at every step
        _case("fr8_softmax_bf16_k300_d1500", "pgc", "FR", 8, 1, "softmax", "bf16", 1500, 300, 700, ragged=True,
              out="host", monitor=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more run of the same kinds: streaming losses in both types, few,
    some and many classes in half precision, few and some in single."""
    kind = rng.choice(["rows", "rows", "few", "few32", "some", "some32", "many"])
    mode = rng.choice(["pgc"] * 7 + ["is_sgd", "gc", "naive_cr"])
    scheme = rng.choice(["FR", "CR"]) if mode in ("pgc", "gc") else "CR"
    n = rng.choice([4, 6, 8, 12, 16, 24, 32] if mode != "naive_cr" else [4, 6, 8, 12])
    if scheme == "FR":
        s = rng.choice([c for c in range(2, 9) if n % c == 0]) - 1
    else:
        s = rng.randint(1, min(5, n // 2))
    if mode == "naive_cr" or (mode == "gc" and scheme == "CR"):
        s = min(s, 3)
        n = min(n, 12)
    if kind == "rows":
        loss, dtype, K = rng.choice(["logistic", "lsq"]), rng.choice(["f32", "bf16"]), 1
        if mode == "naive_cr":
            loss = "logistic"           # its stale coefficients do not let least squares settle
        d = _log_uniform(rng, 32, 16384)
        total = _log_uniform(rng, 1 << 18, 1 << 29)            # features of all partitions
    else:
        loss = "softmax"
        dtype = "f32" if kind.endswith("32") else "bf16"
        K = rng.randint(2, 16) if kind.startswith("few") else \
            _log_uniform(rng, 17, 127) if kind.startswith("some") else _log_uniform(rng, 128, 1500)
        d = _log_uniform(rng, 64, 3072 if kind == "few" else 4096)
        total = min(_log_uniform(rng, 1 << 18, 1 << 28), (1 << 34) // K)
    m = max(16, min(16384, total // (n * d)))
    out = rng.choice(["device", "device", "host"])
    return {"mode": mode, "scheme": scheme, "n": n, "s": s, "loss": loss, "dtype": dtype, "d": d, "K": K, "m": m,
            "ragged": rng.random() < 0.5, "out": out, "monitor": out == "host" and rng.random() < 0.25}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rows(case):
    m = case["m"]
    if not case["ragged"]:
        return [m] * case["n"]
    return [m - (k * 29 + 7) % (m // 3 + 1) for k in range(case["n"])]


def _lr(case):
    """A rate the run is stable at: smaller where features outnumber rows."""
    if _uniform(case):
        return UNIFORM_LR
    return LR[case["loss"]] / (1.0 + math.sqrt(case["d"] / sum(_rows(case)))) ** 2


def _uniform(case):
    return case["loss"] == "softmax" and case["K"] <= 16


def _generator(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + k) % (1 << 62))
    return g


def _planted(case, seed):
    """The model that the labels come from, entries N(0, 1/d)."""
    g = _generator(seed, 0)
    shape = (case["K"], case["d"])
    return torch.randn(shape, generator=g, device="cuda") / math.sqrt(case["d"])


def _partition(case, seed, k, planted):
    g = _generator(seed, k + 1)
    shape = (_rows(case)[k], case["d"])
    make = torch.rand if _uniform(case) else torch.randn
    X = make(shape, generator=g, device="cuda")
    if case["dtype"] == "bf16":
        X = X.to(torch.bfloat16)
    z = X.float() @ planted.t()
    if case["loss"] == "logistic":
        y = (torch.rand(shape[0], generator=g, device="cuda") < torch.sigmoid(z[:, 0])).float()
    elif case["loss"] == "lsq":
        y = z[:, 0] + 0.1 * torch.randn(shape[0], generator=g, device="cuda")
    else:
        gumbel = -torch.log(-torch.log(torch.rand(z.shape, generator=g, device="cuda").clamp_(1e-7, 1 - 1e-7)))
        y = torch.argmax(z + gumbel, dim=1).to(torch.int32)
    return X, y.contiguous()


def _masks(case, seed, steps=64):
    """Each step's s stragglers: the workers with the largest exponential delay."""
    rng = np.random.default_rng([int(seed), 2])
    masks = np.zeros((steps, case["n"]), dtype=np.uint8)
    for mask, delay in zip(masks, rng.exponential(size=masks.shape)):
        mask[np.argsort(delay)[case["n"] - case["s"]:]] = 1
    return masks


def _coded(case):
    """Whether the mode uploads with gradient coding's cyclic coefficients."""
    return case["mode"] == "naive_cr" or (case["mode"] == "gc" and case["scheme"] == "CR")


def _draws(case, seed):
    return np.random.default_rng([int(seed), 3]).standard_normal((case["s"], case["n"] - 1))


def prepare(case, seed):
    """A loaded run that has taken its warm-up step, half-way to the planted model."""
    planted = _planted(case, seed)
    run_ = B.PGC(case["scheme"], case["n"], case["s"], case["loss"], case["dtype"], case["d"], K=case["K"],
                 rows=_rows(case), lr=_lr(case), w0=(0.5 * planted).cpu().numpy(), mode=case["mode"])
    Xs, ys = zip(*(_partition(case, seed, k, planted) for k in range(case["n"])))
    torch.cuda.synchronize()
    run_.load(Xs, ys)
    del Xs, ys
    if _coded(case):
        run_.set_gc_encoding(_draws(case, seed))
    size = case["K"] * case["d"]
    host = case["out"] == "host"
    grad, beta = (torch.zeros(size, pin_memory=True) if host else torch.zeros(size, device="cuda") for _ in range(2))
    masks = _masks(case, seed)
    run_.step(masks[0], grad, beta)
    return {"run": run_, "masks": masks, "next": 1, "grad": grad, "beta": beta, "monitor": case["monitor"]}


def run(state):
    mask = state["masks"][state["next"] % 64]
    state["next"] += 1
    info = state["run"].step(mask, state["grad"], state["beta"])
    out = {"grad": state["grad"], "beta": state["beta"], "evaluated": info["eval_partition"]}
    if state["monitor"]:
        out["loss"] = state["run"].loss()
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how exact it is
# ---------------------------------------------------------------------------

def work(case):
    """Features and labels of the evaluated partitions read once; their
    gradients written to the stores; the decode's other slots (slot totals and
    the stragglers' stores) and the parameters read, gradient and parameters
    written.  Loss: every partition's features again.  Flops: both products."""
    n, s, d, K = case["n"], case["s"], case["d"], case["K"]
    c = 1 if case["mode"] == "is_sgd" else s + 1
    rows = _rows(case)
    part = [0 + g * c for g in range(n // c)] if case["mode"] == "pgc" and case["scheme"] == "FR" else range(n)
    evaluated = sum(rows[k] for k in part)
    size = 2 if case["dtype"] == "bf16" else 4
    copies = len(part) * (c if case["mode"] == "gc" and case["scheme"] == "CR" else 1)
    if _coded(case):
        decoded = (n - s) * c
    else:
        decoded = c + (s * c if case["scheme"] == "CR" else 0)
    total = evaluated * (d * size + 4) + (copies + decoded + 3) * K * d * 4
    flops = 4.0 * evaluated * d * K
    if case["monitor"]:
        total += sum(rows) * (d * size + 4)
        flops += 2.0 * sum(rows) * d * K
    return {"bytes": float(total), "flops": flops}


def tolerance(case):
    """Sums in single precision, but for half-precision softmax with few or many
    classes, whose kernels multiply parameters and residuals rounded to bf16."""
    if case["loss"] == "softmax" and case["dtype"] == "bf16" and not 16 < case["K"] < 128:
        return {"rel": 1e-2}
    return {"rel": 2e-5 if _coded(case) else 1e-5}


# ---------------------------------------------------------------------------
# the same step in 64 bits
# ---------------------------------------------------------------------------

def _gradient(case, X, y, w):
    """Mean gradient of one partition at w [K, d], in row blocks."""
    g = torch.zeros_like(w)
    for r in range(0, X.shape[0], 8192):
        x, t = X[r:r + 8192].double(), y[r:r + 8192]
        z = x @ w.t()
        if case["loss"] == "softmax":
            z = torch.softmax(z, dim=1)
            z[torch.arange(z.shape[0], device=z.device), t.long()] -= 1.0
        else:
            z = (torch.sigmoid(z) if case["loss"] == "logistic" else z) - t.double()[:, None]
        g += z.t() @ x
    return g / X.shape[0]


def _loss_sum(case, X, y, w):
    z = X.double() @ w.t()
    if case["loss"] == "softmax":
        return float((torch.logsumexp(z, 1) - z.gather(1, y.long()[:, None])[:, 0]).sum())
    z, t = z[:, 0], y.double()
    f = torch.nn.functional.softplus(z) - t * z if case["loss"] == "logistic" else 0.5 * (z - t) ** 2
    return float(f.sum())


def _encoding(case, seed):
    """Cyclic-repetition coefficients c[j][l] of worker j on partition (j + l) mod n."""
    n, s = case["n"], case["s"]
    H = _draws(case, seed)
    H = np.concatenate([H, -H.sum(1, keepdims=True)], axis=1)
    coeff = np.ones((n, s + 1))
    for j in range(n):
        at = [(j + l) % n for l in range(1, s + 1)]
        coeff[j, 1:] = np.linalg.solve(H[:, at], -H[:, j])
    return coeff


def _store_weights(case, seed, mask):
    """Weight of worker i's stored gradient of partition (slot l) in the decode: [n][c]."""
    n, s = case["n"], case["s"]
    c = 1 if case["mode"] == "is_sgd" else s + 1
    got = mask == 0
    if _coded(case):
        coeff = _encoding(case, seed)
        full = np.zeros((n, n))
        for j in range(n):
            full[j, [(j + l) % n for l in range(c)]] = coeff[j]
        d = np.zeros(n)
        d[got] = np.linalg.lstsq(full[got].T, np.ones(n), rcond=None)[0]
        return coeff * d[:, None] / n
    if case["scheme"] == "CR":
        return np.repeat(np.where(got, 1.0 / ((n - s) * c), 0.0)[:, None], c, 1)
    a = np.zeros(n)                                   # FR: one of each group is decoded, all hold the same
    for g in range(n // c):
        a[g * c + int(np.argmax(got[g * c:(g + 1) * c]))] = 1.0 / n
    return np.repeat(a[:, None], c, 1)


def _decode(case, seed, mask, gradients):
    """sum over workers and slots of weight x gradients[l][partition held there]."""
    n = case["n"]
    weights = _store_weights(case, seed, mask)
    c = weights.shape[1]
    total = None
    per = {}
    for i in range(n):
        for l in range(c):
            k = (i // c) * c + l if case["scheme"] == "FR" else (i + l) % n
            per[(l, k)] = per.get((l, k), 0.0) + weights[i, l]
    for (l, k), a in per.items():
        if a:
            g = gradients[l][k]
            total = a * g if total is None else total.add_(g, alpha=a)
    return total


def exact(case, seed):
    planted = _planted(case, seed)
    parts = (lambda: (_partition(case, seed, k, planted) for k in range(case["n"])))
    lr = float(np.float32(_lr(case)))
    masks = _masks(case, seed)
    n = case["n"]
    c = 1 if case["mode"] == "is_sgd" else case["s"] + 1
    w = (0.5 * planted).double()
    first = [_gradient(case, X, y, w) for X, y in parts()]
    w = w - lr * _decode(case, seed, masks[0], [first] * c)
    if case["mode"] == "gc":
        evaluated, slot = range(n), -1
    elif case["scheme"] == "FR":
        evaluated, slot = range(0, n, c), 0
    else:
        evaluated, slot = range(n), 0
    wanted = set(evaluated)
    second = [_gradient(case, X, y, w) if k in wanted else None for k, (X, y) in enumerate(parts())]
    latest = [second if l == slot or slot < 0 else first for l in range(c)]
    grad = _decode(case, seed, masks[1], latest)
    w = w - lr * grad
    out = {"grad": grad.reshape(-1), "beta": w.reshape(-1), "evaluated": None}
    if case["monitor"]:
        out["loss"] = sum(_loss_sum(case, X, y, w) for X, y in parts()) / sum(_rows(case))
    return out
