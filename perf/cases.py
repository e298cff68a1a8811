"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points of `paper_1801_04348_gb300.pgk` the
way a program calls them without tuning first (prog = None, no tuning cache, no cost
model): single products in each arithmetic form, groups of products, the other two
kernels of the paper (transposition and 1D Jacobi) and a training step of the cost
model.  Sizes come from the configurations, the tests and the benchmark of this
repository:

  f32_256              256^3, the correctness grid's size: one small call, launch and latency
  f32_4096             4096^3 on the SIMT units, an ordinary large FP32 product
  grouped_f32          512 uneven FP32 products in one persistent launch, replayed as a graph
  split_8192           the benchmark's own product at FP32 accuracy on the tensor cores
  split_ragged         odd sizes, padded row strides, accumulating into C (beta = 1)
  split_skinny         16384 x 64 x 16384: a wide matrix times a few columns, bound by reading A
  bf16_4096            an ordinary large product in BF16
  fp8_8192x1024x4096   a non-square product in FP8 with 128 x 128 tile scales
  grouped_split        the 512 uneven products at FP32 accuracy on the tensor cores
  transpose_16384      the transposition at the largest order of the paper's table (2^14)
  jacobi_32770         four time steps at the paper's length 2^15 + 2
  train_256            forward, backward and Adam update of one minibatch of the cost model

`draw` gives further cases of the same kinds: sizes log-uniform over the range, most of
them odd, all of them no dearer than the largest listed case.

Errors: `exact` follows the definition of each form in binary64.  BF16 and FP8 round or
quantise the operands first, as the form is defined, so what is left is the error of the
sums; the split form is compared with the product of the FP32 operands, since it stands
in for it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1801_04348_gb300 import inputs, pgk

FORMS = {"f32": pgk.F32, "bf16": pgk.BF16, "fp8": pgk.FP8_E4M3, "split": pgk.SPLIT_BF16}
LARGEST = 8192 ** 3          # multiply-adds of the largest tensor-core product
LARGEST_F32 = 4096 ** 3      # and of the largest one on the SIMT units
TRAIN_ROWS = 15360           # rows of the timing log that the cost model trains on


def _gemm(name, form, M, N, K, pad=0, beta=0):
    return {"name": name, "kind": "gemm", "form": form, "M": M, "N": N, "K": K, "pad": pad, "beta": beta}


def listed():
    return [
        _gemm("f32_256", "f32", 256, 256, 256),
        _gemm("f32_4096", "f32", 4096, 4096, 4096),
        {"name": "grouped_f32", "kind": "grouped", "form": "f32", "G": 512, "lo": 32, "hi": 2048,
         "multiple": 16, "graph": 1},
        _gemm("split_8192", "split", 8192, 8192, 8192),
        _gemm("split_ragged", "split", 513, 1030, 777, pad=5, beta=1),
        _gemm("split_skinny", "split", 16384, 64, 16384),
        _gemm("bf16_4096", "bf16", 4096, 4096, 4096),
        _gemm("fp8_8192x1024x4096", "fp8", 8192, 1024, 4096),
        {"name": "grouped_split", "kind": "grouped", "form": "split", "G": 512, "lo": 32, "hi": 2048,
         "multiple": 16, "graph": 0},
        {"name": "transpose_16384", "kind": "transpose", "rows": 16384, "cols": 16384},
        {"name": "jacobi_32770", "kind": "jacobi", "n": 32770, "steps": 4},
        {"name": "train_256", "kind": "train", "batch": 256},
    ]


def _log_int(rng, lo, hi):
    """An integer log-uniform in [lo, hi], odd more often than not."""
    x = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.4:
        x |= 1
    elif rng.random() < 0.5:
        x = (x + 15) // 16 * 16
    return max(lo, min(hi, x))


def draw(rng):
    kind = rng.choices(["f32", "tensor", "skinny", "grouped", "transpose", "jacobi", "train"],
                       weights=[3, 6, 2, 2, 1, 1, 1])[0]
    if kind == "f32":
        while True:
            M, N, K = (_log_int(rng, 32, 8192) for _ in range(3))
            if M * N * K <= LARGEST_F32:
                break
        return {k: v for k, v in _gemm("", "f32", M, N, K, rng.choice([0, 0, 4, 5]),
                                       rng.choice([0, 0, 1])).items() if k != "name"}
    if kind == "tensor":
        while True:
            M, N, K = (_log_int(rng, 64, 16384) for _ in range(3))
            if M * N * K <= LARGEST and max(M * K, K * N, M * N) <= 2 ** 28:
                break
        form = rng.choice(["split", "split", "bf16", "fp8"])
        return {k: v for k, v in _gemm("", form, M, N, K, rng.choice([0, 0, 0, 4, 5]),
                                       rng.choice([0, 0, 0, 1])).items() if k != "name"}
    if kind == "skinny":
        N = rng.randint(1, 64)
        while True:
            M, K = _log_int(rng, 512, 32768), _log_int(rng, 512, 65536)
            if M * K <= 2 ** 28:
                break
        K = (K + 3) // 4 * 4
        return {k: v for k, v in _gemm("", rng.choice(["split", "bf16"]), M, N, K, rng.choice([0, 0, 4]),
                                       rng.choice([0, 0, 1])).items() if k != "name"}
    if kind == "grouped":
        return {"kind": "grouped", "form": rng.choice(["f32", "split", "bf16"]), "G": _log_int(rng, 8, 512),
                "lo": 32, "hi": rng.choice([512, 1024, 2048]), "multiple": rng.choice([1, 16]), "graph": 0}
    if kind == "transpose":
        return {"kind": "transpose", "rows": _log_int(rng, 64, 16384), "cols": _log_int(rng, 64, 16384)}
    if kind == "jacobi":
        return {"kind": "jacobi", "n": _log_int(rng, 1024, 2 ** 26), "steps": rng.randint(1, 8)}
    return {"kind": "train", "batch": _log_int(rng, 64, 14000)}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _matrix(rows, cols, pad, g, normal):
    """rows x cols with a row stride of cols + pad: uniform in [-1, 1], or normal."""
    w = torch.empty(rows, cols + pad, device="cuda")
    if normal:
        w.normal_(generator=g)
    else:
        w.uniform_(-1.0, 1.0, generator=g)
    return w[:, :cols]


def _operands(case, seed):
    g = _generator(seed)
    M, N, K, pad = case["M"], case["N"], case["K"], case["pad"]
    normal = case["form"] != "f32"
    A = _matrix(M, K, pad, g, normal)
    B = _matrix(K, N, pad, g, normal)
    C = _matrix(M, N, pad, g, True)
    return A, B, C


def _group(case, seed):
    """The problems of a group, packed one after another: (A, B, C) views and the buffers."""
    dims = inputs.log_uniform_dims(case["G"], 0, case["lo"], case["hi"], case["multiple"]).tolist()

    def room(n):
        return (n + 127) // 128 * 128

    na, nb, nc = (sum(room(d[i] * d[j]) for d in dims) for i, j in ((0, 2), (2, 1), (0, 1)))
    g = _generator(seed)
    a = torch.empty(na, device="cuda").normal_(generator=g)
    b = torch.empty(nb, device="cuda").normal_(generator=g)
    c = torch.zeros(nc, device="cuda")
    triples, oa, ob, oc = [], 0, 0, 0
    for M, N, K in dims:
        triples.append((a[oa:oa + M * K].view(M, K), b[ob:ob + K * N].view(K, N), c[oc:oc + M * N].view(M, N)))
        oa, ob, oc = oa + room(M * K), ob + room(K * N), oc + room(M * N)
    return triples, c


def _training_set(case, seed):
    g = _generator(seed)
    X = torch.empty(TRAIN_ROWS, 7, device="cuda").normal_(generator=g)
    t = torch.empty(TRAIN_ROWS, device="cuda").normal_(generator=g)
    idx = torch.randperm(TRAIN_ROWS, generator=g, device="cuda")[:case["batch"]].to(torch.int32)
    theta = torch.from_numpy(inputs.he_uniform_mlp(seed)).cuda()
    return X, t, idx, theta


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B, C = _operands(case, seed)
        return {"kind": kind, "form": FORMS[case["form"]], "A": A, "B": B, "C": C, "beta": case["beta"]}
    if kind == "grouped":
        triples, c = _group(case, seed)
        return {"kind": kind, "form": FORMS[case["form"]], "problems": pgk.make_problems(triples),
                "C": c, "keep": triples, "graph": case["graph"]}
    if kind == "transpose":
        src = _matrix(case["rows"], case["cols"], 0, _generator(seed), True)
        return {"kind": kind, "src": src, "dst": torch.empty(case["cols"], case["rows"], device="cuda")}
    if kind == "jacobi":
        a = torch.randint(-10 ** 6, 10 ** 6, (2 * case["n"],), generator=_generator(seed), device="cuda",
                          dtype=torch.int32)
        return {"kind": kind, "a": a, "n": case["n"], "steps": case["steps"]}
    X, t, idx, theta = _training_set(case, seed)
    return {"kind": kind, "X": X, "t": t, "idx": idx, "theta": theta, "grad": torch.empty_like(theta),
            "m": torch.zeros_like(theta), "v": torch.zeros_like(theta), "loss": torch.empty(1, device="cuda"),
            "step": 0}


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind == "gemm":
        pgk.gemm(state["A"], state["B"], state["C"], state["form"], beta=state["beta"])
        return state["C"]
    if kind == "grouped":
        pgk.gemm_grouped(state["problems"], state["form"], use_graph=state["graph"])
        return state["C"]
    if kind == "transpose":
        pgk.transpose(state["src"], state["dst"])
        return state["dst"]
    if kind == "jacobi":
        pgk.jacobi(state["a"], state["n"], state["steps"])
        return state["a"]
    state["step"] += 1
    pgk.mlp_loss_grad(state["X"], state["t"], state["theta"], state["grad"], state["loss"], idx=state["idx"])
    pgk.mlp_adam(state["theta"], state["grad"], state["m"], state["v"], state["step"], lr=1e-3)
    return {"loss": state["loss"], "grad": state["grad"], "theta": state["theta"], "m": state["m"],
            "v": state["v"]}


# -------------------------------------------------------- work and accuracy
def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        products = 3 if case["form"] == "split" else 1   # lo*hi + hi*lo + hi*hi
        return {"bytes": 4 * (M * K + K * N + M * N * (1 + case["beta"])), "flops": 2 * M * N * K * products}
    if kind == "grouped":
        d = inputs.log_uniform_dims(case["G"], 0, case["lo"], case["hi"], case["multiple"])
        M, N, K = d[:, 0], d[:, 1], d[:, 2]
        products = 3 if case["form"] == "split" else 1
        return {"bytes": int(4 * (M * K + K * N + M * N).sum()), "flops": int(2 * (M * N * K).sum()) * products}
    if kind == "transpose":
        return {"bytes": 8 * case["rows"] * case["cols"], "flops": 0}
    if kind == "jacobi":
        # every step writes one half; the steps in between need not reach memory, the first
        # read and the last two halves do
        n = case["n"]
        return {"bytes": 4 * n * (1 + min(2, case["steps"])), "flops": 3 * n * case["steps"]}
    n, p = case["batch"], pgk.MLP_PARAMS
    return {"bytes": 4 * (n * 9 + 7 * p), "flops": 6 * p * n + 12 * p}


def tolerance(case):
    """About four times the distance from `exact` that the sums of each form show (FP32:
    1.1e-6 at K = 4096 and 1.6e-6 at 8192; tensor cores, whose FP32
    accumulators do not round to nearest: split 4.7e-6 to 6.3e-6, BF16 and FP8 4.4e-6 and,
    in the longest sums, 1e-5; training step: 1.4e-7)."""
    kind = case["kind"]
    if kind in ("transpose", "jacobi"):
        return "exact"
    if kind == "train":
        return {"rel": 2e-6}
    return {"rel": {"f32": 6e-6, "split": 2.5e-5}.get(case["form"], 4e-5)}


def _fp8_values(x):
    """x quantised per 128 x 128 tile to E4M3 codes and back, as the form defines it:
    scale = amax / 448 in FP32 (1 for a tile of zeros), code = round-to-nearest of x / scale."""
    R, Cc = x.shape
    p = torch.nn.functional.pad(x, (0, -Cc % 128, 0, -R % 128))
    t = p.view(p.shape[0] // 128, 128, p.shape[1] // 128, 128)
    amax = t.abs().amax(dim=(1, 3), keepdim=True)
    scale = torch.where(amax == 0, torch.ones_like(amax), amax / torch.full_like(amax, 448.0))
    q = (t / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).to(torch.float64)
    return (q * scale.double()).reshape(p.shape)[:R, :Cc]


def _operand64(x, form):
    if form == "bf16":
        return x.to(torch.bfloat16).double()
    return _fp8_values(x) if form == "fp8" else x.double()


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B, C = _operands(case, seed)
        r = _operand64(A, case["form"]) @ _operand64(B, case["form"])
        return r + C.double() if case["beta"] else r
    if kind == "grouped":
        triples, c = _group(case, seed)
        out, at = torch.zeros(c.numel(), dtype=torch.float64, device="cuda"), 0
        for A, B, C in triples:
            out[at:at + C.numel()] = (_operand64(A, case["form"]) @ _operand64(B, case["form"])).reshape(-1)
            at += (C.numel() + 127) // 128 * 128
        return out
    if kind == "transpose":
        return _matrix(case["rows"], case["cols"], 0, _generator(seed), True).t().contiguous()
    if kind == "jacobi":
        n = case["n"]
        a = torch.randint(-10 ** 6, 10 ** 6, (2 * n,), generator=_generator(seed), device="cuda",
                          dtype=torch.int32).long()
        for s in range(case["steps"]):
            src, dst = (a[n:], a[:n]) if s & 1 else (a[:n], a[n:])
            dst[1:n - 1] = torch.div(src[:-2] + src[1:-1] + src[2:], 3, rounding_mode="trunc")
        return a.to(torch.int32)
    X, t, idx, theta = _training_set(case, seed)
    th = theta.double().requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = torch.split(th, [448, 64, 4096, 64, 64, 1])
    x, y = X[idx.long()].double(), t[idx.long()].double()
    h = torch.relu(x @ W1.view(64, 7).t() + b1)
    h = torch.relu(h @ W2.view(64, 64).t() + b2)
    loss = ((h @ w3 + b3 - y) ** 2).mean()
    g, = torch.autograd.grad(loss, th)
    b1_, b2_ = float(np.float32(0.9)), float(np.float32(0.999))
    m, v = (1 - b1_) * g, (1 - b2_) * g * g
    new = theta.double() - 1e-3 * (m / (1 - b1_)) / ((v / (1 - b2_)).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": g, "theta": new, "m": m, "v": v}
