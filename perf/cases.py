"""Performance cases of the emulated FP64 product, through its public Python entry points.

Sizes come from the benchmark and the tests (16384^3, 4096 x 4096 x 65536,
65536 x 1024 x 1024, the uneven batch on [64, 2048], the 8192 x 4096 x 4096 autograd
step) or are generic squares and ragged shapes of the same ranges.
"""
import math

import torch

import paper_2603_10634_gb300 as ozk
from paper_2603_10634_gb300 import workloads


def listed():
    return [
        # one small product on its own: launches and latency
        _dgemm("square_256", 256, 256, 256, 12, phi=0.5),
        # a ragged product with A given as a transposed view, Cauchy-Schwarz scaling
        _dgemm("ragged_fast_ta", 1023, 777, 1501, 14, phi=0.5, mode="fast", ta=True),
        # one ordinary product
        _dgemm("square_1024", 1024, 1024, 1024, 12, phi=1.0),
        # wide-range entries, which need more moduli; B given as a transposed view
        _dgemm("square_2048_n14_tb", 2048, 2048, 2048, 14, phi=2.0, tb=True),
        # a few right-hand sides: the last 100 columns of a wider matrix
        _dgemm("narrow_n", 8192, 100, 4096, 12, phi=1.0, pad=28),
        _dgemm("square_4096", 4096, 4096, 4096, 12, phi=1.0),
        # short and long reductions
        _dgemm("tall_short_k", 65536, 1024, 1024, 12, phi=1.0),
        _dgemm("long_k", 4096, 4096, 65536, 12, phi=1.0),
        # the headline product
        _dgemm("square_16384", 16384, 16384, 16384, 12, phi=1.0),
        # many uneven small products, planned once and executed again and again
        {"name": "batch_48", "kind": "batch", "count": 48, "lo": 64, "hi": 2048, "shapes": 0, "N": 12, "phi": 1.0,
         "mode": "accurate"},
        # a linear layer's forward and both gradients
        {"name": "autograd_8192", "kind": "autograd", "m": 8192, "n": 4096, "k": 4096, "N": 12, "phi": 0.5},
        # operands and result in pinned host memory
        {"name": "host_4096", "kind": "host", "m": 4096, "n": 4096, "k": 4096, "N": 12, "phi": 1.0, "mode": "accurate"},
    ]


def _dgemm(name, m, n, k, N, phi, mode="accurate", ta=False, tb=False, pad=0):
    return {"name": name, "kind": "dgemm", "m": m, "n": n, "k": k, "N": N, "phi": phi, "mode": mode, "ta": ta, "tb": tb,
            "pad": pad}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    phi = rng.choice([0.5, 1.0, 2.0])
    N = rng.choice([12, 12, 12, 13, 14, 16, 8, 20])
    mode = rng.choice(["accurate", "accurate", "accurate", "fast"])
    kind = rng.choice(["dgemm"] * 7 + ["batch", "autograd", "host"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(4, 48), "lo": 64, "hi": 2048, "shapes": rng.randint(1, 1000), "N": N,
                "phi": phi, "mode": mode}
    while True:
        if kind == "dgemm":
            m, n, k = _log_int(rng, 64, 65536), _log_int(rng, 64, 16384), _log_int(rng, 64, 65536)
        else:
            m, n, k = _log_int(rng, 128, 8192), _log_int(rng, 128, 4096), _log_int(rng, 128, 4096)
        # well below the largest listed product, with operands below its 2 x 16384^2
        if m * n * k <= 4.0e11 and m * k <= 2 ** 28 and k * n <= 2 ** 28 and m * n <= 2 ** 28:
            break
    if kind == "autograd":
        return {"kind": kind, "m": m, "n": n, "k": k, "N": N, "phi": phi}
    if kind == "host":
        return {"kind": kind, "m": m, "n": n, "k": k, "N": N, "phi": phi, "mode": mode}
    return _without_name(_dgemm("", m, n, k, N, phi, mode, rng.random() < 0.25, rng.random() < 0.25,
                                rng.choice([0, 0, 1, 28])))


def _without_name(case):
    return {key: v for key, v in case.items() if key != "name"}


def _operands(c, seed):
    """(A, B) of a dgemm case: row-major, transposed views, or (pad) columns of wider
    row-major matrices."""

    def matrix(rows, cols, transposed, s):
        if transposed:
            return workloads.phi_matrix(cols, rows, c["phi"], s, "cuda").T
        return workloads.phi_matrix(rows, cols + c["pad"], c["phi"], s, "cuda")[:, c["pad"]:]

    return matrix(c["m"], c["k"], c["ta"], 2 * seed), matrix(c["k"], c["n"], c["tb"], 2 * seed + 1)


def _pair(c, seed, device="cuda"):
    return (workloads.phi_matrix(c["m"], c["k"], c["phi"], 4 * seed, device),
            workloads.phi_matrix(c["k"], c["n"], c["phi"], 4 * seed + 1, device))


def _upstream(c, seed):
    return workloads.normal_matrix(c["m"], c["n"], 4 * seed + 2, "cuda")


def _batch(c, seed):
    shapes = workloads.batch_shapes(c["count"], c["lo"], c["hi"], seed=c["shapes"])
    return workloads.batch_problems(shapes, c["phi"], seed=1000 * seed, device="cuda")


def prepare(case, seed):
    c = case
    if c["kind"] == "dgemm":
        return c, *_operands(c, seed)
    if c["kind"] == "batch":
        # a plan holds its operands, outputs and workspace
        As, Bs = _batch(c, seed)
        return c, ozk.BatchPlan(As, Bs, num_moduli=c["N"], mode=c["mode"])
    if c["kind"] == "autograd":
        A, B = _pair(c, seed)
        return c, A.requires_grad_(), B.requires_grad_(), _upstream(c, seed)
    A, B = _pair(c, seed)
    out = torch.empty((c["m"], c["n"]), dtype=torch.float64, pin_memory=True)
    return c, A.cpu().pin_memory(), B.cpu().pin_memory(), out


def run(state):
    c = state[0]
    if c["kind"] == "dgemm":
        return ozk.dgemm(state[1], state[2], num_moduli=c["N"], mode=c["mode"])
    if c["kind"] == "batch":
        return state[1].execute()
    if c["kind"] == "autograd":
        A, B, dC = state[1:]
        C = ozk.matmul(A, B, num_moduli=c["N"])
        dA, dB = torch.autograd.grad(C, (A, B), dC)
        return C.detach(), dA, dB
    return ozk.dgemm_host(state[1], state[2], num_moduli=c["N"], out=state[3], mode=c["mode"])


def work(case):
    """The FP64 product itself: 2 m n k operations, each operand read and each result
    written once (the emulation's own FP8 products and digit planes are its choice)."""
    c = case
    if c["kind"] == "batch":
        shapes = workloads.batch_shapes(c["count"], c["lo"], c["hi"], seed=c["shapes"])
    else:
        shapes = [(c["m"], c["n"], c["k"])]
    flops = sum(2.0 * m * n * k for m, n, k in shapes)
    size = sum(8.0 * (m * k + k * n + m * n) for m, n, k in shapes)
    if c["kind"] == "autograd":  # three products; dC in, dA and dB out
        return {"bytes": 2 * size, "flops": 3 * flops}
    return {"bytes": size, "flops": flops}


def exact(case, seed):
    c = case
    if c["kind"] == "dgemm":
        A, B = _operands(c, seed)
        return A @ B
    if c["kind"] == "batch":
        return [A @ B for A, B in zip(*_batch(c, seed))]
    A, B = _pair(c, seed)
    if c["kind"] == "autograd":
        dC = _upstream(c, seed)
        return A @ B, dC @ B.T, A.T @ dC
    return (A @ B).cpu()
