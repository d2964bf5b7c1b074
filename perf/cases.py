"""The work that a user has this library do, as cases that can be timed.

Every case is one call (for the power-of-two FFT a forward and an inverse
one) of a public entry point of ``paper_2310_16214_gb300`` on device buffers
that the caller owns, with no plan given, as a program that does not tune
calls it.  Sizes are those of the paper's batches (2^24 or 2^26 elements over
N) and of this repository's benchmark and its reports; ``draw`` spreads them
over the sizes that the entry points take.

A case is a dict of plain values:
    kind   "scan", "fft", "fft_pair", "fft_tc", "tridiag", "refined", "uneven"
    n      elements (unknowns) per problem; batch: problems (uneven: problems
           of each operation)
    dtype  scan: "i32" or "f32"; dir: FFT direction -1 or +1; precision:
           "bf16" or "f16" split of the tensor-core FFT; tol: refinement target;
           sizes: seed of the uneven batch's problem sizes
"""
import math
import random

import torch

import paper_2310_16214_gb300 as bp

DEV = "cuda"
UNEVEN_LO, UNEVEN_HI = 5, 13  # sizes 2^5 .. 2^13


def listed():
    return [
        # The plain batch of the paper's first configuration: 8 MB in all, so the
        # call's own latency (argument checks, plan look-up, launch) shows.
        {"name": "scan_small", "kind": "scan", "dtype": "i32", "n": 1024, "batch": 1024},
        # Running sums over long rows at the paper's full batch of 2^26 elements.
        {"name": "scan_long", "kind": "scan", "dtype": "f32", "n": 8192, "batch": 8192},
        # Row lengths of real tables (histogram bins, prefix offsets) are seldom powers of two.
        {"name": "scan_ragged", "kind": "scan", "dtype": "i32", "n": 5000, "batch": 3355},
        # Spectral filtering and convolution: to the frequency domain and back.
        {"name": "fft_pair_4096", "kind": "fft_pair", "n": 4096, "batch": 4096},
        # Instrument frames of decimal length: 2^a 3^b 5^c points.
        {"name": "fft_3000", "kind": "fft", "n": 3000, "batch": 5592, "dir": -1},
        # A length with other prime factors (7, 11, 13), synthesis direction.
        {"name": "fft_1001_inv", "kind": "fft", "n": 1001, "batch": 16760, "dir": 1},
        # Long records, one transform per record: more points than a block holds.
        {"name": "fft_2e20", "kind": "fft", "n": 1 << 20, "batch": 16, "dir": -1},
        # The precision configuration's middle size through the tensor-core entry point.
        {"name": "fft_tc_4096", "kind": "fft_tc", "n": 4096, "batch": 16384, "dir": -1, "precision": "f16"},
        # Implicit line solves (ADI, splines) on a power-of-two grid.
        {"name": "tridiag_1024", "kind": "tridiag", "n": 1024, "batch": 16384},
        # The same on a grid whose lines are not a power of two.
        {"name": "tridiag_3000", "kind": "tridiag", "n": 3000, "batch": 5592},
        # Solves to float64 accuracy from float32 coefficients.
        {"name": "refined_1024", "kind": "refined", "n": 1024, "batch": 16384, "tol": 1e-12},
        # A mixed batch of scans, FFTs and solves of many sizes in one graph launch.
        {"name": "uneven_4096", "kind": "uneven", "batch": 4096, "sizes": 1},
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _batch(rng, n, lo_log, hi_log):
    """Problems for a call of 2^lo_log to 2^hi_log elements."""
    return max(1, _log_int(rng, 1 << lo_log, 1 << hi_log) // n)


def draw(rng):
    kind = rng.choice(["scan", "scan", "fft_pair", "fft", "fft", "fft_long", "fft_tc", "tridiag", "tridiag", "refined",
                       "uneven"])
    if kind == "scan":
        n = 1 << rng.randint(4, 15) if rng.random() < 0.4 else _log_int(rng, 16, 32768)
        return {"kind": "scan", "dtype": rng.choice(["i32", "f32"]), "n": n, "batch": _batch(rng, n, 17, 26)}
    if kind == "fft_pair":
        n = 1 << rng.randint(4, 14)
        return {"kind": "fft_pair", "n": n, "batch": _batch(rng, n, 17, 24)}
    if kind == "fft":
        # any length; half of them products of 2, 3 and 5
        n = _log_int(rng, 17, 12288)
        if rng.random() < 0.5:
            n = min((2 ** a * 3 ** b * 5 ** c for a in range(14) for b in range(9) for c in range(6)),
                    key=lambda m: (abs(math.log(m / n)), m))
        hi = 24 if n <= 4096 else 22
        return {"kind": "fft", "n": n, "batch": _batch(rng, n, 17, hi), "dir": rng.choice([-1, 1])}
    if kind == "fft_long":
        n = 1 << rng.randint(15, 22)
        return {"kind": "fft", "n": n, "batch": _batch(rng, n, 22, 24), "dir": rng.choice([-1, 1])}
    if kind == "fft_tc":
        n = 1 << rng.randint(9, 14)
        return {"kind": "fft_tc", "n": n, "batch": _batch(rng, n, 20, 25), "dir": rng.choice([-1, 1]),
                "precision": rng.choice(["bf16", "f16"])}
    if kind == "tridiag":
        n = 1 << rng.randint(4, 13) if rng.random() < 0.5 else _log_int(rng, 17, 8192)
        return {"kind": "tridiag", "n": n, "batch": _batch(rng, n, 17, 24)}
    if kind == "refined":
        n = 1 << rng.randint(5, 12)
        return {"kind": "refined", "n": n, "batch": _batch(rng, n, 17, 24), "tol": rng.choice([1e-12, 1e-14])}
    return {"kind": "uneven", "batch": _log_int(rng, 256, 4096), "sizes": rng.randrange(2, 1 << 20)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _pm1(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float32).mul_(2).sub_(1)


def _ints(g, *shape):
    return torch.randint(-1000, 1001, shape, generator=g, device=DEV, dtype=torch.int32)


def _complex(g, *shape):
    return torch.view_as_complex(_pm1(g, *shape, 2))


def _systems(g, batch, n):
    """Diagonally dominant systems (a, b, c, d): a, c and the solution uniform
    on [-1, 1], b = |a| + |c| + U[1, 2], d in float64 rounded once."""
    a, c, x = (_pm1(g, batch, n) for _ in range(3))
    a[:, 0] = 0
    c[:, n - 1] = 0
    b = a.abs() + c.abs() + 1 + torch.rand(batch, n, generator=g, device=DEV, dtype=torch.float32)
    d = b.double() * x.double()
    d[:, 1:] += a[:, 1:].double() * x[:, :-1].double()
    d[:, :-1] += c[:, :-1].double() * x[:, 1:].double()
    return a, b, c, d.float()


def _uneven_counts(case):
    """(operation, size, problems) of the mixed batch: sizes log-uniform."""
    rng = random.Random(case["sizes"])
    out = []
    for op in range(3):
        drawn = [rng.randint(UNEVEN_LO, UNEVEN_HI) for _ in range(case["batch"])]
        out += [(op, 1 << e, drawn.count(e)) for e in range(UNEVEN_LO, UNEVEN_HI + 1) if e in drawn]
    return out


def _uneven_problems(case, seed):
    """Arenas of the mixed batch: per operation and size one [count][n] block
    per array, so that every problem starts on a 16-byte boundary."""
    g = _gen(seed)
    return [(op, n, m, (_ints(g, m, n),) if op == 0 else (_complex(g, m, n),) if op == 1 else _systems(g, m, n))
            for op, n, m in _uneven_counts(case)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        blocks = _uneven_problems(case, seed)
        outs = [torch.empty_like(ins[-1]) for _, _, _, ins in blocks]
        ops = (bp.OP_SCAN, bp.OP_FFT, bp.OP_TRIDIAG)
        items = [{"op": ops[op], "n": n, "in": [t[k] for t in ins], "out": out[k], "dtype": bp.I32, "dir": -1}
                 for (op, n, m, ins), out in zip(blocks, outs) for k in range(m)]
        return {"kind": kind, "blocks": blocks, "outs": outs, "batch": bp.UnevenBatch(items)}
    n, batch = case["n"], case["batch"]
    g = _gen(seed)
    st = dict(case)
    if kind == "scan":
        st["x"] = _ints(g, batch, n) if case["dtype"] == "i32" else _pm1(g, batch, n)
        st["y"] = torch.empty_like(st["x"])
    elif kind in ("fft", "fft_pair", "fft_tc"):
        st["x"] = _complex(g, batch, n)
        st["y"] = torch.empty_like(st["x"])
        if kind == "fft_pair":
            st["z"] = torch.empty_like(st["x"])
    else:
        st["sys"] = _systems(g, batch, n)
        st["y"] = torch.empty(batch, n, device=DEV, dtype=torch.float64 if kind == "refined" else torch.float32)
    return st


def run(state):
    kind = state["kind"]
    if kind == "uneven":
        state["batch"].launch()
        return state["outs"]
    n, batch, y = state["n"], state["batch"], state["y"]
    if kind == "scan":
        bp.scan_batched(state["x"], y, n, batch)
    elif kind == "fft":
        bp.fft_batched(state["x"], y, n, batch, state["dir"])
    elif kind == "fft_pair":
        bp.fft_batched(state["x"], y, n, batch, -1)
        bp.fft_batched(y, state["z"], n, batch, 1)
        return [y, state["z"]]
    elif kind == "fft_tc":
        bp.fft_tc_batched(state["x"], y, n, batch, state["dir"],
                          bp.TC_F16 if state["precision"] == "f16" else bp.TC_BF16)
    elif kind == "tridiag":
        bp.tridiag_batched(*state["sys"], y, n, batch)
    else:
        bp.tridiag_refined(*state["sys"], y, n, batch, tol=state["tol"])
    return [y]


# ----------------------------------------------------------- work and values

def work(case):
    kind = case["kind"]
    if kind == "uneven":
        todo = _uneven_counts(case)
        return {"bytes": sum(n * m * (8, 16, 20)[op] for op, n, m in todo),
                "flops": sum(int(n * m * (1, 5 * math.log2(n), 8)[op]) for op, n, m in todo)}
    n, total = case["n"], case["n"] * case["batch"]
    fft = int(5 * total * math.log2(n))
    return {
        "scan": {"bytes": 8 * total, "flops": total},
        "fft": {"bytes": 16 * total, "flops": fft},
        "fft_pair": {"bytes": 24 * total, "flops": 2 * fft},  # input once, spectrum and result once
        "fft_tc": {"bytes": 16 * total, "flops": fft},
        "tridiag": {"bytes": 20 * total, "flops": 8 * total},
        "refined": {"bytes": 24 * total, "flops": 2 * 8 * total + 13 * total},
    }[kind]


def _exact_scan(x):
    if x.dtype == torch.int32:
        return torch.cumsum(x.long(), dim=1).to(torch.int32)  # wraps modulo 2^32
    return torch.cumsum(x.double(), dim=1)


def _exact_fft(x, direction):
    x = x.to(torch.complex128)
    return torch.fft.fft(x, dim=1) if direction < 0 else torch.fft.ifft(x, dim=1, norm="forward")


def _exact_solve(a, b, c, d):
    """Thomas' algorithm in float64, all systems at once."""
    a, b, c, d = (t.double().t().contiguous() for t in (a, b, c, d))
    n = b.shape[0]
    for i in range(1, n):
        w = a[i] / b[i - 1]
        b[i] -= w * c[i - 1]
        d[i] -= w * d[i - 1]
    d[n - 1] /= b[n - 1]
    for i in range(n - 2, -1, -1):
        d[i] = (d[i] - c[i] * d[i + 1]) / b[i]
    return d.t().contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        fns = (_exact_scan, lambda x: _exact_fft(x, -1), _exact_solve)
        return [fns[op](*ins) for op, _, _, ins in _uneven_problems(case, seed)]
    n, batch = case["n"], case["batch"]
    g = _gen(seed)
    if kind == "scan":
        return [_exact_scan(_ints(g, batch, n) if case["dtype"] == "i32" else _pm1(g, batch, n))]
    if kind == "fft_pair":
        x = _complex(g, batch, n)
        return [_exact_fft(x, -1), x.to(torch.complex128) * n]
    if kind in ("fft", "fft_tc"):
        return [_exact_fft(_complex(g, batch, n), case["dir"])]
    return [_exact_solve(*_systems(g, batch, n))]
