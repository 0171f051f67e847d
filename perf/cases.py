"""The work whose speed counts: what a program that uses this library has it do.

Six kinds of case, each one call (or one forward and backward) through the public
entry points of ``pr`` and ``autograd``:

  plain     a whole array to one value                        pr.reduce / pr.reduce_arg
  segments  the segments of a CSR offsets array               pr.segmented_reduce
  rows      the rows of a matrix                              pr.reduce_rows
  grad      one axis of [outer, n, inner] and its gradient    autograd.reduce + backward
  scan      prefix scan                                       pr.scan
  search    line search on the reduction                      pr.line_search

``listed()`` names twelve of them, ``draw`` takes more from the same ranges: inputs
of up to 1 GiB, n from 2^10 on, rows and segments from a few elements to a million.
"""
import math

import torch

from paper_1710_07358_gb300 import autograd, pr

# A drawn case reads at most as much as the largest listed one, in elements of 4 bytes.
MOST_BYTES = 1 << 30


def listed():
    return [
        # A loss or a norm over a small tensor: one of many such calls in a program's loop,
        # where the cost of a call is what counts.
        dict(name="scalar_small", kind="plain", dtype="f32", op="sum", precision="plain", arg=False, n=1000),
        # The paper's own vector: int32 sum of 5 533 214 elements.
        dict(name="paper_vector", kind="plain", dtype="i32", op="sum", precision="plain", arg=False, n=5_533_214),
        # The benchmark's headline: fp32 sum of 2^28 elements, far beyond L2.
        dict(name="headline_sum", kind="plain", dtype="f32", op="sum", precision="plain", arg=False, n=1 << 28),
        # A long 16-bit sum that must not lose digits, of a ragged length.
        dict(name="precise_bf16", kind="plain", dtype="bf16", op="sum", precision="compensated", arg=False,
             n=100_000_007),
        # The benchmark's batch: 4096 segments, lengths log-uniform up to 2^20.
        dict(name="segments_mixed", kind="segments", dtype="f32", op="sum", arg=False, nseg=4096, spread="log",
             length=1 << 20),
        # Sums over the neighbours of every node of a graph in CSR form: many short
        # segments, some of them empty.
        dict(name="segments_graph", kind="segments", dtype="f32", op="sum", arg=False, nseg=1_000_000, spread="exp",
             length=24),
        # The best of 1000 classes for every sample of a batch, with its index.
        dict(name="rows_argmax", kind="rows", dtype="f32", op="max", arg=True, rows=32768, cols=1000),
        # The benchmark's differentiation workload: 64 rows of 2^20, forward and backward.
        dict(name="grad_wide_max", kind="grad", dtype="f32", op="max", outer=64, n=1 << 20, inner=1),
        # A sum over the features of many samples inside a training step: short rows.
        dict(name="grad_narrow_sum", kind="grad", dtype="f32", op="sum", outer=200_000, n=120, inner=1),
        # Max pooling over the middle axis of [batch, tokens, features], a ragged token count.
        dict(name="grad_axis_max", kind="grad", dtype="f32", op="max", outer=64, n=577, inner=768),
        # Counts to offsets: the step before a compaction or a counting sort.
        dict(name="scan_offsets", kind="scan", dtype="i32", op="sum", exclusive=True, n=20_000_003),
        # The step size of a traffic assignment over a national network's links.
        dict(name="search_links", kind="search", links=1_000_003, power=4, depth=2, tol=1e-6),
    ]


def _between(rng, lo, hi):
    """A whole number, its logarithm uniform on [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["plain", "segments", "rows", "rows", "grad", "grad", "scan", "search"])
    if kind == "plain":
        dtype = rng.choice(["f32", "f32", "f16", "bf16", "f64", "i32", "u32", "i64"])
        if dtype in ("i32", "u32", "i64"):
            op = rng.choice(["sum", "max", "min", "and", "or", "xor"])
        else:
            op = rng.choice(["sum", "sum", "max", "min"])
        half = op == "sum" and dtype in ("f32", "f16", "bf16")
        precision = rng.choice(["plain", "compensated", "fp64_combine"]) if half else "plain"
        return dict(kind=kind, dtype=dtype, op=op, precision=precision, arg=op in ("max", "min") and rng.random() < 0.5,
                    n=_between(rng, 1 << 10, MOST_BYTES // pr.ELEM_SIZE[dtype]))
    if kind == "segments":
        spread = rng.choice(["log", "exp"])
        nseg = _between(rng, 64, 4096) if spread == "log" else _between(rng, 1000, 1_000_000)
        op = rng.choice(["sum", "max"])
        return dict(kind=kind, dtype=rng.choice(["f32", "f32", "bf16", "i32"]), op=op, arg=op == "max" and rng.random() < 0.5,
                    nseg=nseg, spread=spread, length=_between(rng, 64, 1 << 20) if spread == "log" else _between(rng, 4, 64))
    if kind == "rows":
        op = rng.choice(["sum", "max", "min"])
        cols = _between(rng, 16, 1 << 17)
        return dict(kind=kind, dtype=rng.choice(["f32", "f32", "bf16", "f16", "f64", "i32"]), op=op,
                    arg=op != "sum" and rng.random() < 0.5, rows=max(1, _between(rng, 1 << 14, 1 << 26) // cols), cols=cols)
    if kind == "grad":
        inner = 1 if rng.random() < 0.5 else _between(rng, 2, 4096)
        n = _between(rng, 16, 1 << 14)
        return dict(kind=kind, dtype=rng.choice(["f32", "f32", "f32", "f64"]), op=rng.choice(["sum", "max", "prod"]),
                    outer=max(1, _between(rng, 1 << 14, 1 << 25) // (n * inner)), n=n, inner=inner)
    if kind == "scan":
        dtype, op = rng.choice([("i32", "sum"), ("i64", "sum"), ("f32", "max"), ("i32", "max")])
        return dict(kind=kind, dtype=dtype, op=op, exclusive=rng.random() < 0.5, n=_between(rng, 1 << 12, 1 << 26))
    return dict(kind=kind, links=_between(rng, 10_000, 4_000_000), power=rng.choice([4, 4, 5]), depth=rng.choice([1, 2]),
                tol=rng.choice([1e-4, 1e-6]))


def _values(g, shape, dtype, op):
    """Elements as the path meets them: words and flag words, and measured values about zero."""
    if dtype in ("i32", "u32", "i64"):
        wide = dtype == "i64"
        lo, hi = (-(1 << 20), 1 << 20) if op == "sum" and not wide else (-(1 << 62), 1 << 62) if wide else (-(1 << 31), (1 << 31) - 1)
        kind = torch.int64 if wide else torch.int32
        x = torch.randint(lo, hi, shape, generator=g, device="cuda", dtype=kind)
        if op in ("and", "or"):  # flags that every word has, or that none has
            flags = torch.randint(lo, hi, (1,), generator=g, device="cuda", dtype=kind)
            x = x | flags if op == "and" else x & flags
        return x.view(torch.uint32) if dtype == "u32" else x
    if dtype == "f64":
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.randn(shape, generator=g, device="cuda").to(pr.torch_dtype(dtype))


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    s = dict(case)
    if kind == "plain":
        s["x"] = _values(g, (case["n"],), case["dtype"], case["op"])
        if case["op"] == "sum" and case["dtype"] in ("f32", "f16", "bf16", "f64"):
            s["x"].add_(1)  # measurements about a mean of one
    elif kind == "segments":
        if case["spread"] == "log":
            u = torch.rand(case["nseg"], generator=g, device="cuda", dtype=torch.float64)
            lengths = torch.exp(u * math.log(case["length"])).ceil().clamp(1, case["length"])
        else:
            u = torch.rand(case["nseg"], generator=g, device="cuda", dtype=torch.float64)
            lengths = (-case["length"] * torch.log1p(-u)).floor()
        s["offsets"] = torch.zeros(case["nseg"] + 1, device="cuda", dtype=torch.int64)
        s["offsets"][1:] = lengths.to(torch.int64).cumsum(0)
        s["x"] = _values(g, (int(s["offsets"][-1]),), case["dtype"], case["op"])
    elif kind == "rows":
        s["x"] = _values(g, (case["rows"], case["cols"]), case["dtype"], case["op"])
    elif kind == "grad":
        flat = case["inner"] == 1
        shape = (case["outer"], case["n"]) if flat else (case["outer"], case["n"], case["inner"])
        x = _values(g, shape, case["dtype"], case["op"])
        if case["op"] == "prod":  # factors about one, a zero in about every second product
            u = torch.rand(shape, generator=g, device="cuda")
            x = (1 + x * (0.3 / math.sqrt(case["n"]))).masked_fill_(u < 0.5 / case["n"], 0)
        s["x"] = x.requires_grad_()
        s["grad"] = torch.randn(shape[:1] + shape[2:], generator=g, device="cuda", dtype=x.dtype)
    elif kind == "scan":
        if case["op"] == "sum":
            s["x"] = torch.randint(0, 1000, (case["n"],), generator=g, device="cuda", dtype=pr.torch_dtype(case["dtype"]))
        else:
            s["x"] = _values(g, (case["n"],), case["dtype"], case["op"])
    else:
        n = case["links"]

        def uniform(lo, hi):
            return torch.rand(n, generator=g, device="cuda") * (hi - lo) + lo
        cap, t0 = uniform(500, 4000), uniform(0.5, 5)
        flow = cap * uniform(0.2, 1.5)
        target = torch.where(uniform(0, 1) < 0.3, cap * uniform(0, 3), torch.zeros_like(cap))
        s["links"] = (flow, target - flow, t0, cap)
    return s


def run(s):
    kind, op = s["kind"], s.get("op")
    if kind == "plain":
        return pr.reduce_arg(s["x"], op) if s["arg"] else pr.reduce(s["x"], op, precision=s["precision"])
    if kind == "segments":
        return pr.segmented_reduce(s["x"], s["offsets"], op, argidx=s["arg"])
    if kind == "rows":
        return pr.reduce_rows(s["x"], op, argidx=s["arg"])
    if kind == "grad":
        y = autograd.reduce(s["x"], op, dim=1)
        return y.detach(), torch.autograd.grad(y, s["x"], s["grad"])[0]
    if kind == "scan":
        return pr.scan(s["x"], op, exclusive=s["exclusive"])
    return pr.line_search(*s["links"], power=s["power"], tol=s["tol"], depth=s["depth"])


def _segment_total(case):
    """Expected number of elements in all segments."""
    if case["spread"] == "log":
        return case["nseg"] * (case["length"] - 1) / math.log(case["length"])
    return case["nseg"] / math.expm1(1 / case["length"])


def work(case):
    kind = case["kind"]
    if kind == "search":
        # every link's four values once, and an evaluation of each for every step
        steps = pr.golden_iterations(0.0, 1.0, case["tol"]) + 2
        return {"bytes": 16 * case["links"] + 32, "flops": 12 * case["links"] * steps}
    es, out = pr.ELEM_SIZE[case["dtype"]], pr.ELEM_SIZE[pr.out_dtype_name(case["dtype"], case["op"])]
    if kind == "plain":
        return {"bytes": case["n"] * es + out + 8 * case["arg"], "flops": case["n"]}
    if kind == "segments":
        n = _segment_total(case)
        return {"bytes": n * es + case["nseg"] * (8 + out + 8 * case["arg"]), "flops": n}
    if kind == "rows":
        n = case["rows"] * case["cols"]
        return {"bytes": n * es + case["rows"] * (out + 8 * case["arg"]), "flops": n}
    if kind == "grad":
        n, outs = case["outer"] * case["n"] * case["inner"], case["outer"] * case["inner"]
        return {"bytes": 2 * n * es + 2 * outs * es, "flops": 2 * n}
    return {"bytes": case["n"] * (es + out), "flops": case["n"]}


def _exact_grad(x, op, g):
    if op == "sum":
        return [x.sum(1), g.unsqueeze(1).expand_as(x)]
    if op == "max":
        y = x.amax(1)
        place = torch.arange(x.shape[1], device=x.device).view((1, -1) + (1,) * (x.dim() - 2))
        first = torch.where(x == y.unsqueeze(1), place, x.shape[1]).amin(1, keepdim=True)
        return [y, (place == first) * g.unsqueeze(1)]
    zero = x == 0
    zeros = zero.sum(1, keepdim=True)
    others = x.masked_fill(zero, 1).prod(1, keepdim=True)
    gx = torch.where(zeros == 0, others / x, torch.where((zeros == 1) & zero, others, 0.0)) * g.unsqueeze(1)
    return [torch.where(zeros == 0, others, 0.0).squeeze(1), gx]


def exact(case, seed):
    """What run() returns, in 64 bits; whole numbers have no such value."""
    if case["kind"] == "search" or case["dtype"] in ("i32", "u32", "i64"):
        return None  # a search's brackets follow comparisons of rounded sums
    s = prepare(case, seed)
    kind, op = case["kind"], case["op"]
    x = s["x"].detach().double()
    if kind == "grad":
        return _exact_grad(x, op, s["grad"].double())
    if kind == "scan":
        if case["exclusive"]:
            x = torch.cat([torch.full_like(x[:1], -math.inf), x[:-1]])
        return torch.cummax(x, 0).values
    if kind == "plain":
        y = x.sum() if op == "sum" else x.max() if op == "max" else x.min()
    elif kind == "rows":
        y = x.sum(1) if op == "sum" else x.amax(1) if op == "max" else x.amin(1)
    else:
        lengths = s["offsets"].diff()
        which = torch.repeat_interleave(lengths)
        y = torch.full_like(x[:1], 0.0 if op == "sum" else -math.inf).repeat(case["nseg"])
        y = y.index_add_(0, which, x) if op == "sum" else y.scatter_reduce_(0, which, x, "amax")
    return [y, None] if case["arg"] else y
