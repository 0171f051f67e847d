"""Rows reduced by groups of lanes (short rows, any length and alignment), and
the flat gradient of short rows: every form the rule sends there against the
general segmented path and the oracle, at the edges of vectors and groups."""
import numpy as np
import pytest

import oracle
from paper_1710_07358_gb300 import pr, synth
from gpu_helpers import Guarded, guarded_like, prod_rel_bound, same_float, sum_bound, to_device, values_of

pytestmark = pytest.mark.gpu

# every (dtype, op, precision, output) the row entry point takes
FORMS = [(d, o, "plain", aux) for d in ("f32", "f16", "bf16", "f64") for o in ("sum", "prod", "max", "min")
         for aux in (("", "arg") if o in ("max", "min") else ("", "aux") if o == "prod" and d in ("f32", "f64") else ("",))]
FORMS += [(d, "sum", p, "") for d in ("f32", "f16", "bf16") for p in ("compensated", "fp64_combine")]
FORMS += [(d, o, "plain", aux) for d in ("i32", "u32", "i64") for o in ("sum", "prod", "max", "min", "and", "or", "xor")
          for aux in (("", "arg") if o in ("max", "min") else ("",))]

# (rows, cols): one lane, part of a vector, every group width 1..32 (grown where
# rows are few), a block per row, and one more or one less than a whole vector
SHAPES = [(1, 1), (7, 3), (129, 31), (3000, 17), (40000, 33), (20000, 63), (9000, 129), (2600, 257), (300, 1000),
          (40, 4097), (257, 8191)]


def values(dtype, op, n, seed):
    if dtype in ("f32", "f16", "bf16"):
        a = 1 + synth.normal_f32(n, seed) * np.float32(2.0 ** -9) if op == "prod" else synth.normal_f32(n, seed)
        a = a.astype(np.float32)
        return a if dtype == "f32" else a.astype(np.float16) if dtype == "f16" else synth.f32_to_bf16_bits(a)
    if dtype == "f64":
        return synth.uniform_f64(n, seed) if op == "prod" else synth.uniform_f64(n, seed, -1, 1)
    return {"i32": synth.uniform_i32, "u32": synth.random_u32, "i64": synth.random_i64}[dtype](n, seed)


def call(f, count, dtype, op, aux):
    """Outputs of one call written into guarded buffers: (values, index or aux bytes)."""
    go, ga, gx = guarded_like(count, pr.out_dtype_name(dtype, op)), guarded_like(count, "i64"), guarded_like(count * 24, "aux")
    f(argidx=aux == "arg", aux=aux == "aux", out=go.tensor, argidx_out=ga.tensor, aux_out=gx.tensor)
    more = ga.check() if aux == "arg" else gx.check() if aux == "aux" else None
    return go.check(), more


@pytest.mark.parametrize("dtype,op,precision,aux", FORMS)
def test_rows_by_groups_match_the_general_path(dtype, op, precision, aux):
    """The same rows as CSR segments go through the segmented kernel; exact
    results agree bit for bit, sums and products within both paths' bounds."""
    import torch
    for rows, cols in SHAPES:
        if cols > 1000 and rows > 100 and dtype not in ("f32", "bf16"):
            continue
        for offset in (0, 1, 3):
            x = to_device(values(dtype, op, rows * cols, rows + cols), dtype, offset)
            if aux == "aux":
                x[::max(cols // 2, 2) * 3 + 1] = 0
            off = torch.arange(rows + 1, dtype=torch.int64, device="cuda") * cols
            a, am = call(lambda **k: pr.reduce_rows(x.view(rows, cols), op, precision=precision, **k), rows, dtype, op, aux)
            b, bm = call(lambda **k: pr.segmented_reduce(x, off, op, precision=precision, **k), rows, dtype, op, aux)
            what = (rows, cols, offset)
            if op == "sum" and dtype in ("f32", "f16", "bf16", "f64"):
                s = x.view(rows, cols).double().abs().sum(1)
                u = (cols + 2) * 2.0 ** -53 if dtype == "f64" else 2.0 ** -24 if precision == "compensated" else 1e-6
                assert bool(((a.double() - b.double()).abs() <= 2 * u * s).all()), what
            elif op == "prod" and dtype in ("f32", "f16", "bf16", "f64"):
                u = prod_rel_bound(cols, "f64" if dtype == "f64" else "f32")
                assert bool(((a.double() - b.double()).abs() <= 2 * u * b.double().abs()).all()), what
                if aux == "aux":
                    pa, pb = pr.prod_aux_fields(am), pr.prod_aux_fields(bm)
                    assert bool(((pa[0] - pb[0]).abs() <= 2 * u * pb[0].abs()).all()), what
                    assert torch.equal(pa[1], pb[1]) and torch.equal(pa[2], pb[2]), what
            else:
                assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), what
                assert am is None or torch.equal(am, bm), what


@pytest.mark.parametrize("dtype,op,aux", [("f32", "sum", ""), ("f32", "max", "arg"), ("bf16", "min", "arg"), ("f64", "prod", ""),
                                          ("i32", "sum", "")])
def test_rows_by_groups_match_the_oracle(dtype, op, aux):
    for rows, cols, offset in ((70, 5, 1), (33, 100, 3), (20, 1000, 0), (9, 4099, 1)):
        x = values(dtype, op, rows * cols, 7 * rows + cols)
        got, idx = call(lambda **k: pr.reduce_rows(to_device(x, dtype, offset).view(rows, cols), op, **k), rows, dtype, op, aux)
        got = values_of(got, pr.out_dtype_name(dtype, op))
        for r in range(rows):
            row = x[r * cols:(r + 1) * cols]
            if dtype == "f32" and op == "sum":
                assert oracle.sum_error(row, dtype, got[r]) <= sum_bound(row, dtype), (r, rows, cols)
            elif op == "prod":
                want = oracle.reduce(row, dtype, op)
                assert abs(got[r] - want) <= prod_rel_bound(cols, dtype) * abs(want), (r, rows, cols)
            elif dtype == "i32":
                assert got[r] == oracle.reduce(row, dtype, op), (r, rows, cols)
            else:
                v, i = oracle.argext(row, dtype, op)
                assert same_float(got[r], v) and int(idx[r]) == i, (r, rows, cols)


def test_rows_by_groups_special_values():
    """NaN, infinities, signed zeros and ties at vector and row ends."""
    import torch
    rows, cols = 50, 37
    x = np.zeros((rows, cols), np.float32)
    x[::2] = -0.0
    x[1, 36] = x[1, 0] = 5.0
    x[2, 36] = np.nan
    x[3, 0] = np.nan
    x[4] = -np.inf
    x[5] = np.inf
    x[6, 20:] = -np.finfo(np.float32).max
    for op in ("max", "min"):
        for offset in (0, 1):
            out, idx = pr.reduce_rows(to_device(x.reshape(-1), "f32", offset).view(rows, cols), op, argidx=True)
            vals = values_of(out, "f32")
            for r in range(rows):
                v, i = oracle.argext(x[r], "f32", op)
                assert same_float(vals[r], v) and int(idx[r]) == i, (op, offset, r)
    s = pr.reduce_rows(to_device(x.reshape(-1), "f32", 1).view(rows, cols), "sum")
    assert torch.isnan(s[2]) and torch.isnan(s[3]) and float(s[4]) == -np.inf and float(s[5]) == np.inf


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("op", ["sum", "max", "prod"])
@pytest.mark.parametrize("rows,cols", [(1, 1), (3000, 1), (1000, 2), (777, 7), (1000, 8), (301, 33), (5, 2047), (3, 8193)])
def test_flat_gradient(dtype, op, rows, cols):
    """Bit for bit the rules' own float expressions, at every alignment of
    grad_in and with x aligned like it or not."""
    import torch
    np_t = np.float32 if dtype == "f32" else np.float64
    x = (1 + 0.1 * synth.normal_f32(rows * cols, rows + cols)).astype(np_t).reshape(rows, cols)
    if op == "prod":                       # rows without, with one and with two zeros
        x[1::3, 0] = 0
        x[2::3, -1] = 0
        x[2::3, 0] = 0
    g = synth.normal_f32(rows, 3).astype(np_t)
    gt = torch.from_numpy(g).cuda()
    for off_x, off_g in ((0, 0), (1, 1), (0, 3)):
        t = to_device(x.reshape(-1), dtype, off_x).view(rows, cols)
        _, more = pr.reduce_rows(t, op, argidx=op == "max", aux=op == "prod") if op != "sum" else (None, None)
        buf = Guarded(rows * cols + off_g, t.dtype, fill=7)
        gi = buf.tensor[off_g:]
        pr.reduce_backward(op, t, gt, argidx=more if op == "max" else None, aux=more if op == "prod" else None, out=gi)
        buf.check()
        assert bool((buf.tensor[:off_g] == 7).all())
        if op == "sum":
            want = np.broadcast_to(g[:, None], x.shape)
        elif op == "max":
            want = np.where(np.arange(cols) == x.argmax(1)[:, None], g[:, None], np_t(0))
        else:
            p_nz, zc, zi = (v.cpu().numpy() for v in pr.prod_aux_fields(more))
            gp = (g.astype(np.float64) * p_nz).astype(np_t)[:, None]
            zc, zi = zc[:, None], zi[:, None]
            with np.errstate(divide="ignore"):
                want = np.where(zc == 0, gp / x, np.where((zc == 1) & (np.arange(cols) == zi), gp, np_t(0)))
        assert np.array_equal(gi.cpu().numpy().reshape(rows, cols), want), (off_x, off_g)
