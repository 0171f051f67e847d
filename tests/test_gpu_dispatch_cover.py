"""Kernels that the dispatch rules left without a test of their own: long rows
(k_rows) of every type, the gradient of long rows (k_backward), the shared
axis splits with several rows a warp step, and the axis gradient by narrow and
by many-row columns.  The shapes' dispatch arithmetic is restated where a shape
has to reach one kernel, for the number of SMs there is."""
import numpy as np
import pytest

import oracle
from paper_1710_07358_gb300 import pr, synth
from gpu_helpers import Guarded, prod_rel_bound, same_float, sum_bound, to_device, values_of
from test_gpu_groups import FORMS, call, values

pytestmark = pytest.mark.gpu


def sm_count():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("dtype,op,aux", [("bf16", "sum", ""), ("f16", "max", "arg"), ("bf16", "min", "arg"), ("f64", "sum", ""),
                                          ("f64", "prod", ""), ("f64", "prod", "aux"), ("f64", "min", "arg"), ("i32", "sum", ""),
                                          ("i32", "max", "arg"), ("u32", "xor", ""), ("i64", "sum", ""), ("i64", "min", "arg")])
def test_long_rows_of_every_type(dtype, op, aux):
    """17 rows of more than 4096 vectors: fewer rows than SMs."""
    cols = 4097 * (32 // pr.ELEM_SIZE[dtype])
    rows = 17
    assert rows * 3 < sm_count() * 5
    x = values(dtype, op, rows * cols, 31)
    if aux == "aux":
        x = x.copy()
        x[5::cols] = 0                                     # one zero in every row
        x[9:9 * cols:cols] = 0                             # a second one in some
    t = to_device(x, dtype).view(rows, cols)
    got, more = call(lambda **k: pr.reduce_rows(t, op, **k), rows, dtype, op, aux)
    got = values_of(got, pr.out_dtype_name(dtype, op))
    if aux == "aux":
        p_nz, zc, zi = (v.cpu().numpy() for v in pr.prod_aux_fields(more))
    for r in range(rows):
        row = x[r * cols:(r + 1) * cols]
        if op == "sum" and dtype in ("bf16", "f64"):
            assert oracle.sum_error(row, dtype, got[r]) <= sum_bound(row, dtype), r
        elif aux == "aux":
            wp, wz, wi = oracle.prod_aux(row, dtype)
            assert zc[r] == wz and zi[r] == wi and abs(p_nz[r] - wp) <= prod_rel_bound(cols, dtype) * abs(wp), r
        elif op == "prod":
            want = oracle.reduce(row, dtype, op)
            assert abs(got[r] - want) <= prod_rel_bound(cols, dtype) * abs(want), r
        elif aux == "arg":
            v, i = oracle.argext(row, dtype, op)
            assert same_float(float(got[r]), float(v)) and int(more[r]) == i, r
        else:
            assert got[r] == oracle.reduce(row, dtype, op), r


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("op", ["sum", "max", "prod"])
@pytest.mark.parametrize("rows,cols,off_x,off_g", [(5, 40001, 0, 0), (5, 40001, 1, 3), (4, 32769, 3, 0), (3, 65536, 0, 1)])
def test_gradient_of_long_rows(dtype, op, rows, cols, off_x, off_g):
    """Rows above 32768, rows off the vector grid, x aligned like grad_in or
    not; products without, with one and with two zeros."""
    import torch
    np_t = np.float32 if dtype == "f32" else np.float64
    x = (1 + 0.001 * synth.normal_f32(rows * cols, cols)).astype(np_t).reshape(rows, cols)
    if op == "prod":
        x[1, cols // 2] = 0
        x[2, 0] = x[2, -1] = 0
    g = synth.normal_f32(rows, 3).astype(np_t)
    t = to_device(x.reshape(-1), dtype, off_x).view(rows, cols)
    _, more = pr.reduce_rows(t, op, argidx=op == "max", aux=op == "prod") if op != "sum" else (None, None)
    buf = Guarded(rows * cols + off_g, t.dtype, fill=7)
    gi = buf.tensor[off_g:]
    pr.reduce_backward(op, t, torch.from_numpy(g).cuda(), argidx=more if op == "max" else None,
                       aux=more if op == "prod" else None, out=gi)
    buf.check()
    assert bool((buf.tensor[:off_g] == 7).all())
    if op == "sum":
        want = np.broadcast_to(g[:, None], x.shape)
    elif op == "max":
        want = np.where(np.arange(cols) == x.argmax(1)[:, None], g[:, None], np_t(0))
    else:
        p_nz, zc, zi = (v.cpu().numpy()[:, None] for v in pr.prod_aux_fields(more))
        assert list(zc[:3, 0]) == [0, 1, 2]
        gp = (g[:, None].astype(np.float64) * p_nz).astype(np_t)
        with np.errstate(divide="ignore"):
            want = np.where(zc == 0, gp / x, np.where((zc == 1) & (np.arange(cols) == zi), gp, np_t(0)))
    assert np.array_equal(gi.cpu().numpy().reshape(rows, cols), want)


# (outer, n, bytes a row) of shared splits: bx < 32 lanes a row (4, 2, 8 and 16),
# four warps a split, and 16 rows a warp and more
SHARED = [(100, 1200, 128), (150, 1500, 64), (60, 1024, 256), (40, 600, 512), (600, 40, 1024)]


def lanes_and_warps(n, row_bytes):
    bx = 1
    while bx < 32 and bx < row_bytes // 32:
        bx *= 2
    most, coop = max(n // (32 // bx * 8), 1), 1
    while coop < 8 and 2 * coop <= most:
        coop *= 2
    return bx, coop


def test_shapes_reach_what_they_are_for():
    reached = [lanes_and_warps(n, b) for _, n, b in SHARED]
    assert {bx for bx, _ in reached} >= {2, 4, 8, 16, 32} and {c for _, c in reached} >= {4, 8}
    for outer, n, b in SHARED:
        assert outer * n * b > 6.8e6                       # inputs below take the plain splits
        assert b % 32 == 0


@pytest.mark.parametrize("dtype,op,precision,aux", FORMS)
def test_shared_splits_with_narrow_rows(dtype, op, precision, aux):
    """Against the row reductions of the transposed input."""
    import torch
    es = pr.ELEM_SIZE[dtype]
    for outer, n, row_bytes in SHARED:
        inner = row_bytes // es
        x = to_device(values(dtype, op, outer * n * inner, n), dtype).view(outer, n, inner)
        if aux == "aux":
            x.view(-1)[::n * inner // 3 + 1] = 0
        count = outer * inner

        def axis(**k):
            for name in ("out", "argidx_out"):
                k[name] = k[name].view(outer, inner)
            return pr.reduce_axis(x, op, 1, precision=precision, **k)
        a, am = call(axis, count, dtype, op, aux)
        t = x.transpose(1, 2).contiguous().view(count, n)
        b, bm = call(lambda **k: pr.reduce_rows(t, op, precision=precision, **k), count, dtype, op, aux)
        what = (outer, n, inner)
        if op == "sum" and dtype in ("f32", "f16", "bf16", "f64"):
            s = t.double().abs().sum(1)
            u = (n + 2) * 2.0 ** -53 if dtype == "f64" else 2.0 ** -23 if precision != "plain" else 1e-6
            assert bool(((a.double() - b.double()).abs() <= 2 * u * s).all()), what
        elif op == "prod" and dtype in ("f32", "f16", "bf16", "f64"):
            u = prod_rel_bound(n, "f64" if dtype == "f64" else "f32")
            assert bool(((a.double() - b.double()).abs() <= 2 * u * b.double().abs()).all()), what
            if aux == "aux":
                pa, pb = pr.prod_aux_fields(am), pr.prod_aux_fields(bm)
                assert bool(((pa[0] - pb[0]).abs() <= 2 * u * pb[0].abs()).all()), what
                assert torch.equal(pa[1], pb[1]) and torch.equal(pa[2], pb[2]), what
        else:
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), what
            assert am is None or torch.equal(am, bm), what


@pytest.mark.parametrize("kind", ["axis", "handed", "group", "long"])
@pytest.mark.parametrize("dtype,op", [("f32", "max"), ("f32", "min"), ("f64", "max"), ("bf16", "min"), ("i32", "max")])
def test_extremes_with_ties_nan_and_zeros(kind, dtype, op):
    """Shared axis splits, the hand-over, staged batches and long segments:
    NaN first or last, infinities, zeros of both signs, ties."""
    import torch
    rng = np.random.default_rng(3)
    count, n = {"axis": (256, 900), "handed": (300, 37), "group": (9000, 37), "long": (8200, 3001)}[kind]
    rows = min(count, 400)
    x = rng.integers(-3, 4, (rows, n)).astype(np.float32)             # ties everywhere
    if dtype != "i32":
        x[1::7] = 0.0
        x[1::7, ::2] = -0.0
        x[2::7, n - 1] = np.nan
        x[3::7, 0] = np.nan
        x[4::7] = -np.inf
        x[5::7, n // 2] = np.inf
        x[6::7] = np.inf
    conv = {"f32": np.float32, "f64": np.float64, "i32": np.int32}
    host = (x.view(np.uint32) >> 16).astype(np.uint16) if dtype == "bf16" else x.astype(conv[dtype])
    t = to_device(host.reshape(-1), dtype).view(rows, n)
    if kind == "axis":
        wide = t.transpose(0, 1).contiguous().view(1, n, rows).expand(64, n, rows).contiguous()
        out, idx = pr.reduce_axis(wide, op, 1, argidx=True)
        assert bool((idx == idx[0]).all())
        out, idx = out[37], idx[37]
    else:
        reps = -(-count // rows)
        data = t.repeat(reps, 1)[:count].reshape(-1)
        off = torch.arange(count + 1, dtype=torch.int64, device="cuda") * n
        out, idx = pr.segmented_reduce(data, off, op, argidx=True)
        plain = pr.segmented_reduce(data, off, op)
        assert torch.equal(plain.view(torch.uint8), out.view(torch.uint8))
        first = torch.arange(count, device="cuda") % rows
        assert torch.equal(idx, idx[first])
        out, idx = out[:rows], idx[:rows]
    vals = values_of(out, dtype)
    for r in range(rows):
        v, i = oracle.argext(host[r], dtype, op)
        assert same_float(float(vals[r]), float(v)) and int(idx[r]) == i, (r, vals[r], v, int(idx[r]), i)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("op", ["sum", "max", "prod"])
@pytest.mark.parametrize("outer,n,inner,offset", [(30, 60000, 8, 0), (200, 9001, 3, 1), (9000, 129, 12, 0), (1, 2100, 20001, 0)])
def test_gradient_by_narrow_columns(dtype, op, outer, n, inner, offset):
    """Columns of one to eight lanes a row with two steps a warp and more."""
    import torch
    sms = sm_count()
    es = 4 if dtype == "f32" else 8
    ve = next((b // es for b in (32, 16) if inner * es % b == 0 and offset == 0), 1)
    qv = inner // ve
    bx = 1
    while bx < 32 and bx < qv:
        bx *= 2
    steps = -(-n // (32 // bx))
    assert outer * -(-qv // bx) * steps // (sms * 64) > (128 if inner == 20001 else 1), "too small for the column form"
    np_t = np.float32 if dtype == "f32" else np.float64
    x = (1 + 0.001 * synth.normal_f32(outer * n * inner, n)).astype(np_t).reshape(outer, n, inner)
    if op == "prod":
        x[:, n // 2, 1::3] = 0
        x[:, 0, 2::3] = 0
        x[:, n - 1, 2::3] = 0
    g = synth.normal_f32(outer * inner, 3).astype(np_t).reshape(outer, inner)
    t, gt = to_device(x.reshape(-1), dtype).view(outer, n, inner), torch.from_numpy(g).cuda()
    _, more = pr.reduce_axis(t, op, 1, argidx=op == "max", aux=op == "prod") if op != "sum" else (None, None)
    buf = Guarded(outer * n * inner + offset, t.dtype, fill=7)
    gi = buf.tensor[offset:]
    pr.reduce_axis_backward(op, t, 1, gt, argidx=more if op == "max" else None, aux=more if op == "prod" else None, out=gi)
    buf.check()
    assert bool((buf.tensor[:offset] == 7).all())
    rows = np.arange(n)[None, :, None]
    if op == "sum":
        want = np.broadcast_to(g[:, None, :], x.shape)
    elif op == "max":
        want = np.where(rows == x.argmax(1)[:, None, :], g[:, None, :], np_t(0))
    else:
        p_nz, zc, zi = (v.cpu().numpy().reshape(outer, 1, inner) for v in pr.prod_aux_fields(more))
        gp = (g[:, None, :].astype(np.float64) * p_nz).astype(np_t)
        with np.errstate(divide="ignore", invalid="ignore"):
            want = np.where(zc == 0, gp / x, np.where((zc == 1) & (rows == zi), gp, np_t(0)))
    assert np.array_equal(gi.cpu().numpy().reshape(x.shape), want)


def test_search_values_beyond_the_float_range():
    """phi where a thread's float32 sums reach 2^115, and with links that are
    not finite: the warp sums' float64 form.  With beta 0, flows of 2^20 (whose
    fourth power float32 holds) and free-flow times of 2^93, every term and
    every sum is exact."""
    import torch
    n = 1 << 14
    flow, time = torch.full((n,), 2.0 ** 20, device="cuda"), torch.full((n,), 2.0 ** 93, device="cuda")
    zero, one = torch.zeros(n, device="cuda"), torch.ones(n, device="cuda")
    phi = pr.beckmann(flow, flow, time, one, [0.0, 1.0], beta=0.0)
    assert phi.tolist() == [n * 2.0 ** 113, n * 2.0 ** 114]
    for bad in (torch.inf, torch.nan):
        x = flow.clone()
        x[7] = bad
        assert not any(np.isfinite(v) for v in pr.beckmann(x, zero, time, one, [0.0, 0.5], beta=0.0).tolist())
