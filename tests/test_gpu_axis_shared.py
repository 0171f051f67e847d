"""Axis reductions whose blocks' warps share a row split, and the axis gradient
by columns: every form against the row reductions of the transposed input, and
the gradients bit for bit against their own float expressions."""
import numpy as np
import pytest

from paper_1710_07358_gb300 import pr, synth
from gpu_helpers import Guarded, prod_rel_bound, to_device
from test_gpu_groups import FORMS, call, values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,op,precision,aux", FORMS)
def test_shared_splits_match_rows(dtype, op, precision, aux):
    """Short axes of at least 7 MB with whole vectors per row: two, four and
    eight warps a split, columns that leave lanes idle, several rows a warp
    step, one split and more."""
    import torch
    es = pr.ELEM_SIZE[dtype]
    for outer, n, inner in ((8, 960, 1024 // es), (300, 72, 416 // es * 4), (64, 17, 16384 // es), (2000, 33, 128 // es)):
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
            u = (n + 2) * 2.0 ** -53 if dtype == "f64" else 2.0 ** -24 if precision == "compensated" else 1e-6
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


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("op", ["sum", "max", "prod"])
@pytest.mark.parametrize("outer,n,inner,offset", [(40, 1200, 96, 0), (40, 1200, 96, 1), (3, 1501, 1024, 0), (2, 700, 2049, 0),
                                                  (1, 40000, 8, 0), (5, 20000, 3, 1), (30, 1000, 33, 0)])
def test_gradient_by_columns(dtype, op, outer, n, inner, offset):
    import torch
    np_t = np.float32 if dtype == "f32" else np.float64
    x = (1 + 0.1 * synth.normal_f32(outer * n * inner, n)).astype(np_t).reshape(outer, n, inner)
    if op == "prod":                       # columns without, with one and with two zeros
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
