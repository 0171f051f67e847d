"""Many segments at once: the kernels for short and long ones (k_seg_group,
k_seg_long) and the hand-over of k_segmented, every form against the tiles of
k_segmented, which the same segments take in small slices that each hold one
segment too long for the hand-over; samples against the oracle."""
import threading

import numpy as np
import pytest

import oracle
from paper_1710_07358_gb300 import pr, synth
from gpu_helpers import prod_rel_bound, same_float, sum_bound, to_device, values_of
from test_gpu_groups import FORMS, call, values

pytestmark = pytest.mark.gpu

SLICE = 400      # segments: fewer than any launch of the other kernels takes
LONGER = 8300    # elements: more than the hand-over takes


def lengths(kind, nseg, seed):
    rng = np.random.default_rng(seed)
    n = {"tiny": rng.integers(0, 4, nseg), "short": np.floor(rng.exponential(24, nseg)).astype(np.int64),
         "middle": rng.integers(1, 700, nseg), "skewed": np.minimum(rng.pareto(1.1, nseg) * 4, 5000).astype(np.int64)}[kind]
    n[:3] = 0                                    # empty at both ends
    n[-2:] = 0
    n[SLICE // 2::SLICE] = LONGER
    return n.astype(np.int64)


def general(x, off, dtype, op, precision, aux):
    """The segments in slices that take the tile kernel, one launch each."""
    import torch
    outs, mores = [], []
    nseg = off.numel() - 1
    for s in range(0, nseg, SLICE):
        part = off[s:min(s + SLICE, nseg) + 1].contiguous()
        o, m = call(lambda **k: pr.segmented_reduce(x, part, op, precision=precision, **k), part.numel() - 1, dtype, op, aux)
        outs.append(o.clone())
        mores.append(None if m is None else m.clone())
    return torch.cat(outs), (None if mores[0] is None else torch.cat(mores))


@pytest.mark.parametrize("dtype,op,precision,aux", FORMS)
def test_many_segments_match_the_tiles(dtype, op, precision, aux):
    import torch
    for kind, offset in (("tiny", 1), ("short", 0), ("short", 3), ("middle", 1), ("skewed", 0)):
        nseg = 8192 + 7
        n = lengths(kind, nseg, 5)
        if kind == "short":
            n[100] = 20000                       # several chunks
            n[4000] = 8192 * 70 + 11             # and more than one group of 64
        off = torch.from_numpy(synth.offsets_from_lengths(n) + (3 if offset else 0)).cuda()
        total = int(off[-1]) + 2
        x = to_device(values(dtype, op, total, 11 + offset), dtype, offset)
        if aux == "aux":
            x[::97] = 0
        a, am = call(lambda **k: pr.segmented_reduce(x, off, op, precision=precision, **k), nseg, dtype, op, aux)
        b, bm = general(x, off, dtype, op, precision, aux)
        count = torch.from_numpy(np.maximum(n, 1)).cuda().double()
        if op == "sum" and dtype in ("f32", "f16", "bf16", "f64"):
            c = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), x.double().abs().cumsum(0)])
            s = c[off[1:]] - c[off[:-1]] + 1e-9 * c[-1] / len(n)     # (the running sum's own rounding)
            u = (count + 2) * 2.0 ** -53 if dtype == "f64" else 2.0 ** -24 if precision == "compensated" else 1e-6
            assert bool(((a.double() - b.double()).abs() <= 2 * u * s).all()), (kind, offset)
        elif op == "prod" and dtype in ("f32", "f16", "bf16", "f64"):
            u = (count + 1) * (2.0 ** -53 if dtype == "f64" else 2.0 ** -24)
            ok = ((a.double() - b.double()).abs() <= 2 * u * b.double().abs()) | (a == b) | (a.isnan() & b.isnan())
            assert bool(ok.all()), (kind, offset)
            if aux == "aux":
                pa, pb = pr.prod_aux_fields(am), pr.prod_aux_fields(bm)
                assert bool((((pa[0] - pb[0]).abs() <= 2 * u * pb[0].abs()) | (pa[0] == pb[0])).all()), (kind, offset)
                assert torch.equal(pa[1], pb[1]) and torch.equal(pa[2], pb[2]), (kind, offset)
        else:
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), (kind, offset)
            assert am is None or torch.equal(am, bm), (kind, offset)
        assert pr.last_device_error() == 0


@pytest.mark.parametrize("nseg", [1, 33, 300, 5000, 9000])
@pytest.mark.parametrize("dtype,op,arg", [("f32", "sum", False), ("f32", "max", True), ("bf16", "min", True), ("i64", "sum", False)])
def test_short_segments_match_the_oracle(nseg, dtype, op, arg):
    """The hand-over (fewer segments) and k_seg_group, on sampled segments."""
    import torch
    n = np.floor(np.random.default_rng(nseg).exponential(40, nseg)).astype(np.int64)
    n[nseg // 2] = 700
    off = synth.offsets_from_lengths(n)
    x = values(dtype, op, int(off[-1]), 3)
    got, idx = call(lambda **k: pr.segmented_reduce(to_device(x, dtype, 1), torch.from_numpy(off).cuda(), op, **k), nseg, dtype,
                    op, "arg" if arg else "")
    got = values_of(got, pr.out_dtype_name(dtype, op))
    for s in list(range(0, nseg, max(1, nseg // 150))) + [nseg // 2, nseg - 1]:
        seg = x[off[s]:off[s + 1]]
        if arg:
            v, i = oracle.argext(seg, dtype, op)
            assert same_float(got[s], v) and int(idx[s]) == i, s
        elif dtype == "i64":
            assert got[s] == (oracle.reduce(seg, dtype, op) if seg.size else 0), s
        else:
            assert oracle.sum_error(seg, dtype, got[s]) <= sum_bound(seg, dtype) if seg.size else got[s] == 0.0, s


def workload(seed=1):
    import torch
    n = lengths("short", 9000, seed)
    n[77] = 30000
    off = torch.from_numpy(synth.offsets_from_lengths(n)).cuda()
    x = torch.from_numpy(synth.uniform_i32(int(off[-1]), seed)).cuda()
    c = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), x.to(torch.int64).cumsum(0)])
    return x, off, c[off[1:]] - c[off[:-1]]


def test_many_segments_malformed_offsets_and_the_next_call():
    import torch
    x, off, want = workload()
    bad = off.clone()
    bad[5000], bad[5001] = off[5001], off[4000]
    bad[8000] = off[-1]
    pr.segmented_reduce(x, bad, "sum")
    assert pr.last_device_error() == 1
    for _ in range(2):
        assert torch.equal(pr.segmented_reduce(x, off, "sum"), want)
    assert pr.last_device_error() == 0


def test_many_segments_second_launch_fails():
    import torch
    x, off, want = workload()
    assert torch.equal(pr.segmented_reduce(x, off, "sum"), want)
    pr.inject_fault("launch", 1)
    with pytest.raises(pr.PrError) as e:
        pr.segmented_reduce(x, off, "sum")
    assert e.value.status == 3 and not pr.inject_fault("none")
    assert torch.equal(pr.segmented_reduce(x, off, "sum"), want)


def test_many_segments_graph_threads_and_streams():
    import torch
    x, off, want = workload()
    s = torch.cuda.Stream()
    out = torch.empty_like(want)
    with torch.cuda.stream(s):
        pr.prepare(s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):              # captured at once: nothing is allocated
        pr.check(pr.pr_segmented_reduce(x.data_ptr(), off.data_ptr(), 9000, pr.DTYPES["i32"], 0, out.data_ptr(), s.cuda_stream))
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    work = [workload(k) for k in range(4)]           # two threads a stream
    torch.cuda.synchronize()
    bad = []

    def go(k):
        st = (torch.cuda.default_stream(), s)[k % 2]
        with torch.cuda.stream(st):
            for _ in range(40):
                r = pr.segmented_reduce(work[k][0], work[k][1], "sum")
                if not torch.equal(r, work[k][2]):
                    bad.append(k)
    ts = [threading.Thread(target=go, args=(k,)) for k in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad
