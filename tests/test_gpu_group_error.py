"""How far rows and segments reduced by groups of lanes may be from the exact
value, by bounds derived from the order in which a lane takes its elements."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1710_07358_gb300 import pr
from gpu_helpers import to_device, values_of

pytestmark = pytest.mark.gpu

# (segments, elements of each), by rows and by segments: one lane to a block a
# row; the hand-over of k_segmented, staged and direct batches, long segments
ROWS = [(3000, 17), (20000, 63), (2600, 120), (2600, 121), (1200, 1000), (1200, 1001), (400, 4100), (260, 8192)]
SEGMENTS = [(300, 23), (300, 1000), (5000, 61), (9000, 23), (9000, 60), (9000, 200), (8300, 2500)]


def reduced(x, count, each, dtype, op, offset, rows, **k):
    """The result of every row, or of every segment of equal length."""
    import torch
    t = to_device(x, dtype, offset)
    if rows:
        out = pr.reduce_rows(t.view(count, each), op, **k)
    else:
        out = pr.segmented_reduce(t, torch.arange(count + 1, dtype=torch.int64, device="cuda") * each, op, **k)
    return out[0] if isinstance(out, tuple) else out


@pytest.mark.parametrize("rows,count,each", [(True,) + s for s in ROWS] + [(False,) + s for s in SEGMENTS])
@pytest.mark.parametrize("aux", [False, True])
def test_fp64_products_round_once(rows, count, each, aux):
    """n factors merge on the integer pipes, under 3 * 2^-63 each, and the
    result rounds to double once (2^-53)."""
    rng = np.random.default_rng(each)
    x = 1 + 0.5 * rng.random(count * each) - 0.25 * (rng.random(count * each) < 0.5)
    for offset in (0, 1):
        got = values_of(reduced(x, count, each, "f64", "prod", offset, rows, aux=aux), "f64")
        bound = (Fraction(1, 2 ** 53) + Fraction(3 * each, 2 ** 63)) * (1 + Fraction(1, 2 ** 20))
        for r in range(0, count, max(1, count // 12)):
            num, den = 1, 1
            for v in x[r * each:(r + 1) * each]:
                a, b = float(v).as_integer_ratio()
                num, den = num * a, den * b
            exact = Fraction(num, den)
            if exact >= Fraction(2) ** 1024:
                assert got[r] == np.inf, (r, offset)
            else:
                assert abs(Fraction(got[r]) - exact) <= bound * exact, (r, offset)


@pytest.mark.parametrize("rows,count,each", [(True,) + s for s in ROWS] + [(False,) + s for s in SEGMENTS])
@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
def test_fp64_combine_sums_round_once(rows, count, each, dtype):
    """The result rounds to fp32 once (2^-24 of itself).  Before that only the
    sum of a lane's rounding errors rounds: with k elements a lane (at most 128
    here) its j-th addition errs by 2^-24 of at most j 2^-24 of the sum of
    magnitudes, k^2 2^-49 in all."""
    import torch
    x = torch.randn(count * each, generator=torch.Generator().manual_seed(each), dtype=torch.float64)
    x = x.to(pr.torch_dtype(dtype))
    want, size = x.view(count, each).double().sum(1).cuda(), x.view(count, each).double().abs().sum(1).cuda()
    host = x.view(torch.int16).numpy().view(np.uint16) if dtype != "f32" else x.numpy()
    for offset in (0, 1):
        got = reduced(host, count, each, dtype, "sum", offset, rows, precision="fp64_combine").double()
        assert bool(((got - want).abs() <= 2.0 ** -24 * want.abs() + min(each, 128) ** 2 * 2.0 ** -49 * size).all()), offset


def test_fp64_combine_infinities_and_nan():
    """An infinity is the sum, opposite ones and NaN are NaN, wherever they lie."""
    import torch
    for each in (23, 200, 4100):
        x = torch.ones(9, each)
        x[1, 0] = x[2, -1] = x[3, each // 2] = torch.inf
        x[4, 1] = -torch.inf
        x[5, 0], x[5, -1] = torch.inf, -torch.inf
        x[6, each // 2] = torch.nan
        for count in (9, 9000):
            t = x.repeat((count + 8) // 9, 1)[:count]
            for rows in (True, False):
                got = reduced(t.numpy().reshape(-1), count, each, "f32", "sum", 1, rows, precision="fp64_combine")
                assert torch.equal(got.cpu().nan_to_num(-7.0, 8.0, 9.0), t.sum(1).nan_to_num(-7.0, 8.0, 9.0)), (each, count, rows)


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("each,levels", [(17, 4), (33, 6)])
def test_sums_beside_one_large_element(dtype, each, levels):
    """Each small element is half a unit in the last place of the large one, so
    every addition to it may lose one.  A vector is a tree of at most eight
    (three roundings), the lane's sum keeps what it loses, its result rounds
    once, and at most four lanes combine (two levels)."""
    count = 200000
    big, small = 2.0 ** 15, 2.0 ** -9
    x = np.full((count, each), small, np.float32)
    x[np.arange(count), np.arange(count) % each] = big
    host = x.astype(np.float16) if dtype == "f16" else (x.view(np.uint32) >> 16).astype(np.uint16) if dtype == "bf16" else x
    want = big + (each - 1) * small
    for offset in (0, 1, 5):
        got = reduced(host.reshape(-1), count, each, dtype, "sum", offset, True).double().cpu().numpy()
        assert np.abs(got - want).max() <= levels * small, offset


def test_fp64_long_segments_beside_one_large_element():
    """Vectors of the small elements are half a unit in the last place of the
    large one: a lane's chain may lose one a step, and blocks of four steps
    end each chain.  Lost at most: the large element's own vector (1), its
    block's other steps (3), and what the chunk's cut vectors and last block
    add up to (6)."""
    import torch
    nseg, each = 8200, 16384
    n = np.ones(nseg, np.int64)
    long = np.arange(5, nseg, 410)
    n[long] = each
    off = np.concatenate([[0], np.cumsum(n)])
    x = np.full(int(off[-1]), 0.5)
    for k, s in enumerate(long):
        x[off[s] + (k * 761) % each] = 2.0 ** 54
    got = pr.segmented_reduce(torch.from_numpy(x).cuda(), torch.from_numpy(off).cuda(), "sum").cpu().numpy()
    assert np.abs(got[long] - 2.0 ** 54 - (each - 1) / 2).max() <= 10 * 2


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("aux", [False, True])
def test_products_of_factors_near_one(dtype, aux):
    """Trees of four and exact joins: three of four factors round (2^-24 each,
    with aux none but the joins), and 64 more cover the lanes', warps' and
    final roundings; the bound without them, n - 1 roundings, is what any
    order gives."""
    import torch
    if aux and dtype != "f32":
        pytest.skip("the gradient's state exists for f32 and f64")
    for rows, count, each in [(True,) + s for s in ROWS] + [(False,) + s for s in SEGMENTS]:
        x = 1 + torch.randn(count * each, generator=torch.Generator().manual_seed(each)) * (0.3 / each ** 0.5)
        x = x.to(pr.torch_dtype(dtype))
        want = x.double().view(count, each).prod(1).cuda()
        host = x.view(torch.int16).numpy().view(np.uint16) if dtype != "f32" else x.numpy()
        got = reduced(host, count, each, dtype, "prod", 1, rows, aux=aux).double()
        assert bool(((got - want).abs() <= (0.75 * each + 64) * 2.0 ** -24 * want.abs()).all()), (rows, count, each)


@pytest.mark.parametrize("op", ["sum", "prod"])
def test_special_values_in_trees(op):
    """Infinities, NaN, zeros of both signs and overflow, wherever they lie."""
    import torch
    for each in (3, 23, 200, 4100):
        x = torch.ones(12, each)
        x[1, 0] = x[2, -1] = x[3, each // 2] = torch.inf
        x[4, 1] = -torch.inf
        x[5, 0], x[5, -1] = torch.inf, -torch.inf
        x[6, each // 2] = torch.nan
        x[7, 1], x[7, 2] = 0.0, torch.inf
        x[8, each // 2] = -0.0
        x[9] = -0.0
        x[10, :3] = 3e38
        x[11, 0] = 1e-30
        x[11, 1] = 1e-30
        want = torch.stack([getattr(torch, op)(r) for r in x]) if op == "sum" else x.double().prod(1).float()
        for count in (12, 9000):
            t = x.repeat((count + 11) // 12, 1)[:count]
            w = want.repeat((count + 11) // 12)[:count]
            for rows in (True, False):
                got = reduced(t.numpy().reshape(-1), count, each, "f32", op, 1, rows).cpu()
                keep = torch.arange(count) % 12 != (10 if op == "sum" else 99)   # (order decides that sum's overflow)
                same = (got == w) | (got.isnan() & w.isnan())
                if op == "sum":
                    same |= (got - w).abs() <= each * 2.0 ** -24 * w.abs()
                assert bool(same[keep].all()), (each, count, rows, got[:12], w[:12])
                if op == "prod":
                    assert torch.equal(torch.signbit(got[w == 0]), torch.signbit(w[w == 0])), (each, count, rows)
