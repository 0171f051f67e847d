"""How far axis reductions whose blocks' warps share a row split may be from
the exact value, by bounds derived from the order in which a lane takes a
column's elements."""
import numpy as np
import pytest

from paper_1710_07358_gb300 import pr
from gpu_helpers import to_device

pytestmark = pytest.mark.gpu


def planted(outer, n, inner, dtype, big, small):
    """Columns of `small` with one `big` each, at every row in turn."""
    import torch
    x = torch.full((outer, n, inner), small, dtype=torch.float64)
    o, i = torch.arange(outer)[:, None], torch.arange(inner)[None, :]
    x[o, (o * 101 + i * 37) % n, i] = big
    return x.to(pr.torch_dtype(dtype)).cuda(), big + (n - 1) * small


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("outer,n,inner", [(64, 577, 768), (32, 1024, 768), (1, 5000, 4096), (100, 1500, 64), (60, 1024, 128)])
def test_fp64_combine_columns_beside_one_large_element(dtype, outer, n, inner):
    """Each small element is half a unit in the last place of the large one.  It
    may be lost where it meets the large one in a pair of rows (one); a lane's
    sum keeps what it loses, the rest adds up in fp64, and the result rounds
    once (one more)."""
    big, small = 2.0 ** 15, 2.0 ** -9
    x, want = planted(outer, n, inner, dtype, big, small)
    got = pr.reduce_axis(x, "sum", 1, precision="fp64_combine").double()
    assert float((got - want).abs().max()) <= 2 * small


@pytest.mark.parametrize("outer,n,inner", [(1, 5000, 4096), (16, 4096, 512)])
def test_fp64_columns_after_a_large_element(outer, n, inner):
    """The large element in row 0, then 31 rows of ones, a quarter unit in its
    last place each, then zeros: four rows of ones are exact, so only the three
    that share the large element's step may be lost, and two where the rows of
    a second warp join (a chain would lose all 31)."""
    import torch
    x = torch.zeros(outer, n, inner, dtype=torch.float64, device="cuda")
    x[:, :32] = 1.0
    x[:, 0] = 2.0 ** 54
    got = pr.reduce_axis(x, "sum", 1) - 2.0 ** 54
    assert float((got - 31).abs().max()) <= 3 + 2


@pytest.mark.parametrize("op", ["sum", "prod"])
@pytest.mark.parametrize("precision", ["plain", "fp64_combine"])
def test_columns_with_special_values(op, precision):
    """Infinities, NaN and zeros of both signs at every row of a column, in the
    shared splits."""
    import torch
    if op == "prod" and precision != "plain":
        pytest.skip("a product has no such mode")
    outer, n, inner = 64, 577, 768
    x = torch.ones(outer, n, inner)
    place = torch.arange(inner) * 7 % n
    for o, v in enumerate((torch.inf, -torch.inf, torch.nan, 0.0, -0.0)):
        x[o, place, torch.arange(inner)] = v
    x[5, place, torch.arange(inner)], x[5, (place + 9) % n, torch.arange(inner)] = torch.inf, -torch.inf
    x[6, place, torch.arange(inner)], x[6, (place + 300) % n, torch.arange(inner)] = torch.inf, 0.0
    x[7] = -0.0
    want = x.double().sum(1) if op == "sum" else x.double().prod(1)
    got = pr.reduce_axis(x.cuda(), op, 1, precision=precision).cpu()
    assert torch.equal(got.double().nan_to_num(-7.0, 1e9, -1e9), want.nan_to_num(-7.0, 1e9, -1e9))
    if op == "prod":
        assert torch.equal(torch.signbit(got[want == 0]), torch.signbit(want[want == 0]))


@pytest.mark.parametrize("outer,n,inner", [(64, 577, 768), (32, 1024, 768), (3, 10000, 256), (1, 5000, 4096)])
@pytest.mark.parametrize("aux", [False, True])
def test_column_products_of_factors_near_one(outer, n, inner, aux):
    """Pairs of rows, each joined with its rounding error kept: half of the
    roundings of any order (2^-24 each), and 64 for what combines the partials."""
    import torch
    x = 1 + torch.randn(outer, n, inner, generator=torch.Generator().manual_seed(n)) * (0.3 / n ** 0.5)
    want = x.double().prod(1)
    got = pr.reduce_axis(x.cuda(), "prod", 1, aux=aux)
    got = (got[0] if aux else got).double().cpu()
    assert bool(((got - want).abs() <= (0.5 * n + 64) * 2.0 ** -24 * want.abs()).all())
