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
