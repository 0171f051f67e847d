"""The autotuner leaves the table alone where the call it is asked about takes
a kernel that has no configuration: many segments, rows by groups of lanes, and
axis shapes whose splits are shared inside a block."""
import pytest

from paper_1710_07358_gb300 import pr

pytestmark = pytest.mark.gpu

# a configuration that no measurement would choose, so that a kept one is seen
ODD = dict(block=128, blocks_per_sm=1, unroll=4, vec_bytes=16)
ODD_AXIS = dict(block=64, blocks_per_sm=8, unroll=4, vec_bytes=32)


def tuned(kind, n, odd, call):
    old = pr.get_config(kind, "f32", "max", "plain", n)
    try:
        pr.set_config(kind, "f32", "max", "plain", n, odd)
        best = call()
        return best, pr.get_config(kind, "f32", "max", "plain", n)
    finally:
        pr.set_config(kind, "f32", "max", "plain", n, old)


def test_many_segments():
    import torch
    x = torch.randn(9000 * 300, device="cuda")
    off = torch.arange(9001, dtype=torch.int64, device="cuda") * 300
    assert tuned("segmented", 9000, ODD, lambda: pr.autotune("segmented", x, "max", offsets=off)) == (ODD, ODD)


def test_rows_by_groups():
    import torch
    x = torch.randn(3000, 1000, device="cuda")
    assert tuned("rows", x.numel(), ODD, lambda: pr.autotune("rows", x, "max")) == (ODD, ODD)


def test_shared_axis_splits():
    import torch
    x = torch.randn(64, 577, 768, device="cuda")
    assert tuned("axis", x.numel(), ODD_AXIS, lambda: pr.autotune("axis", x, "max", dim=1)) == (ODD_AXIS, ODD_AXIS)


def test_calls_that_use_their_configuration_are_tuned():
    import torch
    x = torch.randn(20, 1 << 19, device="cuda")
    best, kept = tuned("rows", x.numel(), ODD, lambda: pr.autotune("rows", x, "max"))
    assert best == kept and best != ODD
    y = torch.randn(2000, 300, 1024, device="cuda")        # enough columns: no splits
    best, kept = tuned("axis", y.numel(), ODD_AXIS, lambda: pr.autotune("axis", y, "max", dim=1))
    assert best == kept
