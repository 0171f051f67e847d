"""The index of an axis extremum is that of the first NaN, whatever the NaN's
payload and sign, and wherever it lies in a lane's rows."""
import numpy as np
import pytest

import oracle
from paper_1710_07358_gb300 import pr
from gpu_helpers import to_device

pytestmark = pytest.mark.gpu

# NaN bits of float32; the upper halves are bfloat16 NaNs
PAYLOADS = [0x7fc00000, 0xffc00000, 0x7fff0000, 0x7f810000]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("op", ["max", "min"])
@pytest.mark.parametrize("outer,n,inner", [(1, 3, 5), (2, 40, 33), (3, 64, 16), (64, 577, 768)])
def test_first_nan_is_the_index(dtype, op, outer, n, inner):
    import torch
    x = np.random.default_rng(n).standard_normal((outer, n, inner)).astype(np.float32).view(np.uint32)
    if dtype == "f16":
        host, nans = x.view(np.float32).astype(np.float16).view(np.uint16), [0x7e00, 0xfe00, 0x7fff, 0x7c01]
    elif dtype == "bf16":
        host, nans = (x >> 16).astype(np.uint16), [b >> 16 for b in PAYLOADS]
    else:
        host, nans = x.copy(), PAYLOADS
    col = np.arange(inner)
    first = (col * 5) % n                                  # row 0 among them
    for o in range(outer):
        host[o, first, col] = np.array(nans, host.dtype)[(col + o) % 4]
        later = np.minimum(first + 1 + col % 3, n - 1)     # a second NaN, often the next row
        host[o, later, col] = np.array(nans, host.dtype)[(col + o + 1) % 4]
    t = to_device((host.view(np.float32) if dtype == "f32" else host).reshape(-1), dtype).view(outer, n, inner)
    out, idx = pr.reduce_axis(t, op, 1, argidx=True)
    assert bool(out.isnan().all())
    assert torch.equal(idx.cpu(), torch.from_numpy(first).expand(outer, inner))
    v, i = oracle.argext(np.ascontiguousarray(host[0, :, 0]).view(np.float32) if dtype == "f32" else host[0, :, 0].copy(), dtype, op)
    assert np.isnan(v) and i == first[0]
