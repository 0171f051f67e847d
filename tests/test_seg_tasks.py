"""The task list of many-segment launches: its arithmetic on the CPU (the
header's own functions, compiled as host code) and, on a GPU, offsets that ask
for far more tasks than the list holds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_07358_gb300", "csrc")

SOURCE = """
#include "segtasks.h"
using namespace pr;
// Lists every segment as k_seg_group does, and looks at each record's place as
// k_seg_long does.  Returns the number of records, or -1 - s for the first
// segment s with a record outside the list or over another's.
extern "C" int64_t list(const int64_t* off, int64_t nseg, unsigned tasks, unsigned char* taken, int64_t* unlisted) {
    const int64_t total = off[nseg] - off[0];
    const SegSplit sp = seg_split_lengths(total, nseg, tasks);
    SegCount count = 0;
    int64_t records = 0;
    for (int64_t s = 0; s < nseg; s++) {
        const int64_t len = off[s + 1] - off[s];
        if (len <= sp.most) continue;
        const unsigned n = seg_chunks(len, sp);
        const SegCount first = count;
        count += n;
        const unsigned c = seg_listed(first, n, tasks);
        for (unsigned k = 0; k < c; k++) {
            const unsigned slot = (unsigned)first + k;
            if (slot >= tasks || slot < (unsigned)first || taken[slot]) return -1 - s;
            taken[slot] = 1;
            records++;
        }
        *unlisted += n - c;
    }
    return records;
}
"""


@pytest.fixture(scope="module")
def lister(tmp_path_factory):
    d = tmp_path_factory.mktemp("segtasks")
    src = d / "list.cpp"
    src.write_text(SOURCE)
    so = str(d / "liblist.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(src)], check=True)
    f = ctypes.CDLL(so).list
    f.restype = ctypes.c_int64
    f.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_uint, ctypes.c_void_p, ctypes.c_void_p]

    def go(off, tasks):
        off = np.ascontiguousarray(off, dtype=np.int64)
        taken = np.zeros(tasks, np.uint8)
        unlisted = np.zeros(1, np.int64)
        return f(off.ctypes.data, off.size - 1, tasks, taken.ctypes.data, unlisted.ctypes.data), int(unlisted[0])
    return go


@pytest.mark.parametrize("tasks", [4864, 65536])
@pytest.mark.parametrize("total", [1 << 25, 1 << 28, 1 << 31])
def test_overlapping_segments_stay_inside_the_list(lister, tasks, total):
    """Offsets 0, total, 0, total, ...: more tasks than 32 bits count."""
    each = -(-total // max(8192, total // (tasks // 2) + 1))      # tasks of one segment
    nseg = 2 * ((1 << 32) // each + 5000)
    off = np.zeros(nseg + 1, np.int64)
    off[1::2] = total
    off[-1] = total
    records, unlisted = lister(off, tasks)
    assert records == tasks and records + unlisted > 1 << 32


@pytest.mark.parametrize("tasks", [4864, 65536])
def test_well_formed_segments_all_fit(lister, tasks):
    rng = np.random.default_rng(tasks)
    for nseg, longest in ((512, 1 << 30), (8192, 1 << 20), (100_000, 1 << 14), (1_000_000, 1 << 12), (70_000, 2049)):
        n = np.ceil(np.exp(rng.uniform(0, np.log(longest), nseg))).astype(np.int64)
        if longest == 2049:
            n[:] = longest                       # every segment just long enough
        records, unlisted = lister(np.concatenate([[0], np.cumsum(n)]), tasks)
        assert records >= 0 and unlisted == 0, (nseg, longest)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,op,arg", [("i32", "sum", False), ("f32", "max", True)])
def test_offsets_that_ask_for_too_many_tasks(dtype, op, arg):
    """Refused records raise the error word, and the next call is right."""
    import torch
    from paper_1710_07358_gb300 import pr
    total, nseg = 1 << 25, (1 << 21) + 6
    x = torch.arange(total, device="cuda", dtype=torch.int32).to(pr.torch_dtype(dtype))
    bad = torch.zeros(nseg + 1, dtype=torch.int64, device="cuda")
    bad[1::2] = total
    bad[-1] = total
    pr.segmented_reduce(x, bad, op, argidx=arg)
    assert pr.last_device_error() == 1
    good = torch.arange(nseg + 1, dtype=torch.int64, device="cuda").clamp(max=nseg // 2) * 2
    got = pr.segmented_reduce(x, good, op, argidx=arg)
    pair = x[:nseg // 2 * 2].view(-1, 2)
    if arg:
        assert torch.equal(got[0][:nseg // 2], pair[:, 1])
        assert torch.equal(got[1][:nseg // 2], (pair[:, 1] > pair[:, 0]).long())
    else:
        assert torch.equal(got[:nseg // 2], pair.sum(1)) and bool((got[nseg // 2:] == 0).all())
    assert pr.last_device_error() == 0
