"""Run-length encoding of runs over thousands of tiles: the last run end before
a tile lies in another span of tiles, up to all of them back."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1109_2348_gb300 import Plan

pytestmark = pytest.mark.gpu

MANY = 1 << 26  # 16,384 tiles, 27 to a span


def _encode(plan, d_in, off):
    import torch
    n = d_in.numel()
    chars = torch.empty(n, dtype=torch.uint8, device="cuda")
    lens = torch.empty(n, dtype=torch.int32, device="cuda")
    ro = torch.empty(off.size, dtype=torch.int64, device="cuda")
    start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    ms = []
    for _ in range(8):
        start.record()
        plan.rle_encode_into(d_in, off, chars, lens, ro)
        end.record()
        end.synchronize()
        ms.append(start.elapsed_time(end))
    r = int(ro[-1])
    return chars[:r].cpu().numpy(), lens[:r].cpu().numpy(), ro.cpu().numpy(), min(ms)


@pytest.mark.parametrize("n", [MANY, 5_000_000, 9 * 4096 + 1])
def test_runs_over_many_tiles(n):
    """One run of everything, a run end in the first tile alone, in the last
    alone, and here and there, with blocks that end inside a long run."""
    import torch
    r = np.random.RandomState(n % 1000)
    with Plan(max_blocks=3, max_total_bytes=n, max_block_bytes=n) as plan:
        for ends in ([], [7], [n - 2], np.sort(r.choice(n - 1, 5, replace=False)).tolist()):
            for off in ([0, n], [0, n // 3, n // 3 + 1, n]):
                buf = torch.zeros(n, dtype=torch.uint8, device="cuda")
                for k, e in enumerate(ends):
                    buf[e + 1:] = k + 1
                cuts = np.unique(np.concatenate([np.array(ends, dtype=np.int64) + 1, np.array(off[1:], dtype=np.int64)]))
                chars, lens, ro, _ = _encode(plan, buf, np.array(off, dtype=np.uint64))
                assert np.array_equal(lens, np.diff(np.concatenate([[0], cuts])))
                assert np.array_equal(chars, buf[torch.from_numpy(cuts - 1).cuda()].cpu().numpy())
                assert np.array_equal(ro, np.concatenate([[0], np.searchsorted(cuts, off[1:]) + 1]))


def test_one_run_costs_no_more_than_many():
    """The search for the last run end does not grow with the run: one run of
    2^26 bytes takes about as long as runs of a tile each (at most twice, for
    the spans a tile looks through; walking back over the tiles took five times)."""
    import torch
    off = np.array([0, MANY], dtype=np.uint64)
    with Plan(max_blocks=1, max_total_bytes=MANY, max_block_bytes=MANY) as plan:
        one = _encode(plan, torch.full((MANY,), 7, dtype=torch.uint8, device="cuda"), off)
        many = _encode(plan, (torch.arange(MANY, device="cuda") >> 12).to(torch.uint8), off)
    assert one[0].size == 1 and one[1][0] == MANY and many[0].size == MANY // 4096
    assert one[3] <= 2 * many[3], (one[3], many[3])
