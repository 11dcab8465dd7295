"""Bounded waits that run out (the first tile's look-back words withheld, a
limit of 2,000 polls): the call returns BWT_ETIMEOUT, and the next call on the
same plan, with the knob off, is exact."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1109_2348_gb300 import F_GRAPH, F_LEARNED, Plan, _lib, datagen, model

from gpu_util import assert_matches_oracle, batch_from_blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [F_LEARNED, F_LEARNED | F_GRAPH])
def test_learned_batch_with_plain_and_bucketed_blocks(flags):
    """A run-heavy block of many tiles takes the plain passes, whose waits run
    out; in the graph the chunk sorts of the uniform blocks run beside them, and
    so do the passes over a bucket of 30,000 equal bytes, whose waits run out
    too."""
    import torch
    blocks = [datagen.block(datagen.RUNS16, 3, 200_000), datagen.block(datagen.UNIFORM, 4, 300_000),
              np.concatenate([np.full(30_000, 65, dtype=np.uint8), datagen.block(datagen.UNIFORM, 5, 150_000)]),
              datagen.block(datagen.UNIFORM, 6, 77_777)]
    buf, off = batch_from_blocks(blocks)
    d_in = torch.from_numpy(buf).cuda()
    with Plan(max_blocks=4, max_total_bytes=buf.size, max_block_bytes=300_000, flags=flags) as plan:
        model.install(plan, model.equal_width_splitters())
        L = torch.empty_like(d_in)
        p = torch.empty(4, dtype=torch.int32, device="cuda")
        plan.debug_waits(2000, True)
        rc = plan.forward_into(d_in, off, L, p, raise_on_error=False)
        assert (rc or plan.last_status()) == _lib.BWT_ETIMEOUT
        plan.debug_waits(0, False)
        assert plan.forward_into(d_in, off, L, p) == _lib.BWT_OK
        assert plan.last_status() == _lib.BWT_OK
        st = plan.stats()
        assert st["blocks_routed_plain"] == 1 and st["buckets_overflowed"] >= 1, st
        assert_matches_oracle(buf, off, L.cpu().numpy(), p.cpu().numpy(), "after the timeout")


@pytest.mark.parametrize("tile", [0, 1024, 4096])
def test_inverse(tile):
    """The inverse's byte sort has a look-back of its own; the walks after it
    end only on a permutation, so they leave when it has failed. Tiles of 1,024
    rows (a small batch, or asked for) and of 4,096."""
    import torch
    blocks = [datagen.block(datagen.MARKOV3_Z96, 8, 40_001), datagen.block(datagen.UNIFORM, 9, 20_000)]
    buf, off = batch_from_blocks(blocks)
    d_in = torch.from_numpy(buf).cuda()
    out = torch.zeros_like(d_in)
    with Plan(max_blocks=2, max_total_bytes=buf.size, max_block_bytes=40_001, tile_keys=tile) as plan:
        L, p = plan.forward(d_in, off)
        plan.debug_waits(2000, True)
        assert plan.inverse_into(L, off, p, out, raise_on_error=False) == _lib.BWT_ETIMEOUT
        plan.debug_waits(0, False)
        assert plan.inverse_into(L, off, p, out, raise_on_error=False) == _lib.BWT_OK
    assert torch.equal(out, d_in)
