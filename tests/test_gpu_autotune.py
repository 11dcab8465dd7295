"""What the autotuner installs, seen by a withheld publish: a block of 4,000 bytes
is one tile of 4,096 keys, whose pass waits for nothing, or four of 1,024, whose
waits run out after the 2,000 polls allowed."""
from __future__ import annotations

import json

import pytest

from paper_1109_2348_gb300 import F_GRAPH, Plan, _lib, datagen

from gpu_util import assert_matches_oracle, batch_from_blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, F_GRAPH])
@pytest.mark.parametrize("tile, chosen, small", [(0, 4096, True), (0, 2048, False), (4096, 4096, False)])
def test_tuned_plan_keeps_the_default_tiles(tmp_path, flags, tile, chosen, small):
    """A choice of 8 bits and 4,096 keys read from the cache leaves a plan whose
    tile size was open with the library's default, small tiles for small batches
    included; another choice, or a plan with a size of its own, is fixed."""
    import torch
    buf, off = batch_from_blocks([datagen.block(datagen.UNIFORM, 17, 4000)])
    cache = tmp_path / "tune.jsonl"
    cache.write_text(json.dumps({"gpu": torch.cuda.get_device_name(0),
                                 "key": f"blocks=1;bytes=4000;max_block=4000;flags={flags}", "radix_bits": 8,
                                 "tile_keys": chosen, "round_radix_bits": 0, "ms": 0.1}) + "\n")
    d_in = torch.from_numpy(buf).cuda()
    L, p = torch.empty_like(d_in), torch.empty(1, dtype=torch.int32, device="cuda")
    with Plan(max_blocks=1, max_total_bytes=4000, max_block_bytes=4000, flags=flags, tile_keys=tile) as plan:
        assert plan.autotune(d_in, off, L, p, cache_path=str(cache))[:2] == (8, chosen)
        assert len(cache.read_text().splitlines()) == 1  # read, not swept
        plan.debug_waits(2000, True)
        rc = plan.forward_into(d_in, off, L, p, raise_on_error=False)
        want = _lib.BWT_ETIMEOUT if small or chosen < 4000 else _lib.BWT_OK
        assert (rc or plan.last_status()) == want
        plan.debug_waits(0, False)
        plan.set_radix(8, 4096)  # asked for by name: fixed
        plan.debug_waits(2000, True)
        rc = plan.forward_into(d_in, off, L, p, raise_on_error=False)
        assert (rc or plan.last_status()) == _lib.BWT_OK
        plan.debug_waits(0, False)
        plan.forward_into(d_in, off, L, p)
        assert plan.last_status() == _lib.BWT_OK
        assert_matches_oracle(buf, off, L.cpu().numpy(), p.cpu().numpy(), "after the timeouts")
