"""Edges of single kernels against the oracle, byte for byte."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

from paper_1109_2348_gb300 import F_GRAPH, F_LEARNED, Plan, datagen, model
from gpu_util import assert_matches_oracle, batch_from_blocks, gpu_bwt

pytestmark = pytest.mark.gpu


def _rng_bytes(seed, n, lo, hi):
    return np.random.RandomState(seed).randint(lo, hi, n).astype(np.uint8)


def _chunk_sort_blocks(kind):
    if kind == "wide":  # few rotations a chunk: key ranges of up to 64 bits, whose low bits the words drop
        return [_rng_bytes(1, n, 0, 256) for n in (9, 13, 14, 100, 3328, 3329, 5000)]
    if kind == "last_byte":  # prefixes of 7 equal bytes, told apart by the eighth alone, and far beyond it
        unit = _rng_bytes(2, 7, 0, 256)
        rows = [np.concatenate([unit, _rng_bytes(10 + k, 1 + k % 3, 0, 256)]) for k in range(1500)]
        return [np.concatenate(rows), np.concatenate(rows[:300] + [_rng_bytes(3, 40_000, 0, 256)])]
    if kind == "repeats":  # groups of equal prefixes of every small size beside distinct ones
        text = datagen.block(datagen.MARKOV3_Z96, 77, 30_000)
        return [np.concatenate([text, text[100:9000], text[200:2000], text[:5000]]), np.tile(text[:700], 20)]
    return [np.concatenate([_rng_bytes(5, 60_000, 0, 256), np.tile(_rng_bytes(6, 24, 0, 4), 150)]),
            datagen.block(datagen.MUTATED_UNIT, 9, 120_000)]


@pytest.mark.parametrize("kind", ["wide", "last_byte", "repeats", "mixed"])
@pytest.mark.parametrize("table", ["equal", "coarse", "top"])
def test_chunk_sort_words(kind, table):
    """The chunk sort's 64-bit words: dropped key bits, ties and runs of equal
    prefixes, under an equal-width table (52-bit ranges), a coarse one (a few
    wide buckets, so that all three team sizes occur) and one whose splitters
    crowd at both ends of the key space."""
    spl = model.equal_width_splitters()
    if table == "coarse":
        spl = np.sort(np.repeat(spl[::256], 256)[:spl.size])
    elif table == "top":
        half = np.arange(spl.size // 2, dtype=np.uint64)
        spl = np.sort(np.concatenate([half, ~np.uint64(0) - np.arange(spl.size - half.size, dtype=np.uint64)]))
    buf, off = batch_from_blocks(_chunk_sort_blocks(kind))
    sizes = np.diff(off.astype(np.int64))
    with Plan(max_blocks=off.size - 1, max_total_bytes=buf.size, max_block_bytes=int(sizes.max()),
              flags=F_LEARNED | F_GRAPH) as plan:
        model.install(plan, spl)
        L, prim, _ = gpu_bwt(buf, off, plan)
    assert_matches_oracle(buf, off, L, prim, f"{kind}/{table}")


def _mtf_blocks(kind):
    r = np.random.RandomState(21)
    if kind == "edges":  # sizes around a step, a chunk and a chunk's last step, over alphabets of every size
        return [r.randint(0, a, n).astype(np.uint8) for a in (1, 2, 33, 256)
                for n in (1, 31, 32, 33, 63, 511, 512, 513, 1024, 1535, 4097)]
    if kind == "large_chunks":  # 9 MB: 1,024-byte chunks; runs, then every byte value in turn
        b = r.randint(0, 90, 9_000_000).astype(np.uint8)
        b[1_000_000:1_200_000] = 7
        b[5_000_000:5_002_560] = np.tile(np.arange(255, -1, -1), 10)
        return [b, b[:70_001]]
    if kind == "tiny":  # blocks too short for the chunks' lists to fit the key buffers
        return [r.randint(0, 256, 1 + k % 5).astype(np.uint8) for k in range(300)]
    # over 2^24 bytes: recencies that need more than 24 bits; a byte value last seen at the very start
    b = (datagen.block(datagen.RUNS16, 5, 17_000_000) + 1).astype(np.uint8)
    b[:300] = np.arange(300) % 256
    b[-300:] = np.arange(300)[::-1] % 256
    return [b]


@pytest.mark.parametrize("shift_in, shift_out", [(0, 0), (5, 5), (3, 8)])
@pytest.mark.parametrize("kind", ["edges", "tiny", "large_chunks", "over_24_bits"])
def test_mtf_steps_and_chunks(kind, shift_in, shift_out):
    """Move-to-front by 32-byte steps: sizes around steps and chunks, every
    chunk size, and buffers of equal and of different alignment."""
    import torch
    buf, off = batch_from_blocks(_mtf_blocks(kind))
    sizes = np.diff(off.astype(np.int64))
    d_in = torch.zeros(buf.size + 16, dtype=torch.uint8, device="cuda")
    d_in[shift_in:shift_in + buf.size] = torch.from_numpy(buf).cuda()
    d_out = torch.full((buf.size + 32,), 0xEE, dtype=torch.uint8, device="cuda")
    with Plan(max_blocks=off.size - 1, max_total_bytes=buf.size, max_block_bytes=int(sizes.max())) as plan:
        plan.mtf_encode_into(d_in[shift_in:shift_in + buf.size], off, d_out[shift_out:shift_out + buf.size])
    got = d_out.cpu().numpy()
    want = np.concatenate([oracle.mtf_encode(buf[int(off[b]):int(off[b + 1])]) for b in range(off.size - 1)])
    assert np.array_equal(got[shift_out:shift_out + buf.size], want)
    assert (got[:shift_out] == 0xEE).all() and (got[shift_out + buf.size:] == 0xEE).all()  # nothing written outside


def _inverse_blocks(kind):
    r = np.random.RandomState(31)
    if kind == "tiny":  # blocks of a few bytes: more samples than the plan's key buffer holds
        return [r.randint(0, 3, n).astype(np.uint8) for n in r.randint(1, 12, 700)]
    if kind == "strides":  # around a sample (8 rows), a super (64), the stored bytes of a sample (24)
        return [r.randint(0, a, n).astype(np.uint8) for a in (2, 256)
                for n in (1, 7, 8, 9, 23, 24, 25, 63, 64, 65, 127, 129, 511, 513, 4095, 4097)]
    if kind == "periods":  # several cycles; walks far longer than a sample stores
        return [np.tile(r.randint(0, 256, p).astype(np.uint8), k) for p, k in ((1, 3000), (3, 1001), (64, 65), (700, 9))]
    if kind == "many_supers":  # above and below the supers that one CTA ranks in shared memory
        return [r.randint(0, 100, n).astype(np.uint8) for n in (1_048_560, 1_048_640, 1_400_003)]
    return [r.randint(0, 256, (1 << 24) + 77).astype(np.uint8), r.randint(0, 256, 1000).astype(np.uint8)]


@pytest.mark.parametrize("tile", [1024, 2048, 4096])
@pytest.mark.parametrize("kind", ["tiny", "strides", "periods", "many_supers", "over_24_bits"])
def test_inverse_samples_and_supers(kind, tile):
    """GPU forward, then the inverse into a buffer of odd alignment: the
    blocks come back and nothing outside them is written."""
    import torch
    if kind in ("many_supers", "over_24_bits") and tile != 4096:
        pytest.skip("large blocks: one tile size")
    buf, off = batch_from_blocks(_inverse_blocks(kind))
    sizes = np.diff(off.astype(np.int64))
    d_in = torch.from_numpy(buf).cuda()
    out = torch.full((buf.size + 32,), 0xEE, dtype=torch.uint8, device="cuda")
    with Plan(max_blocks=off.size - 1, max_total_bytes=buf.size, max_block_bytes=int(sizes.max()),
              tile_keys=tile) as plan:
        L, prim = plan.forward(d_in, off)
        if kind not in ("many_supers", "over_24_bits"):
            assert_matches_oracle(buf, off, L.cpu().numpy(), prim.cpu().numpy(), kind)
        plan.inverse_into(L, off, prim, out[5:5 + buf.size])
    assert torch.equal(out[5:5 + buf.size], d_in)
    assert bool((out[:5] == 0xEE).all()) and bool((out[5 + buf.size:] == 0xEE).all())


@pytest.mark.parametrize("shift", [0, 3])
@pytest.mark.parametrize("kind", ["edges", "few", "few_plus_one", "long", "dense", "ends", "spans"])
def test_rle_tiles(kind, shift):
    """Run-length encoding and decoding around the 4,096-byte tiles: runs that
    begin many tiles before their end, tiles without a run end, blocks that end
    at and beside a tile's edge, several blocks in a tile, and inputs and
    outputs that are not 16-byte aligned."""
    import torch
    r = np.random.RandomState(41)
    if kind == "edges":
        blocks = [r.randint(0, 2, n).astype(np.uint8) for n in (4095, 1, 4096, 4097, 15, 16, 17, 8175, 1, 1, 12288)]
    elif kind in ("few", "few_plus_one"):  # eight tiles and one more byte: the largest batch without the sums' pass
        n = 8 * 4096 + (kind == "few_plus_one")
        b = r.randint(0, 2, n).astype(np.uint8)
        b[5000:14_000] = 9  # a run over two whole tiles
        blocks = [b[:20_001], b[20_001:20_002], b[20_002:]]
    elif kind == "long":  # 300,000-byte runs: tiles 32 and more back hold the last run end
        blocks = [np.repeat(np.array([5, 6, 5], dtype=np.uint8), 300_000), np.full(200_000, 6, dtype=np.uint8)]
    elif kind == "spans":  # more tiles, of bytes and of runs, than spans: a warp sums a tile
        blocks = [r.randint(0, 256, n).astype(np.uint8) for n in (4_000_001, 999_999)]
    elif kind == "dense":
        blocks = [np.arange(70_001, dtype=np.uint32).astype(np.uint8), r.randint(0, 256, 9).astype(np.uint8)]
    else:  # a run of one byte at every edge, long runs between
        b = np.zeros(20 * 4096, dtype=np.uint8)
        b[4095::4096] = 1
        blocks = [b, np.ones(4096, dtype=np.uint8), np.ones(4096 - 20, dtype=np.uint8)]
    buf, off = batch_from_blocks(blocks)
    ref_c, ref_l, ref_ro = oracle.rle_batch(buf, off)
    R = int(ref_ro[-1])
    sizes = np.diff(off.astype(np.int64))
    pad = 32
    d_in = torch.zeros(buf.size + pad, dtype=torch.uint8, device="cuda")
    d_in[shift:shift + buf.size] = torch.from_numpy(buf).cuda()
    chars = torch.full((buf.size + pad,), 0xEE, dtype=torch.uint8, device="cuda")
    lens = torch.full((buf.size + pad,), -1, dtype=torch.int32, device="cuda")
    ro = torch.zeros(off.size, dtype=torch.int64, device="cuda")
    out = torch.full((buf.size + pad,), 0xEE, dtype=torch.uint8, device="cuda")
    with Plan(max_blocks=off.size - 1, max_total_bytes=buf.size, max_block_bytes=int(sizes.max())) as plan:
        plan.rle_encode_into(d_in[shift:shift + buf.size], off, chars[shift:], lens[shift:], ro)
        plan.rle_decode_into(chars[shift:], lens[shift:], ro, off, out[shift:])
    assert np.array_equal(ro.cpu().numpy().astype(np.uint64), ref_ro)
    assert np.array_equal(chars[shift:shift + R].cpu().numpy(), ref_c)
    assert np.array_equal(lens[shift:shift + R].cpu().numpy().astype(np.uint32), ref_l)
    assert bool((chars[shift + R:] == 0xEE).all()) and bool((lens[shift + R:] == -1).all())
    assert np.array_equal(out[shift:shift + buf.size].cpu().numpy(), buf)
    assert bool((out[:shift] == 0xEE).all()) and bool((out[shift + buf.size:] == 0xEE).all())


@pytest.mark.parametrize("tile", [1024, 4096])
@pytest.mark.parametrize("flags", [0, F_GRAPH])
def test_interleaved_tiles(tile, flags):
    """The radix passes take the tiles of 128 blocks in turn: more blocks than
    one group, with no two neighbours of the same number of tiles, and a plan
    whose layout changes between calls."""
    r = np.random.RandomState(51)
    sizes = [int(n) for n in np.concatenate([r.randint(1, 30_000, 140), [1, 4096, 4097, 60_000], r.randint(1, 9, 120)])]
    blocks = [r.randint(0, 256, n).astype(np.uint8) for n in sizes]
    with Plan(max_blocks=len(blocks), max_total_bytes=sum(sizes), max_block_bytes=max(sizes), tile_keys=tile,
              flags=flags) as plan:
        for part in (blocks, blocks[100:150], blocks[::-1], blocks[:1]):
            buf, off = batch_from_blocks(part)
            L, prim, _ = gpu_bwt(buf, off, plan)
            assert_matches_oracle(buf, off, L, prim, f"{len(part)} blocks")


@pytest.mark.parametrize("count", [1, 31, 63, 64, 65, 200])
def test_mlp_gradient_of_partial_ctas(count):
    """Four threads a sample, 64 samples a CTA: counts around a warp and a CTA
    against the float64 oracle, to the relative 1e-4 / absolute 1e-6 the
    gradient check uses."""
    import ctypes

    import torch
    from paper_1109_2348_gb300 import _lib
    r = np.random.RandomState(count)
    params = model.init_params(7)
    x = r.rand(count, 8).astype(np.float32)
    t = r.rand(count).astype(np.float32)
    loss, want = oracle.mlp_loss_grad(params.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
    d = [torch.from_numpy(a).cuda() for a in (params, x, t)]
    grad, got_loss = torch.zeros(params.size, device="cuda"), torch.zeros(1, device="cuda")
    vp = [ctypes.c_void_p(a.data_ptr()) for a in (*d, grad, got_loss)]
    lib = _lib.load()
    _lib.check(lib.bwt_mlp_loss_grad(vp[0], vp[1], vp[2], count, vp[3], vp[4], ctypes.c_void_p(0)), "loss_grad")
    np.testing.assert_allclose(grad.cpu().numpy(), want, rtol=1e-4, atol=1e-6)
    np.testing.assert_allclose(got_loss.item(), loss, rtol=1e-4, atol=1e-6)


def test_spread_of_equal_splitters():
    """A model whose output jumps where the first byte does gives runs of equal
    splitters: the compiled table is sorted and spreads each run evenly up to
    the next distinct splitter."""
    import ctypes

    import torch
    from paper_1109_2348_gb300 import _lib
    p = np.zeros(model.NPARAMS, dtype=np.float32)  # y = x0 through one unit a layer
    p[0] = p[288] = p[1344] = 1.0
    norm = np.repeat(np.arange(8, dtype=np.float32) / 8, 32)  # eight steps over the first byte
    d_p, d_n = torch.from_numpy(p).cuda(), torch.from_numpy(norm).cuda()
    d_s = torch.zeros(model.SPLITTERS, dtype=torch.int64, device="cuda")
    vp = [ctypes.c_void_p(a.data_ptr()) for a in (d_p, d_n, d_s)]
    lib = _lib.load()
    _lib.check(lib.bwt_model_compile(*vp, ctypes.c_void_p(0)), "compile")
    got = d_s.cpu().numpy().view(np.uint64)
    want = []
    for j in range(model.SPLITTERS):  # the smallest key whose first byte's step reaches (j + 1) / 4096
        step = -(-(j + 1) * 8 // 4096)
        want.append((step * 32) << 56 if step < 8 else (1 << 64) - 1)
    want = sorted(want)
    out = []
    for i, w in enumerate(want):
        first, end = want.index(w), len(want) - want[::-1].index(w)
        nxt = want[end] if end < len(want) else (1 << 64) - 1
        out.append(w + (nxt - w) * (i - first) // (end - first))
    assert np.array_equal(got, np.array(out, dtype=np.uint64))


@pytest.mark.parametrize("shift", [0, 1, 7])
@pytest.mark.parametrize("longest", [1, 13, 26, 27, 32])
def test_vle_word_packing(longest, shift):
    """Variable-length encoding by whole words: codes of one length up to the
    one that shares a word with its length, just above it and of 32 bits, mixed
    with 1-bit ones, blocks of every size around a thread's 16 bytes and a tile,
    unaligned input."""
    import torch
    r = np.random.RandomState(61)
    length = np.where(np.arange(256) % 3 == 0, longest, r.randint(1, longest + 1, 256)).astype(np.uint8)
    code = r.randint(0, 1 << 32, 256, dtype=np.uint64).astype(np.uint32)
    blocks = [r.randint(0, a, n).astype(np.uint8) for a in (1, 256) for n in (1, 15, 16, 17, 31, 4095, 4096, 4097, 9001)]
    buf, off = batch_from_blocks(blocks)
    sizes = np.diff(off.astype(np.int64))
    d_in = torch.zeros(buf.size + 16, dtype=torch.uint8, device="cuda")
    d_in[shift:shift + buf.size] = torch.from_numpy(buf).cuda()
    with Plan(max_blocks=off.size - 1, max_total_bytes=buf.size, max_block_bytes=int(sizes.max())) as plan:
        got, byte_off, bits = plan.vle_encode(d_in[shift:shift + buf.size], off, code, length)
    got, byte_off = got.cpu().numpy(), byte_off.cpu().numpy()
    for b in range(off.size - 1):
        blk = buf[int(off[b]):int(off[b + 1])]
        want = "".join(format(int(code[x]) & ((1 << int(length[x])) - 1), "b").zfill(int(length[x])) for x in blk)
        assert int(bits[b]) == len(want)
        want = np.frombuffer(int(want.ljust(-(-len(want) // 8) * 8, "0"), 2).to_bytes(-(-len(want) // 8), "big"), np.uint8)
        assert np.array_equal(got[byte_off[b]:byte_off[b + 1]], want), f"block {b}"


@pytest.mark.parametrize("flags", [0, F_GRAPH, F_LEARNED | F_GRAPH])
def test_small_batch_tiles(flags):
    """Batches around the largest that takes 1,024-key tiles (900 of them), a
    call of each kind after the other on one plan, and its inverse."""
    import torch
    r = np.random.RandomState(71)
    sets = [[900 * 1024], [899 * 1024 + 1, 1], [900 * 1024 + 1], [1] * 900, [2] * 901, [1023, 1024, 1025, 5000, 7],
            [100_000]]
    with Plan(max_blocks=1000, max_total_bytes=1_000_000, max_block_bytes=1_000_000, flags=flags) as plan:
        if flags & F_LEARNED:
            model.install(plan, model.equal_width_splitters())
        for sizes in sets:
            blocks = [r.randint(0, 60, n).astype(np.uint8) for n in sizes]
            buf, off = batch_from_blocks(blocks)
            L, prim, st = gpu_bwt(buf, off, plan)
            assert st["tile_keys"] == 4096
            assert_matches_oracle(buf, off, L, prim, str(sizes[:3]))
            back = plan.inverse(torch.from_numpy(L).cuda(), off, torch.from_numpy(prim).cuda())
            assert np.array_equal(back.cpu().numpy(), buf)


def _group_blocks():
    """Blocks whose 8-byte prefixes repeat m times each, for group sizes m at
    the edges of the size classes, with sorted, reversed, equal and mixed
    successors (what decides the order inside a group)."""
    r = np.random.RandomState(81)
    blocks = []
    for m in (33, 64, 65, 72, 73, 255, 256, 257, 288, 289, 511, 1000, 2047, 2048, 2049):
        for kind in range(3):
            unit = r.randint(0, 256, 9).astype(np.uint8)
            tails = r.randint(0, 256, (m, 6)).astype(np.uint8)
            if kind == 1:
                tails[:, :] = tails[0]
            elif kind == 2:
                tails[:, 0] = np.arange(m) // max(1, m // 7)
            blocks.append(np.concatenate([np.concatenate([unit, t]) for t in tails]))
    return blocks


@pytest.mark.parametrize("flags", [0, F_GRAPH])
def test_group_sorts_at_class_edges(flags):
    buf, off = batch_from_blocks(_group_blocks())
    L, prim, _ = gpu_bwt(buf, off, flags=flags)
    assert_matches_oracle(buf, off, L, prim)


@pytest.mark.parametrize("tile", [1024, 2048, 4096])
def test_scatter_units_of_several_tiles(tile):
    """The chunk scatter takes consecutive tiles of a block as one unit of up
    to 8,192 rotations: blocks around that size and its multiples, in a batch
    large enough that a CTA gets several tiles (an equal-width table)."""
    r = np.random.RandomState(91)
    sizes = [8191, 8192, 8193, 4097, 12_288, 16_385, 24_577, 40_000] * 6 + [1] * 40 + [2_500_000 // 8] * 30
    blocks = [r.randint(0, 256, n).astype(np.uint8) for n in sizes]
    buf, off = batch_from_blocks(blocks)
    with Plan(max_blocks=len(sizes), max_total_bytes=buf.size, max_block_bytes=max(sizes), tile_keys=tile,
              flags=F_LEARNED | F_GRAPH) as plan:
        model.install(plan, model.equal_width_splitters())
        L, prim, st = gpu_bwt(buf, off, plan)
    assert st["blocks_routed_plain"] == 0
    assert_matches_oracle(buf, off, L, prim, f"tile {tile}")


@pytest.mark.parametrize("more", [-1, 0, 1, 700])
def test_radix_tiles_around_the_grid(more):
    """The radix passes claim one tile a CTA where the grid has a CTA for each,
    and go on claiming beyond: tile counts about the largest grid of 1,024-key
    tiles (six CTAs an SM), with a partial last tile."""
    import torch
    r = np.random.RandomState(53)
    tiles = 6 * torch.cuda.get_device_properties(0).multi_processor_count + more
    n = tiles * 1024 - 5
    buf = r.randint(0, 4, n).astype(np.uint8)
    off = np.array([0, 300_001, n], dtype=np.uint64)
    with Plan(max_blocks=2, max_total_bytes=n, max_block_bytes=n - 300_001, tile_keys=1024) as plan:
        L, prim = plan.forward(torch.from_numpy(buf).cuda(), off)
    assert_matches_oracle(buf, off, L.cpu().numpy(), prim.cpu().numpy(), more)


@pytest.mark.parametrize("cells", [(14, 15, 16), (15, 1, 0), (3000, 1000)])
def test_crowded_index_cells(cells):
    """The counting kernel's index stores up to 14 splitters of a cell (the keys'
    first 15 bits) and looks at the next cell above that: cells around the limit,
    first and last cells, keys that equal splitters, and the byte before the
    first rotation of the block at a staged tile's edge."""
    import torch
    r = np.random.RandomState(59)
    spl = []
    for i, k in enumerate(cells):  # crowded cells at the key space's start, middle and end
        base = np.uint64([0, 0x4142 << 48, 0xFFFE << 48][i])
        spl.append(base + np.arange(k, dtype=np.uint64) * np.uint64((1 << 36) + 12_345))
    have = np.concatenate(spl)
    rest = np.linspace(1 << 52, (1 << 64) - (1 << 52), 4095 - have.size).astype(np.uint64)
    spl = np.sort(np.concatenate([have, rest]))
    some = spl[r.randint(0, 4095, 400)]
    text = np.concatenate([np.frombuffer(int(x).to_bytes(8, "big"), dtype=np.uint8) for x in some])
    blocks = [np.concatenate([text, r.randint(0x41, 0x43, 20_000).astype(np.uint8)]),
              r.randint(0, 256, 30_011).astype(np.uint8), np.tile(text, 3)[:9_001]]
    buf, off = batch_from_blocks(blocks)
    with Plan(max_blocks=3, max_total_bytes=buf.size, max_block_bytes=int(np.diff(off.astype(np.int64)).max()),
              flags=F_LEARNED) as plan:
        model.install(plan, spl)
        L, prim = plan.forward(torch.from_numpy(buf).cuda(), off)
    assert_matches_oracle(buf, off, L.cpu().numpy(), prim.cpu().numpy(), cells)


@pytest.mark.parametrize("count,batch", [(1000, 256), (64, 64), (130, 1000)])
def test_training_steps_in_order(count, batch):
    """Training's dependent launches against the gradient and the Adam step
    called one after the other, with a partial last batch, one batch an epoch
    and a batch larger than the samples. Both round differently by some 2^-24 a
    step; a step that read old weights or sums would be off by the learning rate,
    1e-3, in most of the parameters."""
    import ctypes

    import torch
    from paper_1109_2348_gb300 import _lib
    lib, r, epochs = _lib.load(), np.random.RandomState(count), 3
    x, t = r.rand(count, 8).astype(np.float32), r.rand(count).astype(np.float32)
    order = np.concatenate([r.permutation(count) for _ in range(epochs)]).astype(np.int32)
    vp = lambda a: ctypes.c_void_p(a.data_ptr())
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        st = ctypes.c_void_p(stream.cuda_stream)
        d_x, d_t, d_o = (torch.from_numpy(a).cuda() for a in (x, t, order))
        got = torch.from_numpy(model.init_params(7)).cuda()
        want = got.clone()
        _lib.check(lib.bwt_model_train(vp(got), vp(d_x), vp(d_t), count, vp(d_o), epochs, batch,
                                       ctypes.c_float(1e-3), ctypes.c_void_p(0), st), "train")
        g, m, v, loss = (torch.zeros(n, device="cuda") for n in (want.numel(),) * 3 + (1,))
        step = 0
        for e in range(epochs):
            for b in range(0, count, batch):
                i = d_o[e * count + b:e * count + min(b + batch, count)].long()
                xs, ts, step = d_x[i].contiguous(), d_t[i].contiguous(), step + 1
                _lib.check(lib.bwt_mlp_loss_grad(vp(want), vp(xs), vp(ts), i.numel(), vp(g), vp(loss), st), "grad")
                _lib.check(lib.bwt_mlp_adam_step(vp(want), vp(g), vp(m), vp(v), step, ctypes.c_float(1e-3), st), "adam")
        diff = (got - want).abs().cpu().numpy()
    assert np.median(diff) <= 1e-6 and diff.max() <= 1e-4, (np.median(diff), diff.max())
