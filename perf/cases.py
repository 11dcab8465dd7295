"""The measured workloads: what users have this library do, through its public entry points.

A case is a dict of plain values:
  op       forward, inverse, rle_encode, rle_decode, mtf_encode, vle_encode or train
  mix      the sources of the batch's blocks (see MIXES)
  blocks   how many blocks
  lo, hi   the range of their sizes in bytes (uniform in it, or uniform in its logarithm with "log")
  learned  forward: bucketing by the learned splitter table, else the plain radix path
  graph    forward: the asynchronous, graph-replayed call, else the host-driven one
  samples, batch, epochs   train only
Sizes come from the case alone, contents from the seed.
"""
from __future__ import annotations

import ctypes
import heapq
import math

import numpy as np
import torch

from paper_1109_2348_gb300 import F_GRAPH, F_LEARNED, Plan, _lib, datagen, model

# The source of block b is MIXES[mix][b % len].
MIXES = {
    "markov2": [datagen.MARKOV2_Z64],
    "markov3": [datagen.MARKOV3_Z96],
    # nine text-like blocks, then one that does not compress
    "text+uniform": [datagen.MARKOV3_Z96] * 9 + [datagen.UNIFORM],
    "mixed": [datagen.UNIFORM, datagen.MARKOV3_Z96, datagen.RUNS16],
    "degenerate": [datagen.CONST, datagen.PERIOD7, datagen.PERIOD1000, datagen.FIBONACCI, datagen.MUTATED_UNIT],
    "all": list(range(9)),
}
SIZE_SEED = 4000
DISTINCT = 180
# Per source: runs per byte of a block's L column, and the bits a byte of its
# move-to-front output takes in a Huffman code of the block's own (rounded,
# 900,000-byte blocks). Only work() uses them, to size outputs it cannot know.
RUNS_PER_BYTE = {datagen.UNIFORM: 1.0, datagen.MARKOV2_Z64: 0.8, datagen.MARKOV3_Z96: 0.9, datagen.RUNS16: 0.08}
VLE_BITS = 6.5


def listed():
    mixed = {"mix": "mixed", "blocks": 64, "lo": 900_000, "hi": 900_000}
    return [
        # the headline: a gigabyte of archive blocks at bzip2 -9's block size, sorted with a trained model
        {"name": "forward_learned_1200x900k", "op": "forward", "mix": "text+uniform", "blocks": 1200, "lo": 900_000,
         "hi": 900_000, "learned": True, "graph": True},
        # many files of all sizes in one batch
        {"name": "forward_learned_256_uneven", "op": "forward", "mix": "markov3", "blocks": 256, "lo": 10_000,
         "hi": 900_000, "learned": True, "graph": True},
        # no model at hand, contents of every kind: the plain radix path with its doubling rounds
        {"name": "forward_plain_mixed64", "op": "forward", **mixed, "learned": False, "graph": True},
        # periodic and near-periodic blocks, where the doubling rounds are all of the work
        {"name": "forward_plain_degenerate5", "op": "forward", "mix": "degenerate", "blocks": 5, "lo": 900_000,
         "hi": 900_000, "learned": False, "graph": True},
        # one bzip2 -1 block: latency
        {"name": "forward_plain_1x100k", "op": "forward", "mix": "markov2", "blocks": 1, "lo": 100_000,
         "hi": 100_000, "learned": False, "graph": True},
        # a handful of small records of ragged sizes, sorted as they come (host-driven rounds): the smallest call
        {"name": "forward_plain_24_small", "op": "forward", "mix": "all", "blocks": 24, "lo": 1, "hi": 6000,
         "log": True, "learned": False, "graph": False},
        # decompression
        {"name": "inverse_mixed64", "op": "inverse", **mixed},
        # the stages around the sort, each on what it gets there: L columns, their runs, the runs' bytes, the positions
        {"name": "rle_encode_mixed64", "op": "rle_encode", **mixed},
        {"name": "rle_decode_mixed64", "op": "rle_decode", **mixed},
        {"name": "mtf_encode_mixed64", "op": "mtf_encode", **mixed},
        {"name": "vle_encode_mixed64", "op": "vle_encode", **mixed},
        # the splitter model, forward and backward: fitted to sampled prefixes and compiled
        {"name": "train_200k", "op": "train", "samples": 200_000, "batch": 4096, "epochs": 2},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["forward", "forward", "forward", "inverse", "rle_encode", "rle_decode", "mtf_encode",
                     "vle_encode", "train"])
    if op == "train":
        return {"op": op, "samples": _log_int(rng, 3_000, 400_000), "batch": rng.choice([1000, 2048, 4096]),
                "epochs": 1}
    learned = op == "forward" and rng.random() < 0.5
    mix = rng.choice(["markov2", "markov3", "text+uniform", "mixed"] + ([] if learned else ["degenerate", "all"]))
    hi = _log_int(rng, 50, 900_000)
    lo = rng.choice([hi, max(1, hi // 2), max(1, hi // 50), 1])
    # bytes in all: learned batches up to a quarter of the largest listed one, the others up to the mixed one;
    # blocks that take every doubling round are few
    most = {True: 270_000_000, False: 57_600_000}[learned]
    if mix in ("degenerate", "all"):
        most = 4_500_000
    c = {"op": op, "mix": mix, "blocks": _log_int(rng, 1, max(1, min(600, most // hi))), "lo": lo, "hi": hi,
         "log": hi >= 10 * lo}
    if op == "forward":
        c["learned"] = learned
        c["graph"] = rng.random() < 0.75
    return c


def _sizes(case):
    u = datagen.uniform_unit(SIZE_SEED + case["blocks"], case["blocks"])
    lo, hi = case["lo"], case["hi"]
    if case.get("log"):
        s = np.exp(np.log(lo) + u * (np.log(hi) - np.log(lo)))
    else:
        s = lo + u * (hi - lo)
    return [int(min(hi, max(lo, round(x)))) for x in s]


def _batch(case, seed):
    """(bytes, offsets) of the batch. The host draws at most DISTINCT blocks of a batch of equal sizes; the others are
    those blocks again, each from another starting point."""
    src, sizes = MIXES[case["mix"]], _sizes(case)
    n = len(sizes)
    k = min(n, DISTINCT) if case["lo"] == case["hi"] else n
    w = datagen.Workload("case", [src[b % len(src)] for b in range(n)],
                         [10_000_000 + 10_000 * seed + b for b in range(n)], sizes)
    off = w.offsets()
    buf = np.empty(int(off[-1]), dtype=np.uint8)
    w.subset(range(k)).generate(out=buf)
    start = np.random.RandomState(seed).randint(0, sizes[0], n)
    for b in range(k, n):
        o, p, m = int(off[b]), int(off[b % k]), sizes[0]
        r = int(start[b])
        buf[o:o + m - r] = buf[p + r:p + m]
        buf[o + m - r:o + m] = buf[p:p + r]
    return buf, off


def _plan(off, flags=0):
    return Plan(max_blocks=off.size - 1, max_total_bytes=int(off[-1]),
                max_block_bytes=int(np.diff(off.astype(np.int64)).max()), flags=flags)


_splitters = None


def _model_splitters():
    """The splitter table of a model trained once, as a program trains or loads it once."""
    global _splitters
    if _splitters is None:
        _splitters = model.train().splitters
    return _splitters


def _huffman(hist):
    """Codes and lengths (at most 32 bits) of a canonical Huffman code over the bytes that occur."""
    used = np.flatnonzero(hist)
    length = np.ones(256, dtype=np.uint8)
    if used.size > 1:
        # counts below a 2^-24 share are raised to it, so that no code is longer than 32 bits
        floor = max(1, int(hist.sum()) >> 24)
        heap = [(max(int(hist[b]), floor), int(b), [int(b)]) for b in used]
        heapq.heapify(heap)
        length[used] = 0
        uid = 256
        while len(heap) > 1:
            wa, _, a = heapq.heappop(heap)
            wb, _, b = heapq.heappop(heap)
            for x in a + b:
                length[x] += 1
            heapq.heappush(heap, (wa + wb, uid, a + b))
            uid += 1
    code = np.zeros(256, dtype=np.uint32)
    nxt = prev = 0
    for b in sorted(used.tolist(), key=lambda b: (length[b], b)):
        nxt <<= int(length[b]) - prev
        code[b] = nxt
        nxt += 1
        prev = int(length[b])
    return code, length


def _train_host(case, seed):
    """Training data of the model on the host: float32 prefixes and targets, minibatch order, first weights."""
    n = case["samples"]
    x = datagen.uniform_unit(30_000 + seed, n * 8).reshape(n, 8).astype(np.float32)
    t = (0.9 * x[:, 0] + 0.09 * x[:, 1] * x[:, 0] + 0.01 * x[:, 2]).astype(np.float32)
    order = np.concatenate([datagen.permutation(40_000 + 100 * seed + e, n) for e in range(case["epochs"])])
    return x, t, order, model.init_params(50_000 + seed)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.op = case["op"]
    if s.op == "train":
        x, t, order, params = _train_host(case, seed)
        s.case = case
        s.x, s.t, s.params0 = (torch.from_numpy(a).cuda() for a in (x, t, params))
        s.order = torch.from_numpy(order.view(np.int32)).cuda()
        # the byte values of text are far from even; any increasing table will do
        s.norm = torch.linspace(0.0, 1.0, 256, dtype=torch.float32).cuda()
        return s
    buf, off = _batch(case, seed)
    d_in = torch.from_numpy(buf).cuda()
    s.off = off
    if s.op == "forward":
        s.d_in = d_in
        flags = (F_LEARNED if case["learned"] else 0) | (F_GRAPH if case["graph"] else 0)
        s.plan = _plan(off, flags)
        if case["learned"]:
            model.install(s.plan, _model_splitters())
        s.L = torch.empty_like(d_in)
        s.primary = torch.empty(off.size - 1, dtype=torch.int32, device=d_in.device)
        return s
    s.plan = _plan(off)
    n, nb, dev = d_in.numel(), off.size - 1, d_in.device
    s.out = torch.zeros(n, dtype=torch.uint8, device=dev)
    L, s.primary = s.plan.forward(d_in, off)
    if s.op == "inverse":
        s.L = L
        return s
    if s.op == "rle_encode":
        s.L = L
        s.lens = torch.zeros(n, dtype=torch.int32, device=dev)
        s.run_off = torch.zeros(nb + 1, dtype=torch.int64, device=dev)
        return s
    chars, lens, s.run_off = s.plan.rle_encode(L, off)
    s.chars = chars.clone()
    if s.op == "rle_decode":
        s.lens = lens.clone()
        return s
    s.off = s.run_off.cpu().numpy().view(np.uint64)
    if s.op == "vle_encode":
        s.mtf = s.plan.mtf_encode(s.chars, s.off)
        code, length = _huffman(torch.bincount(s.mtf.int(), minlength=256).cpu().numpy())
        s.code = torch.from_numpy(code.view(np.int32)).cuda()
        s.length = torch.from_numpy(length).cuda()
        # the table's longest code is 32 bits, but a stream of its own histogram is hardly longer than its input
        s.out = torch.zeros(2 * n + 8 * nb + 64, dtype=torch.uint8, device=dev)
        s.byte_off = torch.zeros(nb + 1, dtype=torch.int64, device=dev)
        s.bits = torch.zeros(nb, dtype=torch.int64, device=dev)
    return s


def _vp(t):
    return ctypes.c_void_p(int(t.data_ptr()))


def run(s):
    if s.op == "forward":
        s.plan.forward_into(s.d_in, s.off, s.L, s.primary)
        return s.L, s.primary
    if s.op == "inverse":
        s.plan.inverse_into(s.L, s.off, s.primary, s.out)
        return s.out
    if s.op == "rle_encode":
        s.plan.rle_encode_into(s.L, s.off, s.out, s.lens, s.run_off)
        return s.out, s.lens, s.run_off
    if s.op == "rle_decode":
        s.plan.rle_decode_into(s.chars, s.lens, s.run_off, s.off, s.out)
        return s.out
    if s.op == "mtf_encode":
        s.plan.mtf_encode_into(s.chars, s.off, s.out)
        return s.out
    if s.op == "vle_encode":
        s.plan.vle_encode_into(s.mtf, s.off, s.code, s.length, s.out, s.byte_off, s.bits)
        return s.out, s.byte_off, s.bits
    lib = _lib.load()
    c = s.case
    params = s.params0.clone()
    loss = torch.zeros(c["epochs"], dtype=torch.float32, device=params.device)
    splitters = torch.empty(_lib.SPLITTERS, dtype=torch.int64, device=params.device)
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    _lib.check(lib.bwt_model_train(_vp(params), _vp(s.x), _vp(s.t), c["samples"], _vp(s.order), c["epochs"],
                                   c["batch"], ctypes.c_float(1e-3), _vp(loss), st), "bwt_model_train")
    _lib.check(lib.bwt_model_compile(_vp(params), _vp(s.norm), _vp(splitters), st), "bwt_model_compile")
    return {"params": params, "loss": loss, "splitters": splitters}


def work(case):
    if case["op"] == "train":
        # forward and backward of 1,344 weights a sample, six operations each (two forward, four backward),
        # and the compilation's 64 forward passes a splitter
        visits = case["samples"] * case["epochs"]
        return {"bytes": visits * (9 * 4 + 4), "flops": visits * 1344 * 6 + 4095 * 64 * 1344 * 2}
    src = MIXES[case["mix"]]
    sizes = _sizes(case)
    n = sum(sizes)
    if case["op"] in ("forward", "inverse"):
        return {"bytes": 2 * n + 4 * len(sizes), "flops": 0}
    runs = sum(RUNS_PER_BYTE.get(src[b % len(src)], 0.05) * m for b, m in enumerate(sizes))
    if case["op"] in ("rle_encode", "rle_decode"):
        return {"bytes": n + 5 * runs, "flops": 0}
    if case["op"] == "mtf_encode":
        return {"bytes": 2 * runs, "flops": 0}
    return {"bytes": runs * (1 + VLE_BITS / 8), "flops": 0}


def exact(case, seed):
    """The training step in 64 bits (forward, backward and Adam from their definitions). Every other output is bytes
    and whole numbers."""
    if case["op"] != "train":
        return None
    x, t, order, p = _train_host(case, seed)
    x, t, p = x.astype(np.float64), t.astype(np.float64), p.astype(np.float64)
    n, batch, lr = case["samples"], case["batch"], float(np.float32(1e-3))
    b1, b2, eps = float(np.float32(0.9)), float(np.float32(0.999)), float(np.float32(1e-8))
    m, v = np.zeros_like(p), np.zeros_like(p)
    step, losses = 0, []
    for e in range(case["epochs"]):
        total, count = 0.0, 0
        for at in range(0, n, batch):
            ix = order[e * n + at:e * n + min(n, at + batch)]
            X, T = x[ix], t[ix]
            W1, c1, W2, c2, W3, c3 = (p[0:256].reshape(32, 8), p[256:288], p[288:1312].reshape(32, 32), p[1312:1344],
                                      p[1344:1376], p[1376])
            h1 = np.maximum(X @ W1.T + c1, 0)
            h2 = np.maximum(h1 @ W2.T + c2, 0)
            err = h2 @ W3 + c3 - T
            total, count = total + float(np.mean(err * err)), count + 1
            dy = 2 * err / len(ix)
            d2 = np.where(h2 > 0, dy[:, None] * W3, 0)
            d1 = np.where(h1 > 0, d2 @ W2, 0)
            g = np.concatenate([(d1.T @ X).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), dy @ h2, [dy.sum()]])
            step += 1
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            p = p - lr * (m / (1 - b1 ** step)) / (np.sqrt(v / (1 - b2 ** step)) + eps)
        losses.append(total / count)
    return {"params": torch.from_numpy(p), "loss": torch.tensor(losses, dtype=torch.float64), "splitters": None}
