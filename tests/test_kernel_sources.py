"""Host checks of rules that the kernels' sources keep (read as text, no GPU)."""
import os
import re

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1109_2348_gb300", "csrc")


def _kernel(name, file):
    """(parameter list, body) of a __global__ function."""
    src = open(os.path.join(CSRC, file)).read()
    m = re.search(r"__global__[^;{]*?\b" + name + r"\((.*?)\)\s*\{(.*?)\n\}\n", src, re.S)
    assert m, f"{name} not found in {file}"
    return m.group(1), m.group(2)


def test_radix_pass_takes_no_tile_after_a_failure():
    """A pass whose wait ran out leaves rows that no longer match the digit
    histograms of the passes after it: modelled here, their destinations leave
    the segment, so a pass asks for the error word with its first claim."""
    rng = np.random.default_rng(1)
    n, tile, radix = 6 * 1024, 1024, 256
    key = rng.integers(0, 1 << 16, n)

    def one_pass(k, shift, base, withheld):
        """Destinations of a pass in which tile 0 does not publish its counts."""
        d = (k >> shift) & (radix - 1)
        dst = np.empty(n, dtype=np.int64)
        seen = np.zeros(radix, dtype=np.int64)  # counts of the earlier tiles, as a tile reads them
        for t in range(0, n, tile):
            dt = d[t:t + tile]
            rank = np.array([np.count_nonzero(dt[:j] == x) for j, x in enumerate(dt)])
            dst[t:t + tile] = base[dt] + seen[dt] + rank
            if t or not withheld:
                seen += np.bincount(dt, minlength=radix)
        return dst

    def bases(shift):
        c = np.bincount((key >> shift) & (radix - 1), minlength=radix)
        return np.cumsum(c) - c

    first = one_pass(key, 0, bases(0), True)
    assert first.min() >= 0 and first.max() < n  # a short prefix stays inside the segment
    rows = np.full(n, (1 << 16) - 1)  # what the buffer held before
    rows[first] = key
    assert one_pass(rows, 8, bases(8), True).max() >= n  # the next pass would not
    _, body = _kernel("k_onesweep", "radix.cu")
    claim = body[body.index("atomicAdd(p.tile_counter"):body.index("for (;;)")]
    assert "ld_volatile(&p.ctrl[CTRL_ERR])" in claim and "at = 0xffffffffu" in claim


def test_cta_leaves_as_one():
    """The branches of a captured graph run side by side, so one branch's kernel
    may set the error word while a CTA of another's starts: a kernel that a
    branch launches asks for it once for the whole CTA, before any other use of
    its barriers, and no thread leaves on a reading of its own."""
    kernels = [("k_name_initial", "doubling.cu"), ("k_sort_micro", "doubling.cu"), ("k_sort_tiny", "doubling.cu"),
               ("k_sort_small", "doubling.cu"), ("k_sort_med", "doubling.cu"), ("k_rename_large", "doubling.cu"),
               ("k_chunk_sort_name", "learned.cu")]
    for name, file in kernels:
        _, body = _kernel(name, file)
        assert "ld_volatile(&ctrl[CTRL_ERR])" not in body, f"{name}: a thread's own reading of the error word"
        at = body.find("if (failed_before(ctrl)) return;")
        assert at >= 0, f"{name} does not ask for the error word"
        assert not re.search(r"__sync|coop_sync|\breturn\b|for \(", body[:at]), f"{name}: asked too late"


def test_training_reads_results_after_the_wait():
    """Training's kernels start while the one before them runs. What that one
    writes (weights, moments, partial sums) is read after the wait and through
    pointers that promise nothing about the values' standing still: such a
    promise lets a compiler move the loads ahead of the wait."""
    for name, shared in (("k_mlp_grad", ("params",)),
                         ("k_mlp_reduce", ("partial", "loss_partial", "params", "m", "v"))):
        params, body = _kernel(name, "mlp.cu")
        before = body[:body.index("step_wait();")]
        for p in shared:
            decl = re.search(r"[^,]*\b" + p + r"\s*(?:,|$)", params.strip()).group(0)
            assert "__restrict__" not in decl, f"{name}: {decl}"
            assert not re.search(r"\b" + p + r"\s*\[", before), f"{name} reads {p} before its wait"


def test_plan_creation_takes_pinned_memory_once():
    """Every pinned allocation and its release cost a program that makes a plan
    for a call: a plan takes its pinned tables in one."""
    src = open(os.path.join(CSRC, "plan.cu")).read()
    body = src[src.index("bwt_status bwt_plan_create("):src.index("bwt_status bwt_plan_destroy(")]
    assert body.count("host_alloc(") == 1
