"""Which way the nucleus kernels settle each row in the GPU nucleus tests,
computed on the CPU from the same seeded inputs.

A row of at most 8192 columns takes one warp: the columns within 12 log2 units
of its maximum (at most 512) are the candidates, and the 1/32-log2-unit bucket of
the cut holds at most 32 of them. A row of more than four 8 KB units (2048 fp32
or 4096 bf16 columns each; and at most 983,040 columns) takes the nucleus row
kernel: unit u goes to region u mod 20, each with room for 160 candidates within
14 log2 units, which raises its bar when it is full; the cut must lie above every
bar and its bucket hold at most 128.

What these leave, and every other row, takes one CTA: a pass over the columns
within 14 log2 units, at most 512 in each of eight regions (vector v of a row goes
to thread v mod 256), the cut's bucket of at most 256; where a region is too small
a second pass at the largest whole bar of 8 to 13 with at most 3200 columns; and
the histogram levels for the rest.

The paper's settings (App. F: T 0.6 with top-p 0.9 or 0.95) never need the
levels on the five workloads. The GPU tests also hold rows that are left for
each of the CTA's three ways, and rows whose bar is raised but which the row
kernel settles."""
import dataclasses
import importlib
import os
import sys

import numpy as np
import pytest
import torch

from paper_2510_15545_gb300 import workload as W

LOG2E = 1.4426950408889634
ROW, WARP, CTA1, CTA2, LEVELS = "row kernel", "warp", "first pass", "second pass", "levels"


def _cta_way(d, m, cut, cross, vec, nvec):
    """The CTA's way for a row: deltas d, masses m, the cut's delta, the columns in
    its bucket, columns per vector and vectors."""
    def fits(bar):
        cols = np.nonzero(d < bar)[0]
        tid = np.where(cols < nvec * vec, (cols // vec) % 256, (cols - nvec * vec) % 256)
        return np.bincount(tid // 32, minlength=8).max() <= 512
    if fits(14):
        return {CTA1} if cut < 13.5 and cross <= 250 else {LEVELS} if cut > 14.1 or cross > 262 \
            else {CTA1, LEVELS}
    bars = [b for b in range(8, 14) if (d < b).sum() <= 3200]
    if not bars or not fits(max(bars)) or cut > max(bars) + 0.1 or cross > 262:
        return {LEVELS}
    # (the kernel estimates the bar from the columns it holds)
    return {CTA2} if cut < max(bars) - 1.1 and cross <= 250 else {CTA2, LEVELS}


def ways(logits: torch.Tensor, T: float, p: float) -> list:
    """Per row, the ways that may settle it (one unless it is near a limit)."""
    V = logits.shape[1]
    f32 = logits.dtype == torch.float32
    unit, vec = (2048, 4) if f32 else (4096, 8)
    z = logits.float().numpy().astype(np.float64) * (LOG2E / T)
    out = []
    for zr in z:
        d = zr.max() - zr
        m = np.exp2(-d)
        order = np.lexsort((np.arange(V), d))  # larger logit first, then smaller column
        before = np.cumsum(m[order]) - m[order]
        cut = d[order[max(0, (before < p * m.sum()).sum() - 1)]]
        cross = int((np.floor(d * 32) == np.floor(cut * 32)).sum())
        cta = _cta_way(d, m, cut, cross, vec, V // vec)
        if V <= 8192:
            n = int((d < 12).sum())
            settled, left = n <= 500 and cut < 11.5 and cross <= 28, \
                n > 520 or cut > 12.1 or cross > 36
            first = WARP
        elif 4 * unit < V <= 983040:
            slot = (np.arange(V) // unit) % 20
            full = np.bincount(slot[d < 14], minlength=20).max()
            to_cut = np.bincount(slot[d <= cut], minlength=20).max()
            settled = full <= 160 and cut < 12.5 and cross <= 120
            left = to_cut > 160 or cut > 14.1 or cross > 136
            first = ROW
        else:
            settled, left, first = False, True, None
        out.append({first} if settled else cta if left else {first} | cta)
    return out


def test_the_table_settings_never_need_the_levels():
    for name, B in (("b64_g8_v152k", 6), ("b1024_g8_v201k_bf16", 4),
                    ("b256_g16_v152k_bf16", 2), ("dtw_4096x64", 4), ("b1_g4_v32k", 1)):
        wl = W.make_workload(name, B=B, seed=3)
        for p in (0.9, 0.95):
            for L in (wl.target_logits, wl.draft_logits):
                assert all(LEVELS not in w for w in ways(L, 0.6, p)), (name, p)


def test_coarse_integer_rows_take_the_histogram_levels():
    wl = W.make_workload("b64_g8_v152k", B=8, seed=11)
    rng = np.random.default_rng(5)
    tl = torch.as_tensor(rng.integers(-3, 4, size=wl.target_logits.shape).astype(np.float32))
    tl[::3, 17] = 60.0
    wl2 = dataclasses.replace(wl, target_logits=tl)
    way = ways(wl2.target_logits[:12], 0.6, 0.9)
    assert all(w == ({ROW} if r % 3 == 0 else {LEVELS}) for r, w in enumerate(way))


def _gpu_rows():
    sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
    return importlib.import_module("test_gpu_nucleus")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("kind,way", [("bucket", CTA1), ("unit", CTA2), ("crowd", LEVELS)])
def test_rows_that_the_row_kernel_leaves(kind, way, dtype):
    """The rows of test_gpu_nucleus.left_rows, each left for the way named."""
    gn = _gpu_rows()
    wl = gn.left_rows(W.make_workload("b64_g8_v152k", B=1, seed=13), kind, dtype)
    assert all(w == {way} for w in ways(wl.target_logits, 0.6, gn.LEFT_TOP_P))


def test_crowded_rows_raise_the_bar_of_the_row_kernel():
    """The rows of test_gpu_nucleus.crowded_rows: every region is too small for
    the candidates within 14 log2 units, none for those within 12, and the cut
    lies there: the regions raise their bars to 12 and the row is settled."""
    wl = _gpu_rows().crowded_rows(W.make_workload("b64_g8_v152k", B=2, seed=13))
    z = wl.target_logits.numpy().astype(np.float64) * (LOG2E / 0.6)
    d = z.max(1, keepdims=True) - z
    m = np.exp2(-d)
    slot = (np.arange(d.shape[1]) // 2048) % 20
    for r in range(len(d)):
        assert np.bincount(slot[d[r] < 14], minlength=20).min() > 160
        assert np.bincount(slot[d[r] < 12], minlength=20).max() <= 160
        assert m[r][d[r] < 11].sum() >= 0.5 * m[r].sum()
