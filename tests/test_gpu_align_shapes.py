"""The alignment kernel at the edges of its forms: the groups of four and
eight rows, the row pairs per lane, the blocks of eight diagonals, the lanes'
change of rows in narrow bands, one warp / four warps / a CTA per pair, more
distinct bytes than it keeps match vectors for, and accumulated costs past 16
bits. Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W

from _parity import to_np

pytestmark = pytest.mark.gpu


def _check(ks, ms, max_len, symbols, windows, seed, n_vocab=200, min_len=0, n_long=0):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)
    rng = np.random.default_rng(seed)
    strings = set()
    while len(strings) < n_vocab:
        strings.add(bytes(rng.choice(symbols, size=int(rng.integers(min_len, max_len + 1)))
                          .astype(np.uint8)))
    while len(strings) < n_vocab + n_long:  # some of 9 to 20 bytes
        strings.add(bytes(rng.choice(symbols, size=int(rng.integers(9, 21))).astype(np.uint8)))
    n_vocab = len(strings)
    voc = W.Vocab.from_strings(sorted(strings))
    d_off = np.concatenate([[0], np.cumsum(ks)]).astype(np.int32)
    t_off = np.concatenate([[0], np.cumsum(ms)]).astype(np.int32)
    d_ids = rng.integers(0, n_vocab, size=int(d_off[-1])).astype(np.int32)
    t_ids = rng.integers(0, n_vocab, size=int(t_off[-1])).astype(np.int32)
    batch = tt.Batch.from_host(d_off, d_ids, t_off, t_ids, device="cuda")
    vt = tt.VocabTable.from_host(voc.blob, voc.off, "cuda")
    for w in windows:
        g = to_np(tt.tt_align(batch, vt, vt, tt.Params(window=w)))
        o = oracle.align(d_off, d_ids, t_off, t_ids, voc.blob, voc.off, voc.blob, voc.off, w)
        for key in ("status", "path_len", "cost", "map"):
            assert np.array_equal(g[key], o[key]), (key, w)
        for b in range(len(ks)):
            p0, L = int(d_off[b] + t_off[b]), int(o["path_len"][b])
            assert np.array_equal(g["path"][2 * p0:2 * (p0 + L)], o["path"][p0:p0 + L].ravel()), (b, w)


EDGES = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65]


@pytest.mark.parametrize("max_k,max_m", [(9, 17), (65, 65), (127, 140), (129, 200), (256, 300)])
def test_lengths_at_edges(max_k, max_m):
    ks = [k for k in EDGES + [127, 128, 129, 255, 256] if k <= max_k]
    ms = [m for m in EDGES + [max_m - 1, max_m] if m <= max_m]
    rng = np.random.default_rng(max_k)
    kk = np.array(ks * 2)
    mm = rng.choice(ms, size=len(kk))
    kk[-1], mm[-1] = max_k, max_m
    _check(kk, mm, 8, np.arange(97, 117), (0, 8, 27, 28, 29, 56, 57, 112, 113, -1), max_k)


def test_more_pairs_than_wide_ctas():
    """More pairs than two per SM: four warps per pair; and small pairs, a warp each."""
    rng = np.random.default_rng(5)
    _check(rng.integers(30, 70, size=700), rng.integers(30, 90, size=700), 6,
           np.arange(97, 123), (8,), 1)
    _check(rng.integers(1, 9, size=700), rng.integers(1, 12, size=700), 8,
           np.arange(97, 123), (8,), 2)


@pytest.mark.parametrize("k", [40, 200])
def test_many_distinct_bytes(k):
    _check([k] * 6, [60] * 6, 8, np.arange(256), (8, -1), k, n_vocab=400)


def test_costs_past_16_bits():
    # (k + m) x (longest token) > 16000: the sweep in 32 bits; distances above
    # and below 127 (the largest that the tile stores)
    _check([100, 33], [90, 100], 200, np.arange(97, 117), (8, -1), 3, n_vocab=40, min_len=100)
    _check([130], [140], 100, np.arange(97, 117), (8,), 4, n_vocab=40, min_len=60)


def test_bands_wider_than_any_pair():
    _check([3, 64, 200], [5, 90, 300], 8, np.arange(97, 117), (767, 768, 2**30, 2**31 - 1), 9)


@pytest.mark.parametrize("n_long", [1, 5, 30, 200])
def test_a_few_long_tokens(n_long):
    """Cells of long tokens scattered over the band, fewer and more than a warp
    takes at once, on one warp, four warps and sixteen per pair."""
    rng = np.random.default_rng(n_long)
    args = (8, np.arange(97, 117), (0, 3, 8, -1), n_long)
    _check(rng.integers(1, 20, size=60), rng.integers(1, 25, size=60), *args, n_long=n_long)
    _check([64] * 400, rng.integers(40, 90, size=400), *args, n_long=n_long)
    _check([200, 130, 64], [250, 31, 90], *args, n_long=n_long)
