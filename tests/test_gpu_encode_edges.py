"""Re-encoding at the sizes where its kernels can go wrong, bit-exact against
the oracle: batches at the edges of the blocks that one CTA of the compaction
takes, capacities that cut at a block's edge or inside one, texts around the
threads of a CTA and at the byte limit, drafts of more tokens than threads,
tokens around eight bytes (where the index's keys change); and the delta-pos
histogram around its launch shapes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
from test_gpu_encode import check, gpu_encode, rand_vocab

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)


@pytest.fixture(scope="module")
def vocabs():
    rng = np.random.default_rng(5)
    return (W.Vocab.from_strings(rand_vocab(rng, 600, 11, b"ab\x00").strings + [b""]),
            rand_vocab(rng, 900, 11, b"ab\x00", dup=20))


@pytest.mark.parametrize("B", [1, 2, 151, 152, 153, 304, 305, 40000])
def test_batches_and_capacities(vocabs, B):
    vd, vt = vocabs
    rng = np.random.default_rng(B)
    ks = rng.integers(0, 6, B)  # some requests are empty
    d_off = np.concatenate([[0], np.cumsum(ks)]).astype(np.int32)
    d_ids = rng.integers(0, len(vd.strings), max(1, int(d_off[-1]))).astype(np.int32)
    d_ids[rng.random(d_ids.size) < 0.01] = len(vd.strings)  # ids out of range
    args = (d_off, d_ids, vd.blob, vd.off, vt.blob, vt.off, 64)
    full = oracle.encode(*args)
    n = int(full["target_off"][-1])
    edge = int(full["target_off"][min(B, max(1, B // 2))])
    for cap in sorted({0, 1, edge, max(0, edge - 1), edge + 1, max(0, n - 1), n, n + 7}):
        check(gpu_encode(d_off, d_ids, vd, vt, 64, capacity=cap), oracle.encode(*args, capacity=cap))


@pytest.mark.parametrize("n_bytes", [1, 7, 8, 9, 127, 128, 129, 255, 257, 2047, 2048, 2049])
def test_texts_of_a_given_length(vocabs, n_bytes):
    _, vt = vocabs
    rng = np.random.default_rng(n_bytes)
    vd = W.Vocab.from_strings([bytes([c]) for c in b"ab\x00"] + [b"ab" * 4, b""])
    one = rng.integers(0, 3, n_bytes).astype(np.int32)             # a byte per token
    gaps = np.insert(one, rng.integers(0, n_bytes + 1, 300), 4)    # and empty tokens between
    d_off = np.cumsum([0, one.size, gaps.size]).astype(np.int32)
    d_ids = np.concatenate([one, gaps]).astype(np.int32)
    g = gpu_encode(d_off, d_ids, vd, vt, 512)
    check(g, oracle.encode(d_off, d_ids, vd.blob, vd.off, vt.blob, vt.off, 512))


@pytest.mark.parametrize("k,m", [(1, 1), (31, 33), (32, 64), (129, 257), (256, 512)])
def test_consistency_sizes(k, m):
    """Texts of the same bytes split into k and m tokens, one byte changed or not."""
    rng = np.random.default_rng(k)
    n = 3 * max(k, m)
    text = rng.choice(list(b"abc"), n).astype(np.uint8).tobytes()

    def split(parts):
        cut = np.concatenate([[0], np.sort(rng.choice(np.arange(1, n), parts - 1, False)), [n]])
        return [text[a:b] for a, b in zip(cut, cut[1:])]
    d, t = split(k), split(m)
    flip = bytearray(t[-1])
    flip[-1] ^= 1
    vd, vt = W.Vocab.from_strings(d), W.Vocab.from_strings(t + [bytes(flip)])
    ids_t = np.tile(np.arange(m), 3)
    ids_t[2 * m - 1] = m               # request 1: its last byte changed
    ids_t[2 * m] = m + 1               # request 2: an id out of range
    d_off = (np.arange(4) * k).astype(np.int32)
    t_off = (np.arange(4) * m).astype(np.int32)
    d_ids, t_ids = np.tile(np.arange(k), 3).astype(np.int32), ids_t.astype(np.int32)
    batch = tt.Batch.from_host(d_off, d_ids, t_off, t_ids)
    g = tt.tt_consistency(batch, tt.VocabTable.from_host(vd.blob, vd.off, "cuda"),
                          tt.VocabTable.from_host(vt.blob, vt.off, "cuda")).cpu().numpy()[:3]
    o = oracle.consistency(d_off, d_ids, t_off, t_ids, vd.blob, vd.off, vt.blob, vt.off, 256, 512)
    assert np.array_equal(g, o)
    assert list(o) == [0, oracle.ST_INCONSISTENT, oracle.ST_ID_RANGE]


@pytest.mark.parametrize("B", [1, 4, 5, 1216, 1217, 5000])
def test_dpos_hist_batches(B):
    """Batches around the CTA's warps and around the size where CTAs grow; paths
    around the entries a warp has in flight."""
    rng = np.random.default_rng(B)
    k, m = rng.integers(1, 80, B), rng.integers(1, 80, B)
    d_off = np.concatenate([[0], np.cumsum(k)]).astype(np.int32)
    t_off = np.concatenate([[0], np.cumsum(m)]).astype(np.int32)
    lens = np.minimum(k + m, rng.choice([0, 1, 31, 32, 33, 127, 128, 129, 160], B)).astype(np.int32)
    path = rng.integers(0, 90, 2 * (int(d_off[-1]) + int(t_off[-1]))).astype(np.int32)
    mp = rng.integers(0, 80, int(t_off[-1])).astype(np.int32)
    batch = tt.Batch.from_host(d_off, np.zeros(int(d_off[-1])), t_off, np.zeros(int(t_off[-1])))
    dev = [torch.as_tensor(x, device="cuda") for x in (path, lens, mp)]
    for mode in (0, 1):
        g = tt.tt_dpos_hist(batch, *dev, mode, 40).cpu().numpy()
        assert np.array_equal(g, oracle.dpos_hist(d_off, t_off, path, lens, mp, mode, 40))
