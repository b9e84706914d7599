"""The repetition penalty's per-request sets (one entry per column, grouped by
row unit) and the two ways a row takes them (fp32 units in place, bf16 units
left out and added back), at the sizes where they can go wrong, against the
oracle: counts around a warp and at the cap, one column repeated, a whole unit
penalized, ragged tails, families of different types."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
from _parity import compare, oracle_step, to_np

pytestmark = pytest.mark.gpu
PEN = dict(temp_draft=0.7, temp_target=0.7, top_k_draft=20, top_p_draft=0.8, top_k_target=20,
           top_p_target=0.8, rep_penalty_draft=1.1, rep_penalty_target=1.3)
CAP = 3072  # columns of a history


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)


def _padded(t):
    """Rows padded to 16 bytes plus one more vector, the padding NaN."""
    R, V = t.shape
    per16 = 16 // t.element_size()
    buf = torch.full((R, (V + per16 - 1) // per16 * per16 + per16), float("nan"),
                     dtype=t.dtype, device="cuda")
    buf[:, :V] = t.to("cuda")
    return buf[:, :V]


def _histories(V, top, rng):
    """One history per request: the shapes named above, each with the rows' own
    leading columns (which decide the lists)."""
    tail = np.arange(V - 9, V)
    unit = np.arange(2048, min(4096 + 5, V)) if V > 2048 else np.arange(V)
    shapes = [np.array([], np.int64), rng.integers(0, V, 1), rng.integers(0, min(V, 2048), 31),
              rng.integers(0, min(V, 2048), 32), rng.integers(0, min(V, 2048), 33),
              np.full(CAP, V - 1), rng.integers(0, V, CAP), np.concatenate([tail, tail[::-1]]),
              unit, rng.permutation(V)[:CAP]]
    return [np.concatenate([s, top[i]])[-CAP:] if i else s for i, s in enumerate(shapes)]


@pytest.mark.parametrize("V", [257, 4099, 20011])
@pytest.mark.parametrize("dt_d,dt_t", [(torch.float32, torch.float32),
                                       (torch.bfloat16, torch.bfloat16),
                                       (torch.float32, torch.bfloat16),
                                       (torch.bfloat16, torch.float32)])
@pytest.mark.parametrize("families", ["both", "draft", "target"])
def test_sets_at_edges(V, dt_d, dt_t, families):
    B, G = 10, 4
    wl = W.homogeneous_workload(B, G, V, seed=V, logit_scale=2.5)
    wl = dataclasses.replace(wl, draft_logits=wl.draft_logits.to(dt_d),
                             target_logits=wl.target_logits.to(dt_t))
    rng = np.random.default_rng(V)
    h = {}
    for fam, logits in (("d", wl.draft_logits), ("t", wl.target_logits)):
        lead = torch.topk(logits.float().reshape(B, -1, V), 6, dim=2).indices.reshape(B, -1)
        hs = _histories(logits.shape[1], lead.numpy(), rng)
        h["hist_off_" + fam] = np.concatenate([[0], np.cumsum([len(x) for x in hs])]).astype(np.int32)
        h["hist_cols_" + fam] = np.concatenate(hs).astype(np.int32)
    wl = dataclasses.replace(wl, **h)
    f = dict(PEN)
    if families == "draft":
        f["rep_penalty_target"] = 1.0
    if families == "target":
        f["rep_penalty_draft"] = 1.0
    inp = tt.device_inputs(wl, "cuda")
    for k, v in f.items():
        setattr(inp["params"], k, v)
    g = to_np(tt.tt_step(inp["batch"], inp["vd"], inp["vt"], _padded(wl.draft_logits),
                         _padded(wl.target_logits), inp["params"]))
    compare(wl, g, oracle_step(wl, **f))


def _with_offsets(wl, off):
    """The workload with every family's history offsets replaced."""
    return dataclasses.replace(wl, hist_off_t=np.array(off, np.int32),
                               hist_off_d=np.array(off, np.int32))


@pytest.mark.parametrize("B", [1024, 1025, 3000])
def test_bad_history_ranges_in_large_batches(B):
    """The two ways the offsets are looked over (by every CTA, and by a kernel
    ahead of them from 1025 requests on): falls at both ends of the batch."""
    G, V, L = 2, 300, 30
    wl = W.homogeneous_workload(B, G, V, seed=B, logit_scale=2.0)
    rng = np.random.default_rng(B)
    good = np.arange(B + 1) * L
    off = good.copy()
    off[2] = off[1] - 5      # request 1 is bad; request 2 reaches back 35: into request 0's place
    off[B - 1] = off[B] + 7  # request B - 2 takes more than its share, B - 1 is bad
    cols = rng.integers(0, V, size=B * L + 7).astype(np.int32)
    wl = dataclasses.replace(wl, hist_cols_t=cols, hist_cols_d=cols)
    inp = tt.device_inputs(_with_offsets(wl, off), "cuda")
    inp["batch"].n_hist_d = inp["batch"].n_hist_t = B * L + 7
    for k, v in PEN.items():
        setattr(inp["params"], k, v)
    g = to_np(tt.tt_step(inp["batch"], inp["vd"], inp["vt"], _padded(wl.draft_logits),
                         _padded(wl.target_logits), inp["params"]))
    bad = [1, 2, B - 1]
    assert np.all(g["status"][bad] == oracle.ST_BAD_OFFSETS)
    assert np.all(np.delete(g["status"], bad) == 0)
    g["_target_off"], g["_draft_off"] = wl.target_off, wl.draft_off
    whole = _with_offsets(wl, off)
    for b in [0, 3, B // 2, B - 3, B - 2]:
        sw = whole.subset([b])
        compare(sw, dict(g), oracle_step(sw, request_base=b, **PEN), req_index=[b])


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("bad,refused,off", [
    # which request's range is bad, which others are refused, the offset after it
    (1, (), [0, 60, 56, 180, 240, 300, 360]),     # request 2 reaches back, up to request 0's place
    (1, (2,), [0, 60, 50, 180, 240, 300, 360]),   # ... and would take part of its place
    (3, (4,), [0, 60, 120, 180, 0, 300, 360]),    # ... of three requests' places
    (0, (), [-1, 60, 120, 180, 240, 300, 360]),
    (5, (), [0, 60, 120, 180, 240, 300, 299]),
])
def test_a_bad_history_range_leaves_the_other_requests_alone(dt, bad, refused, off):
    """A request without a usable history range writes no entries (it wrote its
    tokens' entries at a place that belongs to an earlier request)."""
    B, G, V = 6, 4, 9001
    wl = W.homogeneous_workload(B, G, V, seed=3, logit_scale=2.5)
    wl = dataclasses.replace(wl, draft_logits=wl.draft_logits.to(dt),
                             target_logits=wl.target_logits.to(dt))
    rng = np.random.default_rng(1)
    # each request's history holds the leading columns of its rows
    for fam, logits in (("d", wl.draft_logits), ("t", wl.target_logits)):
        lead = torch.topk(logits.float().reshape(B, -1, V), 6, dim=2).indices.reshape(B, -1)
        cols = np.concatenate([rng.permutation(x.numpy())[:20] for x in lead for _ in range(3)])
        wl = dataclasses.replace(wl, **{"hist_cols_" + fam: cols.astype(np.int32)})
    wl = _with_offsets(wl, off)
    inp = tt.device_inputs(wl, "cuda")
    inp["batch"].n_hist_d = inp["batch"].n_hist_t = 360
    for k, v in PEN.items():
        setattr(inp["params"], k, v)
    g = to_np(tt.tt_step(inp["batch"], inp["vd"], inp["vt"], _padded(wl.draft_logits),
                         _padded(wl.target_logits), inp["params"]))
    for b in range(B):
        if b == bad or b in refused or off[b] < 0 or off[b + 1] < off[b]:
            assert g["status"][b] == oracle.ST_BAD_OFFSETS, b
        else:  # as the request alone
            sw = wl.subset([b])
            o = oracle_step(sw, request_base=b, **PEN)
            compare(sw, dict(g, _target_off=wl.target_off, _draft_off=wl.draft_off), o,
                    req_index=[b])
