"""The nucleus row kernel (rows of more than four 8 KB units: 8192 fp32 or 16384
bf16 columns; top-p without top-k) at the edges of its forms, against the
oracle: units and rounds of units that do not fill, ragged tails, families of
different types (and routes), masked columns, rows whose maxima lie far apart
(the expected maximum of a row is then wrong), flat rows whose candidates
overflow, and its bounded waits."""
import dataclasses
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import torch

import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
from _parity import compare, gpu_step, oracle_step, to_np

pytestmark = pytest.mark.gpu
LLAMA = dict(temp_draft=0.6, temp_target=0.6, top_p_draft=0.9, top_p_target=0.9)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)


def _padded(t: torch.Tensor) -> torch.Tensor:
    """Rows padded to 16 bytes plus one more vector, the padding NaN."""
    R, V = t.shape
    per16 = 16 // t.element_size()
    buf = torch.full((R, (V + per16 - 1) // per16 * per16 + per16), float("nan"),
                     dtype=t.dtype, device="cuda")
    buf[:, :V] = t.to("cuda")
    return buf[:, :V]


def _check(wl, f=LLAMA):
    inp = tt.device_inputs(wl, "cuda")
    prm = inp["params"]
    for k, v in f.items():
        setattr(prm, k, v)
    g = to_np(tt.tt_step(inp["batch"], inp["vd"], inp["vt"], _padded(wl.draft_logits),
                         _padded(wl.target_logits), prm))
    compare(wl, g, oracle_step(wl, **f))


# a unit is 2048 fp32 or 4096 bf16 columns, a round 20 units
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [8192, 8193, 8199, 10240, 16384, 16385, 40960, 40961, 81919, 81920,
                               83967, 122887])
def test_widths_at_edges(V, dtype):
    _check(W.homogeneous_workload(4, 3, V, seed=V, dtype=dtype, logit_scale=2.5))


@pytest.mark.parametrize("V", [983040, 983041])
def test_widths_around_the_widest(V):
    """The widest rows of the row kernel, and the first that go past it."""
    _check(W.homogeneous_workload(1, 2, V, seed=3, logit_scale=2.5))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [8199, 20011, 40961, 81919])
def test_many_rows_per_cta(V, dtype):
    """Nine rows and more on each CTA: the row buffers and the queue are used
    again and again, short last rounds move from warp to warp, and rows are
    expected to reach the maxima of those before them."""
    wl = W.homogeneous_workload(200, 3, V, seed=V, dtype=dtype, logit_scale=2.5, device="cuda")
    assert 7 * wl.B >= 9 * torch.cuda.get_device_properties(0).multi_processor_count
    g = gpu_step(dataclasses.replace(wl, draft_logits=_padded(wl.draft_logits),
                                     target_logits=_padded(wl.target_logits)), **LLAMA)
    assert np.all(g["status"] == 0)
    g["_target_off"], g["_draft_off"] = wl.target_off, wl.draft_off
    for b in np.random.default_rng(V).choice(wl.B, size=12, replace=False):
        sw = wl.subset([b])
        compare(sw, dict(g), oracle_step(sw, request_base=int(b), **LLAMA), req_index=[b])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("sigma", [0.0, 0.3, 1.0, 2.0])
def test_flat_rows_raise_their_bar(sigma, dtype):
    """Every unit holds more candidates than a warp has room for, by some or by
    all of its columns (equal logits: no bar leaves room), and a ragged unit."""
    wl = W.homogeneous_workload(5, 3, 30005, seed=int(10 * sigma), logit_scale=max(sigma, 0.1))
    if sigma == 0.0:
        wl = dataclasses.replace(wl, draft_logits=torch.zeros_like(wl.draft_logits),
                                 target_logits=torch.full_like(wl.target_logits, 2.0))
    wl = dataclasses.replace(wl, draft_logits=wl.draft_logits.to(dtype),
                             target_logits=wl.target_logits.to(dtype))
    for p in (0.3, 0.95):
        _check(wl, dict(LLAMA, top_p_draft=p, top_p_target=p))


@pytest.mark.parametrize("V", [12007, 20011])  # (12007: bf16 rows take the row pass)
def test_families_of_different_types(V):
    wl = W.homogeneous_workload(6, 4, V, seed=3, logit_scale=2.5)
    _check(dataclasses.replace(wl, draft_logits=wl.draft_logits.to(torch.bfloat16)))
    _check(dataclasses.replace(wl, target_logits=wl.target_logits.to(torch.bfloat16)))


def test_maxima_far_apart_and_masked_columns():
    """Rows shifted by up to 40 (a softmax does not see it) and half of the
    columns of some rows at -inf; flat rows beside peaked ones."""
    wl = W.homogeneous_workload(200, 3, 16411, seed=9, logit_scale=2.0)
    rng = np.random.default_rng(1)
    tl = wl.target_logits.clone()
    R, V = tl.shape
    tl[::3] *= 0.1
    tl += torch.as_tensor(rng.uniform(-40, 40, size=(R, 1)).astype(np.float32))
    keep = torch.zeros((R, V), dtype=torch.bool)
    keep.scatter_(1, torch.as_tensor(wl.target_cols.reshape(200, 3).repeat(4, 0)).long(), True)
    mask = torch.as_tensor(rng.random((R, V)) < 0.5) & ~keep
    mask[::2] = False
    tl[mask] = -float("inf")
    wl = dataclasses.replace(wl, target_logits=tl)
    _check(wl.subset(range(24)))
    _check(wl, dict(temp_target=0.6, top_p_target=0.9))


def test_rows_without_a_finite_logit():
    """A row of a request that has no finite logit: TT_REQ_NOT_FINITE for that
    request, the others as without it."""
    wl = W.homogeneous_workload(3, 2, 9004, seed=2)
    tl = wl.target_logits.clone()
    tl[4] = -float("inf")  # the middle request's second row
    outs = []
    for x in (wl.target_logits, tl):
        inp = tt.device_inputs(dataclasses.replace(wl, target_logits=x), "cuda")
        for k, v in LLAMA.items():
            setattr(inp["params"], k, v)
        outs.append(to_np(tt.tt_step(inp["batch"], inp["vd"], inp["vt"], inp["draft_logits"],
                                     inp["target_logits"], inp["params"])))
    assert list(outs[1]["status"]) == [0, 16, 0]
    for key in ("accepted", "next_token"):
        assert list(outs[1][key][[0, 2]]) == list(outs[0][key][[0, 2]])


CHILD = """
import torch, paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
wl = W.homogeneous_workload(160, 2, 40000, seed=1)
inp = tt.device_inputs(wl, "cuda")
prm = inp["params"]
prm.temp_target = prm.temp_draft = 0.6
prm.top_p_target = prm.top_p_draft = 0.9
a = tt.tt_step(inp["batch"], inp["vd"], inp["vt"], inp["draft_logits"], inp["target_logits"], prm)
first = a["status"].cpu().tolist()
b = tt.tt_step(inp["batch"], inp["vd"], inp["vt"], inp["draft_logits"], inp["target_logits"], prm)
second = b["status"].cpu().tolist()
print("FIRST", all(s == 32 for s in first), "SECOND", all(s == 0 for s in second))
"""


def test_bounded_waits_of_the_nucleus_row_kernel():
    """One copy is never made: the waits for it run out and the call reports
    TT_REQ_TIMEOUT on every request; the next call runs normally."""
    env = dict(os.environ, TT_TEST_STALL_STAGE="3", TT_TEST_WAIT_MS="50")
    t0 = time.monotonic()
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True,
                       timeout=240, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert "FIRST True SECOND True" in r.stdout, (r.stdout[-500:], r.stderr[-500:])
    assert time.monotonic() - t0 < 200
