"""The sharded verification's shared row pass and column draw where they can go
wrong: shards of both types in one call, shards that end inside a stage, more
rows than a warp merges at once, and a residual at the row's last column. The
oracle works on the whole rows, holding what the shards hold."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
from _parity import compare, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)


def _shard(cols, dtype):
    """A slice as its own tensor, rows padded to 16 bytes and a vector of NaN."""
    per16 = 16 // torch.empty(0, dtype=dtype).element_size()
    R, w = cols.shape
    buf = torch.full((R, (w + per16 - 1) // per16 * per16 + per16), float("nan"), dtype=dtype,
                     device="cuda")
    buf[:, :w] = cols.to("cuda").to(dtype)
    return buf[:, :w]


F, H = torch.float32, torch.bfloat16


@pytest.mark.parametrize("B,G,widths,dtypes", [
    (5, 3, [2048, 2049, 4096], [F, H, F]),
    (5, 3, [1, 4097, 1, 6000], [H, F, H, H]),
    (3, 40, [3000, 1111, 17, 5000, 2047, 1, 900, 4095], [H, F, F, H, H, F, H, F]),
    (40, 4, [70001, 9999], [H, F]),
    (1, 1, [7], [H]),
])
def test_shards_of_both_types(B, G, widths, dtypes):
    V = sum(widths)
    wl = W.homogeneous_workload(B, G, V, seed=V, logit_scale=1.5)
    whole, shards, c = wl.target_logits.clone(), [], 0
    # some requests' rows end at their last column: the draw lands there
    whole[::5, -1] += 12.0
    for w, dt in zip(widths, dtypes):
        shards.append(_shard(whole[:, c:c + w], dt))
        whole[:, c:c + w] = shards[-1].float().cpu()
        c += w
    wl = dataclasses.replace(wl, target_logits=whole)
    inp = tt.device_inputs(wl, "cuda")
    prm = inp["params"]
    q = np.random.default_rng(V).uniform(0.0, 0.02, int(wl.target_off[-1])).astype(np.float32)
    g = to_np(tt.tt_verify_sharded(inp["batch"], torch.as_tensor(q, device="cuda"), shards, prm))
    o = oracle.verify(wl.target_off, wl.target_cols, q, whole, seed=prm.seed)
    g, o = dict(g, q_hat=q), dict(o, q_hat=q)
    compare(wl, g, o, check_align=False)
