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


# Seeds, and columns with -log2 of their masses (all others have none), of a
# bonus row whose uniform falls between two roundings of one running mass: the
# pair sum that a thread ends on is at or below it, the sum from which one of the
# next threads starts, added up in another order, is above it by its last bit,
# and that thread's first columns have no mass.
BETWEEN = [
    (99, {
        18: 19, 28: 42, 32: 1, 51: 49, 55: 15, 57: 38, 320: 18, 427: 17, 447: 13, 505: 11,
        513: 48, 550: 51, 561: 23, 601: 44, 645: 37, 683: 53, 713: 41, 718: 9, 761: 21, 796: 3,
        880: 22, 914: 52, 920: 5, 1025: 12, 1067: 54, 1079: 50, 1089: 53, 1098: 54, 1140: 29,
        1154: 32, 1161: 53, 1206: 47, 1620: 0}),
    (220, {
        42: 47, 149: 36, 165: 33, 259: 8, 267: 15, 343: 46, 502: 32, 560: 16, 569: 35, 600: 34,
        695: 5, 752: 20, 765: 53, 769: 10, 804: 52, 817: 39, 824: 29, 841: 11, 853: 1, 1002: 28,
        1126: 7, 1215: 23, 1282: 52, 1314: 40, 1330: 43, 1351: 21, 1364: 52, 1947: 0}),
    (252, {
        13: 16, 140: 17, 185: 40, 198: 31, 256: 8, 491: 34, 507: 47, 677: 9, 706: 53, 718: 36,
        740: 37, 807: 12, 818: 43, 825: 3, 873: 13, 920: 23, 938: 30, 1022: 1, 1061: 33,
        1094: 29, 1130: 5, 1190: 53, 2009: 0}),
]


@pytest.mark.parametrize("seed,masses", BETWEEN)
def test_a_column_without_mass_is_never_drawn(seed, masses):
    V = 2048
    wl = W.homogeneous_workload(1, 1, V, seed=1)
    z = torch.full((2, V), -float("inf"))
    z[0] = 0.0
    for c, e in masses.items():
        z[1, c] = -float(e)
    wl = dataclasses.replace(wl, target_logits=z)
    inp = tt.device_inputs(wl, "cuda")
    prm = inp["params"]
    prm.seed, prm.temp_target = seed, float(np.log2(np.e))  # masses are 2^z exactly
    q = torch.zeros(1, device="cuda")                       # the token is accepted
    g = to_np(tt.tt_verify_sharded(inp["batch"], q, [z.to("cuda")], prm, summaries=True))
    assert g["status"][0] == 0 and g["accepted"][0] == 1
    # the row's total, against which the uniform is taken: the masses of 2^-23 and more
    total = np.float32(sum(2.0 ** -e for e in masses.values() if e <= 23))
    assert g["summaries"][0, 1, 0] == 0.0 and g["summaries"][0, 1, 1] == total
    assert int(g["next_token"][0]) in masses
