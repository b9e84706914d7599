"""Top-k lists under a row's bar (units later in a row list only what can still
be in its top-k): rows whose units rise, fall, are equal, tie across units, hold
few finite logits or crowd the bar, against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2510_15545_gb300 as tt
from paper_2510_15545_gb300 import workload as W
from _parity import compare, gpu_step, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    tt.load(build_if_missing=True)


def _shape(row, kind, rng):
    V = row.numel()
    x = torch.arange(V, dtype=torch.float32)
    if kind == 0:
        return x * (8.0 / V)                                     # units rise
    if kind == 1:
        return 8.0 - x * (8.0 / V)                               # units fall
    if kind == 2:
        return torch.zeros(V)                                    # every logit ties
    if kind == 3:
        return torch.as_tensor(rng.integers(0, 3, V), dtype=torch.float32)  # ties in all units
    if kind == 4:                                                # few finite logits, late ones best
        z = torch.full((V,), -float("inf"))
        at = torch.as_tensor(rng.choice(V, 40, replace=False))
        z[at] = at.float() * (4.0 / V)
        return z
    if kind == 5:                                                # one unit holds the whole top
        z = row.clone()
        z[V // 2:V // 2 + 700] = 9.0
        return z
    return row


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [2048, 20000, 45000])
@pytest.mark.parametrize("K", [1, 20, 32])
def test_rows_of_every_shape(dtype, V, K):
    """The shapes at small sizes (one unit, ragged tails)."""
    wl = W.homogeneous_workload(14, 3, V, seed=V + K, logit_scale=2.0)
    rng = np.random.default_rng(K)
    d, t = wl.draft_logits.clone(), wl.target_logits.clone()
    for z in (d, t):
        for r in range(z.shape[0]):
            z[r] = _shape(z[r], r % 7, rng)
    wl = dataclasses.replace(wl, draft_logits=d.to(dtype), target_logits=t.to(dtype))
    f = dict(top_k_draft=K, top_k_target=K, top_p_draft=0.95, top_p_target=0.95)
    compare(wl, gpu_step(wl, **f), oracle_step(wl, **f))


def _sample(wl, f, seed, n=10):
    """One step of the whole batch; some requests against the oracle."""
    g = gpu_step(wl, **f)
    assert np.all(g["status"] == 0)
    g["_target_off"], g["_draft_off"] = wl.target_off, wl.draft_off
    picks = np.random.default_rng(seed).choice(wl.B, size=n, replace=False)
    for b in {0, wl.B - 1} | set(picks.tolist()):
        sw = wl.subset([b])
        compare(sw, dict(g), oracle_step(sw, request_base=int(b), **f), req_index=[b])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [1, 20, 32])
def test_whole_rows_on_one_cta(dtype, K):
    """So many rows that every CTA's share holds whole rows, unit after unit, and
    most units find their row's bar in place (in the batch above, a row's units lie
    on as many CTAs, and few ever see a bar)."""
    V = 45000
    B = 420 if dtype == torch.float32 else 800
    wl = W.homogeneous_workload(B, 3, V, seed=K, logit_scale=2.0, device="cuda")
    units = -(-V // (2048 if dtype == torch.float32 else 4096))
    ctas = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    assert wl.target_logits.shape[0] * units // 2 // ctas >= 1.5 * units
    x = torch.arange(V, dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(K)
    for z in (wl.draft_logits, wl.target_logits):
        # (two rows in eight stay as they are)
        z[0::8] = x * (8.0 / V)                             # units rise
        z[1::8] = 8.0 - x * (8.0 / V)                       # units fall
        z[2::8] = 0.0                                       # every logit ties
        z[3::8] = torch.randint(0, 3, z[3::8].shape, generator=gen, device="cuda").float()
        late = torch.rand(z[4::8].shape, generator=gen, device="cuda") > 1e-3
        z[4::8] = torch.where(late, torch.tensor(-float("inf"), device="cuda"), x * (4.0 / V))
        z[5::8, V // 2:V // 2 + 700] = 9.0                  # one unit holds the whole top
    wl = dataclasses.replace(wl, draft_logits=wl.draft_logits.to(dtype),
                             target_logits=wl.target_logits.to(dtype))
    _sample(wl, dict(top_k_draft=K, top_k_target=K, top_p_draft=0.95, top_p_target=0.95), K)
