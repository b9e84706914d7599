"""The workloads whose speed is followed: calls of the library's public entry
points (``paper_2510_15545_gb300.binding``) as a serving loop makes them, over
the range of its own configurations -- one request to a full serving batch,
fp32 and bf16 logits, plain sampling and every filter setting of the paper's
generation table, the DTW alignment alone, re-encoding, and verification over
a vocabulary-sharded target.

Inputs follow the package's synthetic workloads: seeded byte-string
vocabularies, Zipf logits over a permuted vocabulary, draft tokens drawn from
their own rows, target tokens their greedy re-encoding, and target rows
correlated with the draft row that spells the same bytes, which puts the
acceptance rate into the paper's range.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_15545_gb300 import binding as tt
from paper_2510_15545_gb300 import workload

# Vocabulary pairs of the configurations (draft, target).
VOCABS = [(32000, 32768), (32000, 151936), (128256, 151936), (151936, 201088)]
# Target tokens per draft token when a draft is re-encoded (measured on the
# pairs above: 1.23 to 1.34).
M_PER_K = 1.27
# Integer operations per cell of an alignment: a bit-parallel edit distance of
# two tokens of 4.5 bytes (about 12 operations a byte) and the cell's minimum.
OPS_PER_CELL = 58

# Sampling settings of the paper's generation table: (temperature, top-k,
# top-p, repetition penalty).
SAMPLING = {
    "plain": (1.0, 0, 1.0, 1.0),
    "topk": (0.6, 20, 0.95, 1.0),     # Qwen3
    "nucleus90": (0.6, 0, 0.9, 1.0),  # Llama-3.1-70B
    "nucleus95": (0.6, 0, 0.95, 1.0),  # DeepSeek-R1-Distill
    "penalty": (0.7, 20, 0.8, 1.1),   # Qwen2.5-0.5B
}
MAX_HISTORY = 1024  # longest repetition-penalty history per request


def _case(name, op, B, k, pair, dtype="f32", sampling="plain", cols=0, cols_t=0, zipf=1.1,
          noise=0.5, window=8, shards=1):
    """cols / cols_t: width of the draft / target logits rows when they are
    narrower than the vocabularies (a token's column is then its id modulo the
    width); 0: the vocabularies' own sizes."""
    return dict(name=name, op=op, B=B, k=k, V_d=VOCABS[pair][0], V_t=VOCABS[pair][1], dtype=dtype,
                sampling=sampling, cols_d=cols, cols_t=cols_t or cols, zipf=zipf, noise=noise,
                window=window, shards=shards)


def listed():
    return [
        # One interactive request: four short kernels, latency and launches.
        _case("step_b1", "step", 1, 4, 0),
        # A small serving batch over a large target vocabulary.
        _case("step_b64", "step", 64, 8, 1),
        # A full serving batch, bf16 logits: the bandwidth-bound headline.
        _case("step_b1024_bf16", "step", 1024, 8, 3, "bf16", zipf=1.0, noise=1.0),
        # Long drafts over a small verification vocabulary: alignment and many
        # short rows.
        _case("step_dtw_b4096", "step", 4096, 64, 1, cols=4096),
        # Top-k with top-p (Qwen3) on a medium bf16 batch with long drafts.
        _case("topk_b256_bf16", "step", 256, 16, 2, "bf16", "topk", zipf=1.2, noise=1.0),
        # Top-p alone: a nucleus per row, full serving batch (Llama) and a
        # small fp32 batch (DeepSeek distill).
        _case("nucleus_b1024_bf16", "step", 1024, 8, 3, "bf16", "nucleus90", zipf=1.0, noise=1.0),
        _case("nucleus_b64", "step", 64, 8, 1, "f32", "nucleus95"),
        # Repetition penalty with top-k and top-p (Qwen2.5-0.5B) over each
        # request's history.
        _case("penalty_b64", "step", 64, 8, 1, "f32", "penalty"),
        # The offset study: unbanded alignment of many pairs and the histogram
        # of the path's offsets, from which the window is chosen.
        _case("align_offsets_b4096", "align", 4096, 64, 1, window=-1),
        # The longest drafts, few of them, in the paper's window.
        _case("align_long_b32", "align", 32, 256, 2),
        # Re-encoding drafts into target tokens with the byte check.
        _case("reencode_b256", "encode", 256, 16, 2),
        # Verification over a target split by columns over four ranks.
        _case("sharded_b64", "sharded", 64, 8, 1, shards=4),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["step", "align", "encode", "sharded"], [11, 4, 2, 3])[0]
    pair = rng.randrange(len(VOCABS))
    V_d, V_t = VOCABS[pair]
    dtype = rng.choice(["f32", "bf16"])
    if op == "align":
        k = _log(rng, 4, 256)
        B = _log(rng, 1, max(1, min(4096, (4096 * 64 * 64) // (k * k))))
        c = _case("", op, B, k, pair, window=rng.choice([-1, 2, 8, 8, 16]))
    elif op == "encode":
        k = _log(rng, 2, 128)
        c = _case("", op, _log(rng, 1, 4096 * 64 // k if k > 64 else 4096), k, pair)
    else:
        sampling = rng.choice(["plain", "plain", "topk", "nucleus90", "nucleus95", "penalty"])
        if op == "sharded":
            sampling = "plain"
        k = _log(rng, 2, 64)
        # a quarter of the rows narrower than the vocabulary, odd widths among them
        narrow = rng.random() < 0.25
        cols = _log(rng, 2048, V_d) if narrow else 0
        cols_t = _log(rng, 2048, V_t) if narrow else 0
        row = ((cols or V_d) + M_PER_K * (cols_t or V_t)) * (4 if dtype == "f32" else 2)
        most = 2.5e9 if sampling == "plain" else 1.2e9
        B = _log(rng, 1, max(1, min(2048, int(most / (k * row)))))
        c = _case("", op, B, k, pair, dtype, sampling, cols, cols_t,
                  zipf=rng.choice([1.0, 1.1, 1.2]), noise=rng.choice([0.5, 1.0]),
                  window=rng.choice([4, 8, 8, 16]),
                  shards=rng.choice([2, 3, 4, 8]) if op == "sharded" else 1)
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs

_vocabs = {}


def _vocab(V_d, V_t):
    """The tables of a vocabulary pair, and the injection of the target
    strings that the draft vocabulary also holds; built once per process, as a
    program loads its tokenizers once."""
    if (V_d, V_t) not in _vocabs:
        vd, vt = workload.make_vocab_pair(V_d, V_t, seed=1000 + V_d + V_t, share=0.85)
        to_d = np.array([vd.index.get(s, -1) for s in vt.strings], dtype=np.int64)
        have = np.nonzero(to_d >= 0)[0]
        _vocabs[V_d, V_t] = dict(
            vd=vd, vt=vt, have=torch.from_numpy(have).cuda(),
            to_d=torch.from_numpy(to_d[have]).cuda(),
            len_d=np.diff(vd.off), len_t=np.diff(vt.off),
            table_d=tt.VocabTable.from_host(vd.blob, vd.off),
            table_t=tt.VocabTable.from_host(vt.blob, vt.off),
            index=tt.vocab_index(vt.blob, vt.off))
    return _vocabs[V_d, V_t]


def _widths(c):
    return c["cols_d"] or c["V_d"], c["cols_t"] or c["V_t"]


def _rows(R, V, dtype):
    """R logits rows of V columns whose stride is a multiple of 16 bytes."""
    vec = 4 if dtype == torch.float32 else 8
    stride = (V + vec - 1) // vec * vec
    return torch.zeros((R, stride), dtype=dtype, device="cuda")[:, :V]


def _blocks(R, V):
    step = max(1, (1 << 26) // V)
    for r0 in range(0, R, step):
        yield r0, min(R, r0 + step)


def _zipf_block(c, n, V, rng, gen):
    """n fp32 rows: -s log(rank) under a permutation of the columns per row,
    plus Gaussian noise."""
    a = rng.integers(1, V, size=n)
    while (bad := np.gcd(a, V) != 1).any():
        a[bad] = a[bad] % (V - 1) + 1
    a = torch.from_numpy(a).cuda()[:, None]
    b = torch.from_numpy(rng.integers(0, V, size=n)).cuda()[:, None]
    rank = (torch.arange(V, device="cuda")[None, :] * a + b) % V + 1
    z = torch.log(rank.float()).mul_(-c["zipf"])
    return z.add_(torch.randn((n, V), generator=gen, device="cuda"), alpha=c["noise"])


def _drafts(c, rng, gen, want_rows):
    """Draft ids [B, k] and, with want_rows, the draft logits rows they were
    drawn from (rows narrower than the vocabulary: ids drawn uniformly)."""
    B, k, (W, _) = c["B"], c["k"], _widths(c)
    ids = rng.integers(256, c["V_d"], size=(B, k))
    if not want_rows:
        return ids, None
    T = SAMPLING[c["sampling"]][0]
    rows = _rows(B * k, W, torch.float32 if c["dtype"] == "f32" else torch.bfloat16)
    drawn = []
    for r0, r1 in _blocks(B * k, W):
        z = _zipf_block(c, r1 - r0, W, rng, gen)
        rows[r0:r1] = z
        if not c["cols_d"]:  # the Gumbel-max draw from softmax(z / T)
            e = torch.empty_like(z).exponential_(generator=gen)
            drawn.append((z / T - torch.log(e.clamp_(min=1e-20))).argmax(1))
    if drawn:
        ids = torch.cat(drawn).cpu().numpy().reshape(B, k)
    return ids, rows


def _targets(c, rng, gen, draft_rows, d_ids, t_lists):
    """The m + 1 target rows of every request: rows over the vocabularies are
    correlated (0.9) with the draft row holding the same last byte on the
    strings both vocabularies spell, and lowered by 3 nats elsewhere."""
    v = _vocab(c["V_d"], c["V_t"])
    _, W = _widths(c)
    R = sum(len(t) + 1 for t in t_lists)
    rows = _rows(R, W, torch.float32 if c["dtype"] == "f32" else torch.bfloat16)
    src = []
    for b, t in enumerate(t_lists):
        ends = np.cumsum(v["len_d"][d_ids[b]])
        at = np.searchsorted(ends, np.cumsum(v["len_t"][t]) - 1, side="right")
        src.append(b * c["k"] + np.minimum(np.append(at, c["k"] - 1), c["k"] - 1))
    src = torch.from_numpy(np.concatenate(src)).cuda()
    for r0, r1 in _blocks(R, W):
        z = _zipf_block(c, r1 - r0, W, rng, gen)
        if not c["cols_t"] and draft_rows is not None:
            zd = draft_rows[src[r0:r1]].float()[:, v["to_d"]]
            sd = zd.std(dim=1, keepdim=True)
            noise = torch.randn(zd.shape, generator=gen, device="cuda")
            z -= 3.0
            z[:, v["have"]] = 0.9 * zd + math.sqrt(1 - 0.81) * sd * noise
        rows[r0:r1] = z
    return rows


def _history(c, rng, width):
    """Seeded histories (logits columns): mostly frequent, some rare, repeats."""
    n = rng.integers(64, MAX_HISTORY + 1, size=c["B"])
    off = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    cols = (width * rng.random(int(off[-1])) ** 3).astype(np.int32)
    return off, np.minimum(cols, width - 1)


def _room(c):
    """Target tokens the output buffers hold: as in a serving loop, they are
    sized for the batch shape and not for the tokens of one step."""
    return c["B"] * (2 * c["k"] + 8)


def _outputs(c, names):
    """Zeroed output buffers of the named outputs."""
    B, n = c["B"], _room(c)
    size = dict(accepted=B, next_token=B, status=B, path=2 * (B * c["k"] + n), path_len=B, cost=B,
                map=n, q_hat=n, p_hat=n, lse=n + B)
    return {x: torch.zeros(size[x], device="cuda",
                           dtype=torch.float32 if x in ("q_hat", "p_hat", "lse") else torch.int32)
            for x in names}


def prepare(case, seed):
    c = dict(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(1 << 31)))
    v = _vocab(c["V_d"], c["V_t"])
    B, k, (W_d, W_t) = c["B"], c["k"], _widths(c)
    ids, draft_rows = _drafts(c, rng, gen, c["op"] in ("step", "sharded"))
    strings = v["vd"].strings
    t_lists = [workload.greedy_encode(b"".join(strings[i] for i in row), v["vt"].index)
               for row in ids.tolist()]
    draft_off = np.arange(0, B * k + 1, k, dtype=np.int32)
    target_off = np.concatenate([[0], np.cumsum([len(t) for t in t_lists])]).astype(np.int32)
    t_ids = np.concatenate(t_lists).astype(np.int32)
    d_ids = ids.reshape(-1).astype(np.int32)
    batch = tt.Batch.from_host(draft_off, d_ids, target_off, t_ids,
                               d_ids % W_d if c["cols_d"] else None,
                               t_ids % W_t if c["cols_t"] else None)
    T, top_k, top_p, penalty = SAMPLING[c["sampling"]]
    params = tt.Params(window=c["window"], temp_draft=T, temp_target=T, top_k_draft=top_k,
                       top_k_target=top_k, top_p_draft=top_p, top_p_target=top_p,
                       rep_penalty_draft=penalty, rep_penalty_target=penalty, seed=int(seed))
    s = dict(case=c, batch=batch, params=params, vocab=v, off_t=target_off, d_ids=d_ids,
             t_ids=t_ids, draft=draft_rows)
    if c["op"] == "align":
        s["call"] = tt.AlignCall(batch, v["table_d"], v["table_t"], params, out=_outputs(
            c, ("path", "path_len", "cost", "map", "status")))
    elif c["op"] == "encode":
        s["max_m"] = min(tt.TT_MAX_M, 4 * k + 8)
        s["out"] = dict(target_ids=torch.zeros(B * s["max_m"], dtype=torch.int32, device="cuda"))
        s["ws"] = torch.empty(tt.tt_encode_workspace_bytes(B, s["max_m"]), dtype=torch.uint8,
                              device="cuda")
        s["status"] = torch.zeros(B, dtype=torch.int32, device="cuda")
    else:
        if penalty != 1.0:
            hd, ht = _history(c, rng, W_d), _history(c, rng, W_t)
            s["batch"] = batch = batch.with_history(*hd, *ht)
            s["hist"] = (hd, ht)
        s["target"] = target = _targets(c, rng, gen, draft_rows, ids, t_lists)
        if c["op"] == "sharded":
            s["shards"] = _split(target, c["shards"])
            # q of a target token as the transfer leaves it: a draft probability
            row = torch.from_numpy(np.repeat(np.arange(B) * k, np.diff(target_off))).cuda()
            col = torch.from_numpy(np.repeat(d_ids[::k] % W_d, np.diff(target_off))).cuda()
            s["q_hat"] = torch.cat([torch.softmax(draft_rows[x].float(), 1).gather(1, y[:, None])[:, 0]
                                    for x, y in zip(row.split(512), col.long().split(512))])
            s["ws"] = tt.sharded_workspace(batch, s["shards"])
            s["out"] = _outputs(c, ("accepted", "next_token", "status", "p_hat", "lse"))
            s["draft"] = None
        else:
            s["call"] = tt.StepCall(batch, v["table_d"], v["table_t"], draft_rows, target, params,
                                    out=_outputs(c, tt.STEP_OUTPUTS))
    return s


def _split(rows, S):
    """The rows' columns over S ranks, in order, as arrays of their own."""
    R, W = rows.shape
    cut = [W * i // S for i in range(S + 1)]
    out = []
    for a, b in zip(cut, cut[1:]):
        part = _rows(R, b - a, rows.dtype)
        part.copy_(rows[:, a:b])
        out.append(part)
    return out


def run(state):
    op, v = state["case"]["op"], state["vocab"]
    if op == "step":
        return state["call"]()
    if op == "align":
        out = state["call"]()
        hist = tt.tt_dpos_hist(state["batch"], out["path"], out["path_len"], out["map"], 0, 256)
        return dict(out, hist=hist)
    b = state["batch"]
    if op == "encode":
        out = tt.tt_encode(b.draft_off, b.draft_ids, v["table_d"], v["table_t"], v["index"],
                           state["max_m"], out=state["out"], ws=state["ws"])
        again = tt.Batch(b.draft_off, b.draft_ids, out["target_off"], out["target_ids"], B=b.B,
                         n_draft=b.n_draft, n_target=out["target_ids"].numel(), max_k=b.max_k,
                         max_m=state["max_m"])
        same = tt.tt_consistency(again, v["table_d"], v["table_t"], status=state["status"])
        return dict(out, same=same)
    return tt.tt_verify_sharded(b, state["q_hat"], state["shards"], state["params"],
                                ws=state["ws"], out=state["out"])


def work(case):
    """Logits rows and token bytes read once, outputs written once."""
    c = case
    B, k, (W_d, W_t) = c["B"], c["k"], _widths(c)
    m = M_PER_K * k
    ids = 4 * B * (k + m) + 5 * B * (k + m) + 8 * B * (k + m)  # ids, bytes, offsets
    band = m if c["window"] < 0 else min(m, 2 * max(c["window"], m - k) + 1)
    cells = B * k * band
    if c["op"] == "align":
        return {"bytes": ids + 4 * B * (2 * (k + m) + m), "flops": OPS_PER_CELL * cells}
    if c["op"] == "encode":
        return {"bytes": 2 * ids + 16 * 5 * B * k + 4 * B * m, "flops": 0}
    esz = 4 if c["dtype"] == "f32" else 2
    need = 0 if c["op"] == "sharded" else 0.95 * B * k * W_d
    logits = esz * (need + B * (m + 1) * W_t)
    per_logit = 3  # scale, exponential, sum
    return {"bytes": logits + ids + 16 * B * m,
            "flops": per_logit * logits / esz + (0 if c["op"] == "sharded" else OPS_PER_CELL * cells)}


def tolerance(case):
    if case["op"] in ("align", "encode"):
        return "exact"
    # 32-bit sums and special-function exponentials (1.1e-7 off the 64-bit
    # values at most, as 2-norms); a draw whose uniform lies within rounding of
    # a column's boundary may give the neighbouring column (2 of 1024 requests
    # when the sums are taken in another order)
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.005}


# -------------------------------------------------- the same in 64 bits

def _row_stats(z, cols, T, top_k, top_p):
    """(probability of each row's column, natural log of the kept normaliser)
    of fp32 rows z under the filters, in 64 bits; cols < 0: probability 0."""
    n, V = z.shape
    at = cols.clamp(min=0)[:, None]
    if top_k == 0 and not top_p < 1:
        lse = torch.logsumexp(z.double() / T, 1)
        p = torch.exp(z.gather(1, at)[:, 0].double() / T - lse)
        return torch.where(cols >= 0, p, 0.0), lse
    v, i = torch.sort(z, dim=1, descending=True, stable=True)
    if top_k:
        v, i = v[:, :top_k], i[:, :top_k]
    e = torch.exp((v.double() - v[:, :1].double()) / T)
    if top_p < 1:
        before = torch.cumsum(e, 1) - e
        e = torch.where(before < top_p * e.sum(1, keepdim=True), e, 0.0)
    S = e.sum(1)
    p = torch.where(i == at, e, 0.0).sum(1) / S
    return torch.where(cols >= 0, p, 0.0), torch.log(S) + v[:, 0].double() / T


def _stats(rows, cols, sampling, penal=None):
    T, top_k, top_p, penalty = SAMPLING[sampling]
    ps, ls = [], []
    for r0, r1 in _blocks(len(rows), 2 * rows.shape[1]):
        z = rows[r0:r1].float()
        if penal is not None:
            for r in range(r0, r1):
                x = torch.from_numpy(penal[r]).cuda()
                y = z[r - r0, x]
                z[r - r0, x] = torch.where(y < 0, y * penalty, y / penalty)
        p, lse = _row_stats(z, cols[r0:r1], T, top_k, top_p)
        ps.append(p)
        ls.append(lse)
    return torch.cat(ps), torch.cat(ls)


def _penalized(off, ids, extra, hist):
    """Unique penalized columns of every row: the request's history and its
    sequence tokens before the row (extra: rows beyond the tokens)."""
    h_off, h_cols = hist
    out = []
    for b in range(len(off) - 1):
        seq, h = ids[off[b]:off[b + 1]], h_cols[h_off[b]:h_off[b + 1]]
        for j in range(len(seq) + extra):
            out.append(np.unique(np.concatenate([h, seq[:j]])).astype(np.int64))
    return out


def _edit_distances(v, D, T):
    """Levenshtein distances [B, k, m] of the byte strings of ids D [B, k] and
    T [B, m] (tokens of at most 8 bytes; padding ids are ignored later)."""
    def table(voc, ids):
        n = np.diff(voc.off)[ids]
        at = voc.off[:-1][ids][..., None] + np.arange(8)
        b = np.where(np.arange(8) < n[..., None], voc.blob[np.minimum(at, len(voc.blob) - 1)], 0)
        return torch.from_numpy(b).cuda(), torch.from_numpy(n).cuda()
    (bd, nd), (bt, nt) = table(v["vd"], D), table(v["vt"], T)
    bd, nd, bt, nt = bd[:, :, None], nd[:, :, None], bt[:, None], nt[:, None]
    shape = torch.broadcast_shapes(nd.shape, nt.shape)
    row = [torch.full(shape, j, dtype=torch.int8, device="cuda") for j in range(9)]
    out = nt.expand(shape).to(torch.int8).clone()
    for i in range(1, 9):
        new = [torch.full(shape, i, dtype=torch.int8, device="cuda")]
        for j in range(1, 9):
            same = (bd[..., i - 1] == bt[..., j - 1]).to(torch.int8)
            new.append(torch.minimum(torch.minimum(row[j], new[j - 1]) + 1, row[j - 1] + 1 - same))
        row = new
        for j in range(9):
            out = torch.where((nd == i) & (nt == j), row[j], out)
    return out.int()


def _map(c, v, off_t, d_ids, t_ids):
    """The draft index aligned to each target token: banded DTW, backtrack
    preferring the diagonal, then the previous draft token."""
    B, k = c["B"], c["k"]
    m = np.diff(off_t)
    M = int(m.max())
    T = np.zeros((B, M), dtype=np.int64)
    for b in range(B):
        T[b, :m[b]] = t_ids[off_t[b]:off_t[b + 1]]
    D = d_ids.reshape(B, k).astype(np.int64)
    cost = torch.cat([_edit_distances(v, D[i:i + 256], T[i:i + 256]) for i in range(0, B, 256)])
    mt = torch.from_numpy(m).cuda()
    w = torch.full_like(mt, k + M) if c["window"] < 0 else \
        torch.maximum((mt - k).abs(), torch.full_like(mt, c["window"]))
    inf = 1 << 28
    C = torch.full((k + 1, M + 1, B), inf, dtype=torch.int32, device="cuda")
    C[0, 0] = 0
    cost = cost.permute(1, 2, 0).contiguous()
    for i in range(1, k + 1):
        for j in range(1, M + 1):
            best = torch.minimum(torch.minimum(C[i - 1, j - 1], C[i - 1, j]), C[i, j - 1])
            C[i, j] = torch.where(w >= abs(i - j), (best + cost[i - 1, j - 1]).clamp(max=inf), inf)
    at = torch.arange(B, device="cuda")
    i, j = torch.full_like(mt, k), mt.clone()
    out = torch.full((B, M + 1), -1, dtype=torch.int64, device="cuda")
    for _ in range(k + M):
        go = (i > 0) & (j > 0)
        i, j = i.clamp(min=0), j.clamp(min=0)
        out[at, j] = torch.where(go, torch.maximum(out[at, j], i - 1), out[at, j])
        a, b = (i - 1).clamp(min=0), (j - 1).clamp(min=0)
        dg, up, left = C[a, b, at], C[a, j, at], C[i, b, at]
        diag = (dg <= up) & (dg <= left)
        up_ = ~diag & (up <= left)
        i = torch.where(go & (diag | up_), i - 1, i)
        j = torch.where(go & (diag | ~up_), j - 1, j)
    out = out[:, 1:]
    return torch.cat([out[b, :m[b]] for b in range(B)])


def exact(case, seed):
    """p_hat, q_hat and lse in 64 bits; whole-number outputs have no such value."""
    if case["op"] in ("align", "encode"):
        return None
    s = prepare(case, seed)
    c, off_t = s["case"], s["off_t"]
    W_d, W_t = _widths(c)
    B = c["B"]
    # target row r of request b scores its token; the last one is the bonus row
    cols = np.full(len(s["t_ids"]) + B, -1, dtype=np.int64)
    is_token = np.ones(len(cols), dtype=bool)
    is_token[off_t[1:] + np.arange(B)] = False
    cols[is_token] = s["t_ids"] % W_t
    hist = s.get("hist")
    off_d = np.arange(0, B * c["k"] + 1, c["k"])
    penal_t = _penalized(off_t, s["t_ids"] % W_t, 1, hist[1]) if hist else None
    p, lse = _stats(s["target"], torch.from_numpy(cols).cuda(), c["sampling"], penal_t)
    n = _room(c)

    def pad(x, size):
        return torch.cat([x, x.new_zeros(size - len(x))])
    out = dict(accepted=None, next_token=None, status=None,
               p_hat=pad(p[torch.from_numpy(is_token).cuda()], n), lse=pad(lse, n + B))
    if c["op"] == "step":
        penal_d = _penalized(off_d, s["d_ids"] % W_d, 0, hist[0]) if hist else None
        q, _ = _stats(s["draft"], torch.from_numpy(s["d_ids"] % W_d).cuda().long(), c["sampling"],
                      penal_d)
        i = _map(c, s["vocab"], off_t, s["d_ids"], s["t_ids"])
        base = torch.from_numpy(np.repeat(off_d[:-1], np.diff(off_t))).cuda()
        out.update(path=None, path_len=None, cost=None, map=None, q_hat=pad(q[base + i], n))
    return out
