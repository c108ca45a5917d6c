"""Performance cases of the framework: what its users have it do, by kind of call and size.

A serving loop runs one ROUND per decoding step: the drafter's backbone over every acceptance boundary, the
verification outcome with the selected branch, the drafter's head, and the append of the verified features to the
drafter's cache.  The cases time the calls of that round one by one (a loop that overlaps them with the target's own
work issues them one by one, on different streams) and, for small batches, the whole round as it is issued on one
stream.  Every case goes through the plan objects, which a serving loop builds once and keeps.

Kinds (`kind` of a case):
  step      all-boundary attention, then greedy verify/select on the attention's own output
  select    verify/select in sampling mode (rejection rule, bonus draw, branch gather)
  block     one full backbone block: norms, projections, attention, gated MLP (spine keys and values supplied)
  backbone  a stack of blocks with the spine tokens as query rows
  head      language-model head on the selected branch and the autoregressive head loop, greedy or sampling
  append    projection of the verified features into every drafter layer's cache, in place
  round     backbone -> greedy verify/select -> head -> append
"""
import math

import numpy as np
import torch

import paper_2609_27396_b200 as dp

VOCAB = 151936
DEV = "cuda"


# ------------------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # a small model and one short request: the calls' fixed cost
        dict(name="step_tiny", kind="step", b=1, ctx_lo=128, ctx_hi=128, hq=4, hkv=2, d=64, j=5, bq=4, vocab=1000, agree=0.8),
        # one interactive user on an 8B-shaped model, draft length 7
        dict(name="step_b1", kind="step", b=1, ctx_lo=2048, ctx_hi=2048, hq=32, hkv=8, d=128, j=8, bq=8, vocab=VOCAB, agree=0.8),
        # a batch of ragged contexts on a 14B-shaped model, draft length 15: the default benchmark workload
        dict(name="step_b16", kind="step", b=16, ctx_lo=512, ctx_hi=4096, hq=40, hkv=8, d=128, j=16, bq=16, vocab=VOCAB, agree=0.75),
        # sampling users: rejection rule on probabilities
        dict(name="select_sampling_b8", kind="select", b=8, j=16, bq=16, hidden=4096, vocab=VOCAB),
        # long documents: 32 K tokens of context for each of four requests, one whole block
        dict(name="block_long_b4", kind="block", b=4, ctx_lo=32768, ctx_hi=32768, hq=32, hkv=8, d=128, j=16, bq=16, hidden=4096, inter=12288),
        # one interactive user: the drafter's five layers over 72 rows (reading the weights is the work)
        dict(name="backbone_b1", kind="backbone", b=1, ctx_lo=2048, ctx_hi=2048, hq=32, hkv=8, d=128, j=8, bq=8, hidden=4096, inter=12288, layers=5),
        # a full batch: two layers of a 14B-shaped drafter over 1152 rows
        dict(name="backbone_b16", kind="backbone", b=16, ctx_lo=512, ctx_hi=4096, hq=40, hkv=8, d=128, j=8, bq=8, hidden=5120, inter=17408, layers=2),
        # the remainder of the critical path for a full batch, greedy decoding
        dict(name="head_b16", kind="head", b=16, bq=16, hidden=5120, vocab=VOCAB, rank=256, sampling=False),
        # ... and for sampling users
        dict(name="head_sampling_b8", kind="head", b=8, bq=16, hidden=4096, vocab=VOCAB, rank=256, sampling=True),
        # cache update of five drafter layers for a full batch
        dict(name="append_b16", kind="append", b=16, ctx_lo=512, ctx_hi=4096, j=16, hkv=8, d=128, feat=5120, layers=5),
        # the whole round, one user
        dict(name="round_b1", kind="round", b=1, ctx_lo=2048, ctx_hi=2048, hq=32, hkv=8, d=128, j=8, bq=8, hidden=4096, inter=12288, layers=5,
             vocab=VOCAB, rank=256, agree=0.8),
        # the whole round, four users with ragged contexts
        dict(name="round_b4", kind="round", b=4, ctx_lo=300, ctx_hi=3000, hq=32, hkv=8, d=128, j=8, bq=8, hidden=4096, inter=12288, layers=2,
             vocab=VOCAB, rank=256, agree=0.8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.5e15)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= most:
            return case


def _draw(rng):
    kind = rng.choice(["step", "step", "select", "block", "backbone", "backbone", "head", "head", "append", "round"])
    b = _log_int(rng, 1, 16)
    j, bq = rng.randint(2, 16), rng.randint(1, 16)
    # heads per KV head as in the shapes listed and tested; small models have 64-wide heads
    d = rng.choice([64, 128, 128])
    hkv, group = rng.choice([2, 4, 8]), rng.choice([1, 2, 4, 4, 5, 8])
    ctx_hi = _log_int(rng, 16, 32768 if b <= 4 else 4096)
    ctx_lo = max(1, int(ctx_hi * rng.uniform(0.1, 1.0)))
    heads = dict(hq=hkv * group, hkv=hkv, d=d)
    ctx = dict(b=b, ctx_lo=ctx_lo, ctx_hi=ctx_hi)
    vocab = rng.choice([VOCAB, _log_int(rng, 1000, VOCAB)])          # any width, odd ones among them
    hidden = 64 * _log_int(rng, 8, 80)                               # 512 .. 5120
    inter = 64 * max(8, int(hidden / 64 * rng.uniform(2.5, 3.5)))
    layers = rng.randint(1, 5)
    agree = round(rng.uniform(0.4, 0.95), 2)
    rank = 64 * rng.randint(1, 4)
    if kind == "step":
        return dict(kind=kind, **ctx, **heads, j=j, bq=bq, vocab=vocab, agree=agree)
    if kind == "select":
        return dict(kind=kind, b=b, j=j, bq=bq, hidden=hidden, vocab=vocab)
    if kind == "block":
        return dict(kind=kind, **ctx, **heads, j=j, bq=bq, hidden=hidden, inter=inter)
    if kind == "backbone":
        return dict(kind=kind, **ctx, **heads, j=j, bq=bq, hidden=hidden, inter=inter, layers=layers)
    vocab -= vocab % 8                                               # the head takes whole groups of eight entries
    if kind == "head":
        return dict(kind=kind, b=b, bq=bq, hidden=hidden, vocab=vocab, rank=rank, sampling=rng.random() < 0.4)
    if kind == "append":
        return dict(kind=kind, **ctx, j=j, hkv=hkv, d=d, feat=hidden, layers=layers)
    return dict(kind=kind, **ctx, **heads, j=j, bq=bq, hidden=hidden, inter=inter, layers=layers, vocab=vocab, rank=rank, agree=agree)


# ------------------------------------------------------------------------------------------------------------ inputs
def _lens(case):
    """The requests' context lengths: part of the case, not of the seed."""
    r = np.random.Generator(np.random.Philox(case["b"] * 1000003 + case["ctx_lo"] * 101 + case["ctx_hi"]))
    return [int(x) for x in r.integers(case["ctx_lo"], case["ctx_hi"] + 1, size=case["b"])]


def _offsets(lens):
    off = [0]
    for n in lens:
        off.append(off[-1] + n)
    return off


class _Draws:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)

    def bf16(self, sigma, *shape):
        return torch.randn(*shape, device=DEV, generator=self.g, dtype=torch.bfloat16).mul_(sigma)

    def f32(self, sigma, *shape):
        return torch.randn(*shape, device=DEV, generator=self.g).mul_(sigma)

    def gain(self, n):
        return (1.0 + 0.1 * torch.randn(n, device=DEV, generator=self.g)).to(torch.bfloat16)

    def ints(self, hi, *shape):
        return torch.randint(0, hi, shape, device=DEV, generator=self.g, dtype=torch.int32)

    def uniforms(self, *shape):
        """m * 2^-24, m an integer: what the library's draws take."""
        return torch.randint(0, 1 << 24, shape, device=DEV, generator=self.g).to(torch.float32).mul_(2.0 ** -24)


def _greedy_target(r, case):
    """Logits N(0, 2^2); a draft token is the target's own choice with probability `agree`, else any token."""
    b, j, v = case["b"], case["j"], case["vocab"]
    target = r.f32(2.0, b, j, v)
    top = target[:, : j - 1].argmax(-1).to(torch.int32)
    agree = torch.rand(b, j - 1, device=DEV, generator=r.g) < case["agree"]
    return target, torch.where(agree, top, r.ints(v, b, j - 1)).contiguous()


def _head_weights(r, case, rms=1.0):
    """LM head and the head's W, E, for hidden states of this root mean square.  A trained head has a clear favourite after most tokens: every token's row of E is
    planted in the row of W of one successor (a random permutation), with a margin that holds against the base logits."""
    v, h, k = case["vocab"], case["hidden"], case["rank"]
    w_lm = r.bf16(0.02 * math.sqrt(4096 / h) / rms, v, h)  # base logits of standard deviation 1.3
    e = torch.randn(v, k, device=DEV, generator=r.g)
    e /= e.norm(dim=1, keepdim=True)
    w = torch.randn(v, k, device=DEV, generator=r.g).mul_(0.5)
    w[torch.randperm(v, device=DEV, generator=r.g)] += 20.0 * e
    return w_lm, w.to(torch.bfloat16), e.to(torch.bfloat16)


def _layer_weights(r, case):
    h, i, d = case["hidden"], case["inter"], case["d"]
    qd, kd = case["hq"] * d, case["hkv"] * d
    return dict(w_qkv=r.bf16(0.02, qd + 2 * kd, h), w_o=r.bf16(0.02, h, qd), w_gate_up=r.bf16(0.02, 2 * i, h), w_down=r.bf16(0.02, h, i),
                rms1_w=r.gain(h), rms2_w=r.gain(h), qnorm_w=r.gain(d), knorm_w=r.gain(d))


def _attention(r, case):
    lens, kv, d = _lens(case), case["hkv"], case["d"]
    rows, b, j, bq = sum(lens), case["b"], case["j"], case["bq"]
    return dict(k_ctx=r.bf16(1.0, rows, kv, d), v_ctx=r.bf16(1.0, rows, kv, d), k_spine=r.bf16(1.0, b, j, kv, d), v_spine=r.bf16(1.0, b, j, kv, d))


def _shape(case):
    return dict(n_boundaries=case["j"], block=case["bq"], n_q_heads=case["hq"], n_kv_heads=case["hkv"], head_dim=case["d"])


def _backbone(r, case, slack):
    """Plan, weights and caches of the drafter's blocks; `slack`: spare rows per request behind the filled part."""
    lens, b, h = _lens(case), case["b"], case["hidden"]
    rows_req = case["j"] * case["bq"] + case["j"]
    off = _offsets([n + slack for n in lens])
    s = dict(x=r.bf16(1.0, b, rows_req, h), y=torch.zeros(b, rows_req, h, device=DEV), y16=torch.zeros(b, rows_req, h, device=DEV, dtype=torch.bfloat16))
    s["weights"] = [_layer_weights(r, case) for _ in range(case["layers"])]
    layers = [dp.make_layer_io(x=s["x"], **w, y_f32=s["y"], y_bf16=s["y16"]) for w in s["weights"]]
    s["kc"] = [r.bf16(1.0, off[-1], case["hkv"], case["d"]) for _ in layers]
    s["vc"] = [r.bf16(1.0, off[-1], case["hkv"], case["d"]) for _ in layers]
    s["off"], s["lens"] = off, lens
    s["plan"] = dp.BackbonePlan(ctx_offsets=off, **_shape(case), layers=layers, k_ctx=s["kc"], v_ctx=s["vc"], ctx_lens=lens if slack else None)
    return s


def _cache(r, case, feat, s):
    """Append plan on the caches s["kc"], s["vc"] laid out by s["off"]."""
    kd, n = case["hkv"] * case["d"], case["layers"]
    s["gain"], s["knorm"] = r.gain(feat), [r.gain(case["d"]) for _ in range(n)]
    s["w_kv"] = [r.bf16(0.02, 2 * kd, feat) for _ in range(n)]
    i64 = lambda v: torch.tensor(v, dtype=torch.int64, device=DEV)  # noqa: E731
    s["len0"], s["len"] = i64(s["lens"]), i64(s["lens"])
    s["append"] = dp.CachePlan(batch=case["b"], n_rows=case["j"], w_kv=s["w_kv"], k_ctx=s["kc"], v_ctx=s["vc"], row_start=i64(s["off"][:-1]),
                               capacity=i64([q - p for p, q in zip(s["off"], s["off"][1:])]), ctx_len=s["len"], norm_w=[s["gain"]] * n,
                               knorm_w=s["knorm"])
    s["features"] = r.bf16(1.0, case["b"], case["j"], feat)


def prepare(case, seed):
    r = _Draws(seed)
    kind, b = case["kind"], case["b"]
    if kind == "step":
        j, bq, d, kv = case["j"], case["bq"], case["d"], case["hkv"]
        s = _attention(r, case)
        s.update(q=r.bf16(1.0, b, j, bq, case["hq"], d), k_blk=r.bf16(1.0, b, j, bq, kv, d), v_blk=r.bf16(1.0, b, j, bq, kv, d))
        s["out"] = torch.zeros_like(s["q"])
        s["reps"] = s["out"].view(b, j, bq, case["hq"] * d)
        s["target"], s["tokens"] = _greedy_target(r, case)
        s["plan"] = dp.DraftPlan(ctx_offsets=_offsets(_lens(case)), **_shape(case))
        s["select"] = dp.VerifyPlan(batch=b, n_boundaries=j, vocab=case["vocab"], block=bq, hidden=case["hq"] * d, mode=0)
    elif kind == "select":
        j, v = case["j"], case["vocab"]
        zq = r.f32(3.0, b, j, v)
        p, q = torch.softmax(zq + r.f32(1.0, b, j, v), -1), torch.softmax(zq[:, : j - 1], -1).contiguous()
        # a draft token is drawn from the drafter's own row
        pick = torch.searchsorted(q.double().cumsum(-1), torch.rand(b, j - 1, 1, device=DEV, generator=r.g, dtype=torch.float64) * 0.999999)
        s = dict(target=p, draft=q, tokens=pick[..., 0].clamp_(max=v - 1).to(torch.int32).contiguous(), uniforms=r.uniforms(b, j),
                 reps=r.bf16(1.0, b, j, case["bq"], case["hidden"]))
        s["select"] = dp.VerifyPlan(batch=b, n_boundaries=j, vocab=v, block=case["bq"], hidden=case["hidden"], mode=1)
    elif kind == "block":
        h = case["hidden"]
        s = _attention(r, case)
        s.update(x=r.bf16(1.0, b, case["j"], case["bq"], h), weights=_layer_weights(r, case))
        s["y"], s["y16"] = torch.zeros(s["x"].shape, device=DEV), torch.zeros_like(s["x"])
        io = dp.make_layer_io(x=s["x"], **s["weights"], y_f32=s["y"], y_bf16=s["y16"])
        s["plan"] = dp.DraftPlan(ctx_offsets=_offsets(_lens(case)), **_shape(case), layer=io)
    elif kind == "backbone":
        s = _backbone(r, case, 0)
    elif kind == "head":
        s = dict(reps=r.bf16(1.0, b, case["bq"], case["hidden"]), bonus=r.ints(case["vocab"], b))
        s["w_lm"], s["w"], s["e"] = _head_weights(r, case)
        s["uniforms"] = r.uniforms(b, case["bq"]) if case["sampling"] else None
        s["head"] = dp.HeadPlan(b, case["bq"], case["hidden"], case["vocab"], case["rank"])
    elif kind == "append":
        s = dict(lens=_lens(case), accept=r.ints(case["j"], b))
        s["off"] = _offsets([n + 4 * case["j"] for n in s["lens"]])
        for c in ("kc", "vc"):
            s[c] = [torch.zeros(s["off"][-1], case["hkv"], case["d"], dtype=torch.bfloat16, device=DEV) for _ in range(case["layers"])]
        _cache(r, case, case["feat"], s)
    else:
        s = _backbone(r, case, 4 * case["j"])
        s["target"], s["tokens"] = _greedy_target(r, case)
        s["w_lm"], s["w"], s["e"] = _head_weights(r, case, rms=5.0)
        rows = case["j"] * case["bq"] + case["j"]
        s["select"] = dp.VerifyPlan(batch=b, n_boundaries=case["j"], vocab=case["vocab"], block=case["bq"], hidden=case["hidden"], mode=0, rep_req_rows=rows)
        s["head"] = dp.HeadPlan(b, case["bq"], case["hidden"], case["vocab"], case["rank"])
        _cache(r, case, case["hidden"], s)
    s["case"] = case
    return s


# ------------------------------------------------------------------------------------------------------------ one pass
def _selected(plan):
    return dict(accept_len=plan.accept_len, bonus=plan.bonus, gather_idx=plan.gather_idx, out_tokens=plan.out_tokens, selected=plan.selected,
                select_status=plan.status)


def _headed(plan):
    """Next tokens and the base logits where the call leaves them (step-major), without a copy."""
    n = plan.block * plan.b * plan.vocab * 4
    return dict(next_tokens=plan.next_tokens, base_logits=plan.workspace[:n].view(torch.float32), head_status=plan.status)


def run(s):
    kind = s["case"]["kind"]
    if kind == "step":
        s["plan"](q=s["q"], k_ctx=s["k_ctx"], v_ctx=s["v_ctx"], k_spine=s["k_spine"], v_spine=s["v_spine"], k_blk=s["k_blk"], v_blk=s["v_blk"], out=s["out"])
        s["select"](target=s["target"], draft_tokens=s["tokens"], reps=s["reps"])
        return dict(out=s["out"], status=s["plan"].status, **_selected(s["select"]))
    if kind == "select":
        s["select"](target=s["target"], draft_tokens=s["tokens"], reps=s["reps"], draft_probs=s["draft"], uniforms=s["uniforms"])
        return _selected(s["select"])
    if kind == "block":
        s["plan"](k_ctx=s["k_ctx"], v_ctx=s["v_ctx"], k_spine=s["k_spine"], v_spine=s["v_spine"])
        return dict(y=s["y"], y16=s["y16"], status=s["plan"].status)
    if kind == "backbone":
        s["plan"]()
        return dict(y=s["y"], y16=s["y16"], status=s["plan"].status)
    if kind == "head":
        s["head"].run(s["reps"], s["w_lm"], s["w"], s["e"], s["bonus"], s["uniforms"])
        return _headed(s["head"])
    # the lengths go back to where they were (a serving loop's caches grow; here a state is passed again and again)
    s["len"].copy_(s["len0"])
    if kind == "append":
        s["append"].run(s["features"], s["accept"])
        return dict(k=s["kc"], v=s["vc"], len=s["len"], status=s["append"].status)
    s["plan"]()
    s["select"](target=s["target"], draft_tokens=s["tokens"], reps=s["y16"])
    s["head"].run(s["select"].selected, s["w_lm"], s["w"], s["e"], s["select"].bonus)
    s["append"].run(s["features"], s["select"].accept_len)
    return dict(y=s["y"], status=s["plan"].status, **_selected(s["select"]), **_headed(s["head"]), k=s["kc"], v=s["vc"], len=s["len"],
                append_status=s["append"].status)


# ------------------------------------------------------------------------------------------------------------ what it takes
def _attention_work(case, spine_rows):
    """Bytes of context, spine and block keys and values; flops of the scores and of the weighted sums over visible keys."""
    lens, b, j, bq, d = _lens(case), case["b"], case["j"], case["bq"], case["d"]
    keys = 0
    for n in lens:
        keys += sum(bq * (n + i + 1 + bq) for i in range(j))
        keys += sum(n + i + 1 for i in range(j)) if spine_rows else 0
    return 2 * case["hkv"] * d * 2 * sum(lens), 4.0 * d * case["hq"] * keys


def _block_work(case, spine_rows, layers):
    h, i, d = case["hidden"], case["inter"], case["d"]
    qd, kd = case["hq"] * d, case["hkv"] * d
    m = case["b"] * (case["j"] * case["bq"] + (case["j"] if spine_rows else 0))
    weights = h * (qd + 2 * kd) + qd * h + 3 * h * i
    kv, fl = _attention_work(case, spine_rows)
    by = layers * (2 * weights + kv) + m * h * 8
    if not spine_rows:
        by += 2 * case["b"] * case["j"] * kd * 2
    return by, layers * (fl + 2.0 * m * weights)


def _rows_needed(case):
    """Mean number of a request's target rows that decide it: row 0, and row i while the i drafts before it agree."""
    return sum(case["agree"] ** i for i in range(case["j"]))


def _greedy_bytes(case, hidden):
    return case["b"] * (_rows_needed(case) * case["vocab"] * 4 + 2 * case["bq"] * hidden * 2)


def _head_work(case):
    m, v = case["b"] * case["bq"], case["vocab"]
    return 2 * v * (case["hidden"] + case["rank"]) + m * (2 * case["hidden"] + 2 * case["rank"] + 4 * v), 2.0 * m * v * (case["hidden"] + case["rank"])


def _append_work(case, feat):
    m, n = case["b"] * case["j"], 2 * case["hkv"] * case["d"]
    return case["layers"] * 2 * n * feat + 2 * m * feat + case["layers"] * m * n, 2.0 * case["layers"] * m * n * feat


def work(case):
    kind = case["kind"]
    if kind == "step":
        kv, fl = _attention_work(case, False)
        b, j, bq, d = case["b"], case["j"], case["bq"], case["d"]
        by = kv + 2 * b * j * bq * case["hq"] * d * 2 + 2 * b * (j * bq + j) * case["hkv"] * d * 2 + _greedy_bytes(case, case["hq"] * d)
    elif kind == "select":
        by, fl = case["b"] * (2 * case["vocab"] * 4 + 2 * case["bq"] * case["hidden"] * 2), 0.0
    elif kind == "block":
        by, fl = _block_work(case, False, 1)
    elif kind == "backbone":
        by, fl = _block_work(case, True, case["layers"])
    elif kind == "head":
        by, fl = _head_work(case)
    elif kind == "append":
        by, fl = _append_work(case, case["feat"])
    else:
        parts = [_block_work(case, True, case["layers"]), (_greedy_bytes(case, case["hidden"]), 0.0), _head_work(case), _append_work(case, case["hidden"])]
        by, fl = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    """About four times what the paths differ by from themselves in 64 bits (with the same bf16 roundings between a block's
    parts): attention 0.0023, largest 0.016; blocks 0.004 after two layers, 0.008 after five, largest 0.04; base logits
    6e-6, largest 2e-5.  Tokens are whole numbers: the same."""
    return {"step": {"rel": 1e-2, "max": 0.08}, "select": "exact", "block": {"rel": 1e-2, "max": 0.1}, "backbone": {"rel": 2e-2, "max": 0.16},
            "head": {"rel": 2.5e-5, "max": 1e-4}, "append": {"rel": 1e-2, "max": 0.05}, "round": {"rel": 2e-2, "max": 0.16}}[case["kind"]]


# ------------------------------------------------------------------------------------------------------------ the results in 64 bits
def _norm64(x, gain):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-6) * gain.double()


def _rope64(x, pos):
    """Rotate-half embedding of x [rows][heads][d]."""
    half = x.shape[-1] // 2
    ang = pos.double()[:, None, None] * 1e6 ** (-torch.arange(half, device=DEV, dtype=torch.float64) / half)
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat([lo * ang.cos() - hi * ang.sin(), hi * ang.cos() + lo * ang.sin()], -1)


def _attend64(q, k, v, seen):
    """q [rows][hq][d] on k, v [keys][hkv][d] under the mask seen [rows][keys]."""
    rows, hq, d = q.shape
    hkv, out = k.shape[1], torch.empty_like(q)
    for g in range(hkv):
        h = slice(g * hq // hkv, (g + 1) * hq // hkv)
        z = torch.einsum("rhd,kd->hrk", q[:, h], k[:, g]).mul_(d ** -0.5).masked_fill_(~seen, -math.inf)
        out[:, h] = torch.einsum("hrk,kd->rhd", torch.softmax(z, -1), v[:, g])
    return out


def _visible(case, n, spine_rows):
    """Rows: slots of every boundary, then the spine's; keys: n of context, the spine, every boundary's block."""
    j, bq = case["j"], case["bq"]
    branch = torch.arange(j, device=DEV).repeat_interleave(bq)
    row = torch.cat([branch, torch.arange(j, device=DEV)]) if spine_rows else branch
    spine = torch.arange(j, device=DEV)[None] <= row[:, None]
    own = branch[None] == branch[:, None]
    if spine_rows:
        own = torch.cat([own, own.new_zeros(j, j * bq)])
    return torch.cat([spine.new_ones(len(row), n), spine, own], 1)


def _block64(case, w, x, ctx, spine):
    """One block over the rows of every request, x [b][rows][hidden]; ctx(n): request n's cached keys and values; spine: keys and values, or
    None where the rows behind the slots make them."""
    b, rows, _ = x.shape
    hq, hkv, d, m, lens = case["hq"], case["hkv"], case["d"], case["j"] * case["bq"], _lens(case)
    qkv = _norm64(x, w["rms1_w"]) @ w["w_qkv"].double().T
    q, k, v = (t.reshape(b, rows, -1, d) for t in qkv.split([hq * d, hkv * d, hkv * d], -1))
    i = torch.arange(m, device=DEV)
    pos = torch.cat([i // case["bq"] + 2 + i % case["bq"], torch.arange(rows - m, device=DEV)])
    a = torch.empty(b, rows, hq * d, device=DEV, dtype=torch.float64)
    for n in range(b):
        qn, kn = _rope64(_norm64(q[n], w["qnorm_w"]), lens[n] + pos), _rope64(_norm64(k[n], w["knorm_w"]), lens[n] + pos)
        kc, vc = ctx(n)
        ks, vs = (spine[0][n].double(), spine[1][n].double()) if spine else (kn[m:], v[n, m:])
        a[n] = _attend64(qn, torch.cat([kc.double(), ks, kn[:m]]), torch.cat([vc.double(), vs, v[n, :m]]), _visible(case, lens[n], not spine)).view(rows, -1)
    h = x + a @ w["w_o"].double().T
    gate, up = (_norm64(h, w["rms2_w"]) @ w["w_gate_up"].double().T).chunk(2, -1)
    return h + (torch.nn.functional.silu(gate) * up) @ w["w_down"].double().T


def _backbone64(case, s):
    y = s["x"].double()
    for w, kc, vc in zip(s["weights"], s["kc"], s["vc"]):
        y = _block64(case, w, y, lambda n: [c[s["off"][n]: s["off"][n] + s["lens"][n]] for c in (kc, vc)], None)
    return y


def _logits64(reps, w_lm):
    """[b][bq][hidden] on the LM head, step-major."""
    z = [reps.transpose(0, 1).reshape(-1, reps.shape[-1]).double() @ w.double().T for w in w_lm.split(16384)]
    return torch.cat(z, 1).flatten()


def _append64(case, s, accept):
    ks, vs = [c.double() for c in s["kc"]], [c.double() for c in s["vc"]]
    for k, v, w, gk in zip(ks, vs, s["w_kv"], s["knorm"]):
        kv = _norm64(s["features"].double(), s["gain"]) @ w.double().T
        new_k, new_v = (t.reshape(case["b"], case["j"], case["hkv"], case["d"]) for t in kv.chunk(2, -1))
        for n, r in enumerate(accept):
            first = s["off"][n] + s["lens"][n]
            pos = s["lens"][n] + torch.arange(r + 1, device=DEV)
            k[first: first + r + 1] = _rope64(_norm64(new_k[n, : r + 1], gk), pos)
            v[first: first + r + 1] = new_v[n, : r + 1]
    return ks, vs


def exact(case, seed):
    """What `run` returns in 64 bits throughout, with none of the bf16 roundings in between.  None for whole numbers: they are
    compared as they are."""
    kind, s = case["kind"], prepare(case, seed)
    if kind == "select":
        return None
    if kind == "head":
        return dict(next_tokens=None, base_logits=_logits64(s["reps"], s["w_lm"]), head_status=None)
    if kind == "append":
        k, v = _append64(case, s, s["accept"].tolist())
        return dict(k=k, v=v, len=None, status=None)
    off = _offsets(_lens(case)) if kind in ("step", "block") else s["off"]
    selected = dict(accept_len=None, bonus=None, gather_idx=None, out_tokens=None, selected=None, select_status=None)
    accept = None
    if kind in ("step", "round"):
        agree = s["tokens"] == s["target"][:, : case["j"] - 1].argmax(-1)
        accept = agree.long().cumprod(1).sum(1).tolist()
    if kind == "step":
        b, j, bq = case["b"], case["j"], case["bq"]
        out = torch.empty(s["q"].shape, device=DEV, dtype=torch.float64)
        for n in range(b):
            kn, vn = (torch.cat([s[c + "_ctx"][off[n]: off[n + 1]], s[c + "_spine"][n], s[c + "_blk"][n].flatten(0, 1)]).double() for c in "kv")
            out[n] = _attend64(s["q"][n].flatten(0, 1).double(), kn, vn, _visible(case, off[n + 1] - off[n], False)).view(out[n].shape)
        selected["selected"] = torch.stack([out[n, r] for n, r in enumerate(accept)]).flatten(2)
        return dict(out=out, status=None, **selected)
    if kind == "block":
        x = s["x"].flatten(1, 2).double()
        y = _block64(case, s["weights"], x, lambda n: [s[c][off[n]: off[n + 1]] for c in ("k_ctx", "v_ctx")], (s["k_spine"], s["v_spine"])).view(s["x"].shape)
        return dict(y=y, y16=y, status=None)
    y = _backbone64(case, s)
    if kind == "backbone":
        return dict(y=y, y16=y, status=None)
    bq = case["bq"]
    selected["selected"] = torch.stack([y[n, r * bq: (r + 1) * bq] for n, r in enumerate(accept)])
    k, v = _append64(case, s, accept)
    return dict(y=y, status=None, **selected, next_tokens=None, base_logits=_logits64(selected["selected"], s["w_lm"]), head_status=None, k=k, v=v, len=None,
                append_status=None)
