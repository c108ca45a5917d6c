"""The head loop where its tiles split between tensor memory, the ring and the rest, where the sampling logits do or do not fit in shared
memory, and with logits that are infinite, NaN or the type's lowest value.  Step by step against the oracle under the rules of
tests/test_gpu_head.py."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import dev_bf16
from oracle import head as H
from test_gpu_head import _check, _check_sampling, _run

import paper_2609_27396_b200 as dp

pytestmark = pytest.mark.gpu
SMS = 148


def _uniforms(shape, seed):
    return (np.random.default_rng(seed).integers(0, 1 << 24, size=(shape.batch, shape.block)) * 2.0 ** -24).astype(np.float32)


def _sample(inp, uniforms):
    t = [dev_bf16(x) for x in (inp.sel_reps, inp.w_lm, inp.ar_w, inp.ar_e)]
    toks, plan = dp.draft_head(t[0], t[1], t[2], t[3], torch.from_numpy(inp.bonus).cuda(), uniforms=torch.from_numpy(uniforms).cuda())
    torch.cuda.synchronize()
    assert plan.status.item() == 0
    return toks.cpu().numpy(), plan.base_logits().cpu().numpy().astype(np.float64)


# tiles per CTA: 3 = all in tensor memory at rank 256, 4 and 7 = one and four through the ring, 13 = one through the ring at rank 64; batch 17: N = 32
@pytest.mark.parametrize("tiles,rank,batch", [(3, 256, 2), (4, 256, 17), (7, 256, 16), (5, 192, 1), (13, 64, 3)])
def test_tiles_that_stay(tiles, rank, batch):
    shape = W.HeadShape(batch, 3, 64, SMS * 128 * tiles - 40, rank)
    inp = W.make_head_inputs(shape, 7 * tiles + rank)
    toks, logits = _run(inp)
    assert _check(inp, toks, logits) >= 0.97 * batch * shape.block
    if batch <= 3:
        u = _uniforms(shape, tiles)
        toks, logits = _sample(inp, u)
        assert _check_sampling(inp, toks, logits, u) >= 0.9 * batch * shape.block


# 32 requests of the full vocabulary, and 17 tiles per CTA: a step's logits have no room in shared memory; block 1: nothing stays
@pytest.mark.parametrize("shape", [W.HeadShape(32, 2, 64, 151936, 256), W.HeadShape(1, 2, 64, SMS * 128 * 17 - 8, 64), W.HeadShape(2, 1, 64, 20008, 128)])
def test_sampling_with_logits_elsewhere(shape):
    inp = W.make_head_inputs(shape, 3)
    u = _uniforms(shape, 9)
    toks, logits = _sample(inp, u)
    assert _check_sampling(inp, toks, logits, u) >= 0.9 * shape.batch * shape.block


LOW = float(torch.finfo(torch.bfloat16).min)


@pytest.mark.parametrize("fill,special", [
    (LOW, {}),                                                  # every entry the type's lowest: all weigh the same
    (LOW, {700: -1.5, 5000: 0.25}),                             # a mask
    (-np.inf, {3: -80.0, 6001: -81.0}),
    (np.nan, {}),                                               # no number: token 0
    (np.nan, {4097: -7.0, 8000: -7.0}),
    (0.0, {17: np.inf}),                                        # an infinite logit: token 0
    (0.0, {4100: 3e9, 7000: 3e9}),                              # far above the rest: one of the two
    (-3e9, {}),
    (-200.0, {8191: 90.0}),
])
def test_sampling_of_unusual_logits(fill, special):
    vocab, block = 8192, 4
    base = np.full(vocab, fill, np.float32)
    for k, v in special.items():
        base[k] = v
    base = torch.from_numpy(base).to(torch.bfloat16)
    w_lm = torch.zeros(vocab, 64, dtype=torch.bfloat16)
    w_lm[:, 0] = base
    reps = torch.zeros(2, block, 64, dtype=torch.bfloat16)
    reps[:, :, 0] = 1.0                                          # logits are the first column, whatever the token
    zero = torch.zeros(vocab, 64, dtype=torch.bfloat16, device="cuda")
    u = np.array([[0.0, 0.3, 0.75, 1 - 2.0 ** -24], [0.5, 0.11, 0.9, 0.49999]], np.float32)
    toks, plan = dp.draft_head(reps.cuda(), w_lm.cuda(), zero, zero, torch.zeros(2, dtype=torch.int32, device="cuda"), uniforms=torch.from_numpy(u).cuda())
    torch.cuda.synchronize()
    assert plan.status.item() == 0
    z = base.double().numpy()
    for n in range(2):
        for i in range(block):
            want, got = H.sample_from_logits(z, float(u[n, i])), int(toks[n, i])
            if got != want:                                      # (only where the threshold is at the edge of two entries)
                w = np.where(np.isnan(z), 0.0, np.exp(z - np.nanmax(z)))
                c = np.cumsum(w) / w.sum()
                assert w[got] > 0 and c[got] - w[got] / w.sum() - 1e-6 <= u[n, i] <= c[got] + 1e-6, (n, i, got, want)


def _sample_row(row, u):
    """The tokens and the status of a call whose logits are `row` (bf16) in every step of both requests, with the uniforms u [2][block]."""
    vocab, block = len(row), u.shape[1]
    w_lm = torch.zeros(vocab, 64, dtype=torch.bfloat16)
    w_lm[:, 0] = row
    reps = torch.zeros(2, block, 64, dtype=torch.bfloat16)
    reps[:, :, 0] = 1.0
    zero = torch.zeros(vocab, 64, dtype=torch.bfloat16, device="cuda")
    toks, plan = dp.draft_head(reps.cuda(), w_lm.cuda(), zero, zero, torch.zeros(2, dtype=torch.int32, device="cuda"), uniforms=torch.from_numpy(u).cuda())
    torch.cuda.synchronize()
    return toks.cpu().numpy(), plan.status.item()


# Neighbouring values of these sizes are 65536 and more apart, 32768 at the smallest: an entry weighs 1 or nothing, and the tokens are the oracle's
@pytest.mark.parametrize("block", [1, 4])
@pytest.mark.parametrize("at", ["one", "two", "all"])
@pytest.mark.parametrize("top", [1e7, -1e7, 1e8, -1e8, 188743680.0, -754974720.0, 1551892480.0, -1585446912.0, 1.5e9, -1.5e9, 2.0 ** 31, -3e38, 3e38])
def test_sampling_of_large_logits(top, at, block):
    row = torch.full((8192,), top, dtype=torch.bfloat16)
    if at != "all":
        keep = [4099] if at == "one" else [130, 8190]
        below = row[0].view(torch.int16) + (-1 if top > 0 else 1)          # the next bf16 towards -inf
        row[[v for v in range(8192) if v not in keep]] = below.view(torch.bfloat16)
    u = np.array([[0.0, 0.3, 0.75, 1 - 2.0 ** -24], [0.5, 0.11, 0.9, 0.49999]], np.float32)[:, :block]
    toks, status = _sample_row(row, u)
    assert status == 0
    z = row.double().numpy()
    assert toks.tolist() == [[H.sample_from_logits(z, float(x)) for x in r] for r in u]


@pytest.mark.parametrize("row", [
    {0: -200.0, 8191: 90.0},                       # the lightest entry is e^-290 of the row
    {0: -600.0, 1: -480.0, 2: -350.0, 3: 0.0},     # ... and its neighbours in the same CTA's range are not much heavier
    {40: -104.0, 41: 0.0},                         # below the smallest fp32
    {5000: -87.0, 5001: -86.5, 5002: 0.0},
])
def test_sampling_of_light_entries(row):
    """At u = 0 the lowest entry with any weight in double precision, however light; one step of the uniform further the heavy one."""
    full = torch.full((8192,), -float("inf"), dtype=torch.bfloat16)
    for v, z in row.items():
        full[v] = z
    toks, status = _sample_row(full, np.array([[0.0, 2.0 ** -24], [2.0 ** -24, 0.0]], np.float32))
    assert status == 0
    low, heavy = min(row), max(row, key=row.get)
    assert toks.tolist() == [[low, heavy], [heavy, low]]


def _inputs_of_a_call(seed, vocab, rank=256):
    inp = W.make_head_inputs(W.HeadShape(3, 6, 64, vocab, rank), seed)
    t = [dev_bf16(x) for x in (inp.sel_reps, inp.w_lm, inp.ar_w, inp.ar_e)] + [torch.from_numpy(inp.bonus).cuda()]
    return t, torch.from_numpy(_uniforms(inp.shape, seed)).cuda(), dp.HeadPlan(3, 6, 64, vocab, rank)


@pytest.mark.parametrize("rank,modes", [(256, "sg"), (64, "sg"), (64, "g"), (128, "g")])
def test_calls_on_two_streams(rank, modes):
    """Calls on two streams with no order between them: each loop needs all its CTAs and their tensor memory at once, and both get that."""
    calls = [_inputs_of_a_call(5, 60000, rank), _inputs_of_a_call(6, 40000, rank)]
    calls = [(t, [u if m == "s" else None for m in modes], plan) for t, u, plan in calls]
    want = [[plan.run(*t, uniforms=x).clone() for x in us] for t, us, plan in calls]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    got = [[], []]
    for _ in range(12):
        for i, (t, us, plan) in enumerate(calls):
            with torch.cuda.stream(streams[i]):
                got[i].append([plan.run(*t, uniforms=x).clone() for x in us])
    torch.cuda.synchronize()
    for i, (_, _, plan) in enumerate(calls):
        assert plan.status.item() == 0
        for g in got[i]:
            assert all(torch.equal(x, y) for x, y in zip(g, want[i])), i


@pytest.mark.parametrize("sampling", [False, True])
def test_head_captured_in_a_graph(sampling):
    t, u, plan = _inputs_of_a_call(9, 30000)
    u = u if sampling else None
    first = plan.run(*t, uniforms=u).clone()
    t[4].bitwise_xor_(1)
    if sampling:
        u.mul_(0.5)
    second = plan.run(*t, uniforms=u).clone()
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        plan.run(*t, uniforms=u, stream=s)
    for _ in range(3):
        plan.next_tokens.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(plan.next_tokens, second)
    t[4].bitwise_xor_(1)                             # new inputs in the captured buffers
    if sampling:
        u.mul_(2.0)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(plan.next_tokens, first) and plan.status.item() == 0
