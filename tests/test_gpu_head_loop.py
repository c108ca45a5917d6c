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
