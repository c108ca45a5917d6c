"""The head loop where the number of its CTAs changes: one and two CTAs, the sizes around which a CTA gets one, two or three tiles, and the batch whose base logits
make the tiles shorter (120 rows).  Step by step against the oracle under the rules of tests/test_gpu_head.py."""
import pytest

import workloads as W
from test_gpu_head import _check, _check_sampling, _run
from test_gpu_head_loop import _sample, _uniforms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,rank,batch", [(128, 256, 3), (136, 64, 1), (84 * 128, 192, 2), (86 * 128 + 8, 256, 17), (252 * 128, 128, 4), (254 * 128 + 8, 64, 2), (80000, 256, 16), (151936, 256, 16)])
def test_tiles_per_cta(vocab, rank, batch):
    shape = W.HeadShape(batch, 2, 64, vocab, rank)
    inp = W.make_head_inputs(shape, vocab + rank)
    toks, logits = _run(inp)
    assert _check(inp, toks, logits) >= 0.9 * batch * shape.block
    if batch <= 4:
        u = _uniforms(shape, batch)
        toks, logits = _sample(inp, u)
        assert _check_sampling(inp, toks, logits, u) >= 0.8 * batch * shape.block
