"""The head loop at the edges of its vocabulary tiles: their height is chosen to fill the SMs (32 .. 128 rows), so the sizes around
one tile, one tile per SM at either height, and a second round are where it can go wrong.  Compared step by step with the oracle under
the same near-tie rule as the other head tests (tests/test_gpu_head.py)."""
import pytest

import workloads as W
from test_gpu_head import _check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,rank", [(8, 64), (40, 128), (148 * 32, 192), (148 * 32 + 8, 256), (148 * 128, 64), (148 * 128 + 8, 128), (148 * 192 - 8, 256)])
def test_tile_heights(vocab, rank):
    inp = W.make_head_inputs(W.HeadShape(3, 3, 64, vocab, rank), vocab + rank)
    toks, logits = _run(inp)
    assert _check(inp, toks, logits) >= 8
