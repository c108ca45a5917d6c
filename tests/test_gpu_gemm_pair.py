"""The CTA-pair GEMM at the edges of its activation tiles (any multiple of 16 rows up to 256): a row more than a tile, a last
tile that is part filled, widths that are no multiple of a weight tile, several rounds of tiles.  Tolerances as for the
products of few rows: fp32 sums of K <= 768 exact products are a few 1e-6 off in any order, 1e-4 is asked for; bf16 results
half a bf16 step and what that moves across one."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import attention as OA
from oracle import layer as OL

pytestmark = pytest.mark.gpu


def _bits(rng, shape, sigma):
    return W.f32_to_bf16_bits((rng.standard_normal(shape) * sigma).astype(np.float32))


def _dev(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).cuda().view(torch.bfloat16)


@pytest.mark.parametrize("M,N,K", [(513, 264, 64), (576, 1000, 192), (700, 2048, 128), (769, 520, 768), (1152, 5128, 128), (2049, 776, 64), (257, 20488, 64)])
def test_store_and_residual(M, N, K):
    import paper_2609_27396_b200 as dp
    rng = np.random.default_rng(M * 5 + N + K)
    a, w = _bits(rng, (M, K), 1.0), _bits(rng, (N, K), 0.05)
    r32 = rng.standard_normal((M, N)).astype(np.float32)
    ref = OL.linear(OA.bf16_bits_to_f64(a), OA.bf16_bits_to_f64(w))
    ad, wd = _dev(a), _dev(w)
    out, st = dp.gemm_bf16(ad, wd, epilogue=0)
    f32, st3 = dp.gemm_bf16(ad, wd, epilogue=3)
    res, res16, st1 = dp.gemm_bf16(ad, wd, epilogue=1, resid=torch.from_numpy(r32).cuda(), want_bf16_copy=True)
    torch.cuda.synchronize()
    assert int(st.item()) == int(st1.item()) == int(st3.item()) == 0
    assert np.abs(f32.cpu().numpy().astype(np.float64) - ref).max() < 1e-4
    assert np.abs(res.cpu().numpy().astype(np.float64) - (r32.astype(np.float64) + ref)).max() < 1e-4
    assert np.all(np.abs(out.float().cpu().numpy().astype(np.float64) - ref) <= 2 ** -8 * np.abs(ref) + 1e-4)
    assert torch.equal(res16, res.to(torch.bfloat16))


@pytest.mark.parametrize("M,I,K", [(513, 136, 64), (576, 1032, 192), (1100, 3080, 128), (288, 20008, 64)])
def test_swiglu(M, I, K):
    import paper_2609_27396_b200 as dp
    rng = np.random.default_rng(M + I + K)
    a, w = _bits(rng, (M, K), 1.0), _bits(rng, (2 * I, K), 0.08)
    out, st = dp.gemm_bf16(_dev(a), _dev(w), epilogue=2)
    torch.cuda.synchronize()
    ref = OL.swiglu_linear(OA.bf16_bits_to_f64(a), OA.bf16_bits_to_f64(w))
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 2 ** -7 * np.abs(ref) + 1e-3), float(np.abs(got - ref).max())
    assert int(st.item()) == 0


# activation rows, columns, K, epilogue, tiles left in the last round, activation rows of the units that each of those is cut into
@pytest.mark.parametrize("M,N,K,epi,left,rows", [
    (1152, 15760, 320, 3, 14, 80),      # three units of 80 rows for 240
    (980, 18952, 320, 0, 4, 32),        # eight of 32 for 256; the last tile has 212 rows, its last unit none
    (980, 18952, 320, 1, 4, 32),
    (600, 10440, 320, 2, 24, 112),      # two of 112 for 208
    (1152, 7856, 320, 2, 14, 80),
])
def test_last_round_of_few_tiles(M, N, K, epi, left, rows):
    """The tiles of a nearly empty last round are cut along their activation rows."""
    import paper_2609_27396_b200 as dp
    nt = dp.gemm_route(M, N, K, epilogue=epi)["tile_rows"]
    units = -(-M // nt) * -(-N // (128 if epi == 2 else 256))
    assert units > 74 and units % 74 == left and rows == max(32, (nt // (48 // left) + 15) // 16 * 16)
    rng = np.random.default_rng(M + N + K + epi)
    a, w = _bits(rng, (M, K), 1.0), _bits(rng, (2 * N if epi == 2 else N, K), 0.08)
    x, y = OA.bf16_bits_to_f64(a), OA.bf16_bits_to_f64(w)
    r32 = rng.standard_normal((M, N)).astype(np.float32) if epi == 1 else None
    got, st = dp.gemm_bf16(_dev(a), _dev(w), epilogue=epi, resid=torch.from_numpy(r32).cuda() if epi == 1 else None)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    got = got.float().cpu().numpy().astype(np.float64)
    ref = OL.swiglu_linear(x, y) if epi == 2 else OL.linear(x, y) + (r32 if epi == 1 else 0)
    assert np.all(np.abs(got - ref) <= {0: 2 ** -8, 1: 0, 2: 2 ** -7, 3: 0}[epi] * np.abs(ref) + (1e-3 if epi == 2 else 1e-4))
