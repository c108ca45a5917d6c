"""The GEMM for few activation rows (weights as the rows of the product, K split inside clusters) against plain float64
products, at the edges of its tiles: one row, a row more than a multiple of 16, the last size of every accumulator width,
outputs that leave a part-filled last tile, K shorter than a stage, an odd number of 64-column slabs, several rounds of tiles.

Tolerances.  fp32 results: the products are exact, their sum over K in fp32 is off by at most K 2^-24 sum |a||w| in any order;
with |a| ~ 1, |w| ~ 0.05 that is below 0.05 K^2 2^-24 < 2e-3 at K = 768 and in practice a few 1e-6: 1e-4 is asked for.
bf16 results: half a bf16 step, 2^-9 |ref|, and what 1e-4 of the sum's error moves across a step."""
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


SHAPES = [(1, 8, 64), (8, 264, 192), (16, 1000, 64), (17, 4104, 320), (72, 2048, 768), (80, 520, 448), (128, 1032, 256), (128, 40000, 128),
          (129, 776, 384), (200, 4096, 512), (256, 512, 192), (257, 520, 320), (288, 1024, 768), (400, 264, 640), (512, 136, 256)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_store_and_residual(M, N, K):
    import paper_2609_27396_b200 as dp
    rng = np.random.default_rng(M * 7 + N + K)
    a, w = _bits(rng, (M, K), 1.0), _bits(rng, (N, K), 0.05)
    rb = _bits(rng, (M, N), 1.0)
    ref = OL.linear(OA.bf16_bits_to_f64(a), OA.bf16_bits_to_f64(w))
    ad, wd = _dev(a), _dev(w)
    out, st = dp.gemm_bf16(ad, wd, epilogue=0)
    f32, st3 = dp.gemm_bf16(ad, wd, epilogue=3)
    res, res16, st1 = dp.gemm_bf16(ad, wd, epilogue=1, resid=_dev(rb), want_bf16_copy=True)
    torch.cuda.synchronize()
    assert int(st.item()) == int(st1.item()) == int(st3.item()) == 0
    sum_ref = OA.bf16_bits_to_f64(rb) + ref
    assert np.abs(f32.cpu().numpy().astype(np.float64) - ref).max() < 1e-4
    assert np.abs(res.cpu().numpy().astype(np.float64) - sum_ref).max() < 1e-4
    assert np.all(np.abs(out.float().cpu().numpy().astype(np.float64) - ref) <= 2 ** -8 * np.abs(ref) + 1e-4)
    assert torch.equal(res16, res.to(torch.bfloat16))


@pytest.mark.parametrize("M,I,K", [(1, 8, 64), (8, 136, 192), (72, 3080, 256), (128, 24000, 128), (200, 1032, 320), (256, 520, 192)])
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


def test_same_sum_every_time():
    import paper_2609_27396_b200 as dp
    rng = np.random.default_rng(3)
    a, w = _dev(_bits(rng, (72, 4096), 1.0)), _dev(_bits(rng, (4096, 4096), 0.05))
    first, _ = dp.gemm_bf16(a, w, epilogue=3)
    for _ in range(5):
        assert torch.equal(first, dp.gemm_bf16(a, w, epilogue=3)[0])


def test_parts_of_k_only_in_one_round():
    """A host query over the range: where the tiles take several rounds no CTAs share one (the parts' meeting would not be hidden)."""
    import paper_2609_27396_b200 as dp
    shared = 0
    for M in (1, 8, 24, 40, 72, 100, 112, 128, 160, 288, 400):
        for N in (256, 1024, 4096, 5120, 6144, 10240, 11776, 20480, 50000):
            for K in (512, 4096, 5120, 8192, 17408):
                for epilogue in (0, 2):
                    r = dp.gemm_route(M, N, K, epilogue=epilogue)
                    if r["few_rows"]:
                        assert r["ctas"] == 1 or r["rounds"] == 1, (M, N, K, epilogue, r)
                        assert M <= 128 or r["rounds"] == 1, (M, N, K, epilogue, r)
                        shared += r["ctas"] > 1
    assert shared > 100
