"""The GEMM for few activation rows (weights as the rows of the product, K split inside clusters) against plain float64
products, at the edges of its tiles: one row, a row more than a multiple of 16, the last size of every accumulator width,
outputs that leave a part-filled last tile, K shorter than a stage, an odd number of 64-column slabs, several rounds of tiles.
SHAPES have a short K: one CTA per tile there, and above 128 rows the CTA pairs take them.  SPLIT and the shapes below it say by a host
query which form they run: parts of K that meet inside a cluster, accumulators of two instructions (above 256 rows), several rounds.

Tolerances.  fp32 results: the products are exact, their sum over K in fp32 is off by at most K 2^-24 sum |a||w| in any order;
with |a| ~ 1, |w| ~ 0.05 that is below 0.05 K^2 2^-24 < 2e-3 at K = 768 and in practice a few 1e-6: 1e-4 is asked for.  Longer K (_off):
K / 16 additions, each off by at most one step 2^-23 of the running sum, which stays under six standard deviations 0.05 sqrt(K).
bf16 results: half a bf16 step, 2^-9 |ref|, and what the sum's error moves across a step."""
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


def _off(K):
    return max(1e-4, K / 16 * 2.0 ** -23 * 6 * 0.05 * K ** 0.5)


def _draw(seed, M, rows, K):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16), (0.05 * torch.randn(rows, K, device="cuda", generator=g)).to(torch.bfloat16),
            torch.randn(M, rows, device="cuda", generator=g).to(torch.bfloat16))


def _stores(M, N, K):
    """Every store of the kernel against float64."""
    import paper_2609_27396_b200 as dp
    a, w, resid = _draw(M * 7 + N + K, M, N, K)
    ref = a.double() @ w.double().T
    out, st = dp.gemm_bf16(a, w, epilogue=0)
    f32, st3 = dp.gemm_bf16(a, w, epilogue=3)
    res, res16, st1 = dp.gemm_bf16(a, w, epilogue=1, resid=resid, want_bf16_copy=True)
    assert int(st.item()) == int(st1.item()) == int(st3.item()) == 0
    assert float((f32.double() - ref).abs().max()) < _off(K)
    assert float((res.double() - (resid.double() + ref)).abs().max()) < _off(K) + 2 ** -22 * float(ref.abs().max())
    assert bool(((out.double() - ref).abs() <= 2 ** -8 * ref.abs() + _off(K)).all())
    assert torch.equal(res16, res.to(torch.bfloat16))
    for _ in range(3):   # the parts are added in one order
        assert torch.equal(f32, dp.gemm_bf16(a, w, epilogue=3)[0])


def _swiglu(M, I, K):
    import paper_2609_27396_b200 as dp
    a, w, _ = _draw(M + I + K, M, 2 * I, K)
    out, st = dp.gemm_bf16(a, w, epilogue=2)
    gate, up = (a.double() @ w.double().T).chunk(2, 1)
    ref = torch.nn.functional.silu(gate) * up
    # d silu / d gate is at most 1.1, so either factor's error comes in times the other; exp and division add a few 2^-22
    most = max(float(gate.abs().max()), float(up.abs().max()))
    assert bool(((out.double() - ref).abs() <= 2 ** -8 * ref.abs() + 2.2 * most * _off(K) + 1e-5).all())
    assert int(st.item()) == 0


SPLIT = [(1, 256, 2048), (17, 1032, 2112), (40, 1024, 4096), (72, 4096, 4096), (88, 5120, 17408), (128, 2048, 4096), (129, 520, 4096), (200, 2048, 4096),
         (240, 520, 8192), (264, 512, 4096), (288, 1024, 4096), (400, 2056, 8192)]


@pytest.mark.parametrize("M,N,K", SPLIT)
def test_parts_of_k_meet(M, N, K):
    import paper_2609_27396_b200 as dp
    for epilogue in (0, 1, 3):
        r = dp.gemm_route(M, N, K, epilogue=epilogue)
        assert r["few_rows"] and r["ctas"] > 1 and r["rounds"] == 1 and r["tile_rows"] == ((M + 15) // 16 * 16 if M <= 256 else (M + 31) // 32 * 32), r
    _stores(M, N, K)


@pytest.mark.parametrize("M,I,K", [(1, 512, 4096), (17, 1024, 4096), (40, 1032, 2112), (72, 2048, 4096), (128, 4096, 4096), (136, 1024, 4096), (200, 520, 8192)])
def test_parts_of_k_meet_swiglu(M, I, K):
    import paper_2609_27396_b200 as dp
    r = dp.gemm_route(M, I, K, epilogue=2)
    assert r["few_rows"] and r["ctas"] > 1 and r["rounds"] == 1 and r["operands"] == 2, r
    _swiglu(M, I, K)


@pytest.mark.parametrize("M,N,K,operands,chunk", [(100, 50000, 256, 1, 32), (16, 60000, 256, 2, 16), (72, 60000, 320, 2, 32), (17, 20488, 192, 1, 32), (64, 60000, 256, 1, 64)])
def test_several_rounds_of_tiles(M, N, K, operands, chunk):
    import paper_2609_27396_b200 as dp
    r = dp.gemm_route(M, N, K, epilogue=3)
    assert r["few_rows"] and r["ctas"] == 1 and r["rounds"] > 1 and (r["operands"], r["chunk"]) == (operands, chunk), r
    _stores(M, N, K)


@pytest.mark.parametrize("M,I,K,chunk", [(40, 30000, 256, 48), (128, 24000, 128, 32)])
def test_several_rounds_of_tiles_swiglu(M, I, K, chunk):
    import paper_2609_27396_b200 as dp
    r = dp.gemm_route(M, I, K, epilogue=2)
    assert r["few_rows"] and r["ctas"] == 1 and r["rounds"] > 1 and r["chunk"] == chunk, r
    _swiglu(M, I, K)


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
