"""SiLU of the gated products: every bf16 value as a gate, through both products that have the epilogue."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [96, 2048])   # the product for few rows; CTA pairs
def test_every_gate_value(rows):
    """gate = x (one column of the activations), up = 1: out is silu(x) rounded once to bf16, from an fp32 value a few of its steps off (the exponential's): one step of bf16 at a
    rounding boundary.  Below -88 the exponential overflows and the result is -0; its size is below 1e-36."""
    import paper_2609_27396_b200 as dp
    bits = torch.arange(1 << 16, dtype=torch.int32, device="cuda").to(torch.int16).view(torch.bfloat16)
    x = bits[torch.isfinite(bits)]
    w = torch.zeros(2 * 64, 64, dtype=torch.bfloat16, device="cuda")
    w[:64, 0] = 1
    w[64:, 1] = 1
    for part in x.split(rows):
        a = torch.zeros(rows, 64, dtype=torch.bfloat16, device="cuda")
        a[: len(part), 0] = part
        a[:, 1] = 1
        out = dp.gemm_bf16(a, w, epilogue=2)[0]
        z = part.double()
        want = z / (1 + torch.exp(-z))
        got = out[: len(part), 0].double()
        assert ((got - want).abs() <= 2.0 ** -7 * want.abs() + 1e-36).all()
        assert torch.equal(out[: len(part)], out[: len(part), :1].expand(-1, 64))


SILU_F32 = """
#include "gemm.cuh"
__global__ void eval(const float *g, float *ours, float *plain, float *denominator, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float d = 1.0f + __expf(-g[i]);
  ours[i] = dpara::silu(g[i]);
  plain[i] = g[i] / d;
  denominator[i] = d;
}
extern "C" int silu_f32(const float *g, float *ours, float *plain, float *denominator, int n) {
  eval<<<(n + 255) / 256, 256>>>(g, ours, plain, denominator, n);
  return cudaGetLastError();
}
"""


def test_the_quotient_in_fp32(tmp_path):
    """silu's quotient against float64's and against CUDA's `/`, on its own denominator: half an ulp and 2^-17 of one (the error ahead of the rounding is below 2^-41 of the
    quotient), so at most one ulp from the rounded quotient.  Random bit patterns, every bf16 value, what a gate is in earnest, and where the denominator nears overflow."""
    import ctypes
    from gpu_util import compile_native
    lib = compile_native(tmp_path, SILU_F32)
    gen = torch.Generator(device="cuda").manual_seed(1)
    bits = torch.randint(-(1 << 31), 1 << 31, (1 << 23,), device="cuda", generator=gen, dtype=torch.int64).to(torch.int32).view(torch.float32)
    all_bf16 = (torch.arange(1 << 16, device="cuda", dtype=torch.int64) << 16).to(torch.int32).view(torch.float32)
    uniform = lambda lo, hi, n: torch.rand(n, device="cuda", generator=gen) * (hi - lo) + lo  # noqa: E731
    special = torch.tensor([float("inf"), float("-inf"), float("nan"), 0.0, -0.0, 3.4028235e38, -3.4028235e38, 1e-45, -1e-45, -87.3, -87.34, -88.0, -88.72, -88.73, -89.0],
                           device="cuda")
    g = torch.cat([bits, all_bf16, uniform(-30, 30, 1 << 23), uniform(-90, -85, 1 << 21), uniform(-1e-3, 1e-3, 1 << 20), special]).contiguous()
    ours, plain, d = (torch.empty_like(g) for _ in range(3))
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.silu_f32(p(g), p(ours), p(plain), p(d), g.numel()) == 0
    torch.cuda.synchronize()
    exact = g.double() / d.double()
    assert torch.equal(torch.isnan(ours), torch.isnan(exact)) and torch.equal(torch.isnan(ours), torch.isnan(plain))   # a NaN, or -inf
    fin = torch.isfinite(exact)
    assert torch.equal(ours[~fin].nan_to_num(7.0), plain[~fin].nan_to_num(7.0)) and int((d > 2.0 ** 126).sum()) > 1000 and int(torch.isinf(d).sum()) > 1000
    o, e = ours[fin].double(), exact[fin]
    ulp = torch.ldexp(torch.ones_like(e), torch.frexp(e.abs().clamp(min=2.0 ** -126)).exponent - 24)
    err = (o - e).abs() / ulp
    apart = (o - plain[fin].double()).abs() / ulp
    print(f"largest error {float(err.max()):.7f} ulp, {int((apart > 0).sum())} of {o.numel()} another float than CUDA's `/`")
    assert float(err.max()) <= 0.5 + 2.0 ** -17 and float(apart.max()) <= 1.0
    assert torch.equal(torch.signbit(ours[fin]), torch.signbit(plain[fin]))
