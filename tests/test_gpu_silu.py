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
