"""Cache append whose products leave a last round of a few units: those are cut along the candidate rows, over several layers and parts of K."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,rows,layers", [(16, 16, 5), (10, 20, 5), (13, 13, 8)])   # 12, 12 and 54 (whole tiles) units left of 160, 160 and 128
def test_values_of_every_layer(b, rows, layers):
    """v rows are the projection of the normalised features, rounded to bf16 once: half a step, and what a flipped rounding of a normalised input moves (a few of them at most
    2^-8 * |x| * |w| = 4e-4 each)."""
    import paper_2609_27396_b200 as dp
    g = torch.Generator(device="cuda").manual_seed(5)
    hkv, d, feat, cap = 8, 128, 1280, 64
    bf = lambda sigma, *shape: (sigma * torch.randn(*shape, device="cuda", generator=g)).to(torch.bfloat16)  # noqa: E731
    w = [bf(0.02, 2 * hkv * d, feat) for _ in range(layers)]
    kc, vc = [[torch.zeros(b * cap, hkv, d, dtype=torch.bfloat16, device="cuda") for _ in range(layers)] for _ in range(2)]
    i64 = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    length = i64([3 * n % 7 for n in range(b)])
    accept = torch.randint(0, rows, (b,), device="cuda", generator=g, dtype=torch.int32)
    accept[0], accept[-1] = rows - 1, 0
    old = length.tolist()
    plan = dp.CachePlan(batch=b, n_rows=rows, w_kv=w, k_ctx=kc, v_ctx=vc, row_start=i64([n * cap for n in range(b)]), capacity=i64([cap] * b), ctx_len=length)
    x = bf(1.0, b, rows, feat)
    plan.run(x, accept)
    torch.cuda.synchronize()
    assert int(plan.status.item()) == 0 and length.tolist() == [n + r + 1 for n, r in zip(old, accept.tolist())]
    xn = (x.double() / torch.sqrt((x.double() ** 2).mean(-1, keepdim=True) + 1e-6)).to(torch.bfloat16).double()
    for l in range(layers):
        want = (xn @ w[l][hkv * d:].double().T).view(b, rows, hkv, d)
        for n, r in enumerate(accept.tolist()):
            got = vc[l][n * cap + old[n]: n * cap + old[n] + r + 1].double()
            assert ((got - want[n, : r + 1]).abs() <= 2.0 ** -8 * want[n, : r + 1].abs() + 2e-3).all()
            assert not vc[l][n * cap + old[n] + r + 1: (n + 1) * cap].any() and not vc[l][n * cap: n * cap + old[n]].any()
