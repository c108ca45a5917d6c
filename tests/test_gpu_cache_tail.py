"""Cache append whose products leave a last round of a few units: those are cut along the candidate rows, over several layers and parts of K."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# requests, rows of each, layers, KV heads, features; parts of K, activation rows of a tile and of the units that a last round's tiles are cut into
@pytest.mark.parametrize("b,rows,layers,hkv,feat,parts,tile,unit", [
    (16, 16, 5, 8, 5120, 4, 256, 64),     # 160 units on 74 pairs: 12 left, four units each
    (13, 13, 5, 8, 5120, 4, 176, 48),     # 169 rows: the last of four units reaches behind the tile and the rows
    (25, 13, 5, 8, 1280, 2, 176, 48),     # 325 rows: two activation tiles, the second of 149 rows
    (37, 11, 5, 4, 5120, 4, 208, 64),     # 407 rows, two tiles
    (33, 8, 7, 4, 128, 1, 96, 32),        # 264 rows, three tiles; K whole
    (10, 20, 5, 8, 1280, 1, 208, 208),    # 40 units: nothing is cut
])
def test_values_of_every_layer(b, rows, layers, hkv, feat, parts, tile, unit):
    """Keys (no gain, no rotation) and values are the projection of the normalised features, rounded to bf16 once: half a step, and what a flipped rounding of a normalised
    input moves (2^-8 * |x| * |w|: 8e-5 typically, 1.3e-3 for |x| = 4 against |w| = 0.08; one input in 10^4 flips, half a one a row of 5120)."""
    import paper_2609_27396_b200 as dp
    d, cap, M, N = 128, 64, b * rows, 2 * hkv * 128
    g = torch.Generator(device="cuda").manual_seed(5)
    bf = lambda sigma, *shape: (sigma * torch.randn(*shape, device="cuda", generator=g)).to(torch.bfloat16)  # noqa: E731
    w = [bf(0.02, N, feat) for _ in range(layers)]
    kc, vc = [[torch.zeros(b * cap, hkv, d, dtype=torch.bfloat16, device="cuda") for _ in range(layers)] for _ in range(2)]
    i64 = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    length = i64([3 * n % 7 for n in range(b)])
    accept = torch.randint(0, rows, (b,), device="cuda", generator=g, dtype=torch.int32)
    accept[0], accept[-1] = rows - 1, rows - 1
    old = length.tolist()
    plan = dp.CachePlan(batch=b, n_rows=rows, w_kv=w, k_ctx=kc, v_ctx=vc, row_start=i64([n * cap for n in range(b)]), capacity=i64([cap] * b), ctx_len=length, use_rope=False)
    # the plan as the call makes it: its parts of K from the planes in its workspace, which lie behind the normalised rows and in front of the lengths
    up = lambda n: -(-n // 256) * 256  # noqa: E731
    assert plan.workspace_bytes == up(2 * M * feat) + up(layers * M * N * 4 * parts) + up(8 * b)
    r = dp.gemm_route(M, N, feat, epilogue=3, n_groups=layers, split_k=parts, one_chain=True)
    assert (r["few_rows"], r["tile_rows"], r["chunk"]) == (0, tile, unit)
    x = bf(1.0, b, rows, feat)
    plan.run(x, accept)
    torch.cuda.synchronize()
    assert int(plan.status.item()) == 0 and length.tolist() == [n + r + 1 for n, r in zip(old, accept.tolist())]
    xn = (x.double() / torch.sqrt((x.double() ** 2).mean(-1, keepdim=True) + 1e-6)).to(torch.bfloat16).double()
    for l in range(layers):
        for cache, at in ((kc[l], 0), (vc[l], hkv * d)):
            want = (xn @ w[l][at: at + hkv * d].double().T).view(b, rows, hkv, d)
            for n, r in enumerate(accept.tolist()):
                got = cache[n * cap + old[n]: n * cap + old[n] + r + 1].double()
                assert ((got - want[n, : r + 1]).abs() <= 2.0 ** -8 * want[n, : r + 1].abs() + 2e-3).all()
                assert not cache[n * cap + old[n] + r + 1: (n + 1) * cap].any() and not cache[n * cap: n * cap + old[n]].any()
