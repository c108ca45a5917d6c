"""A stack of blocks needs every boundary: a part of them is refused, whichever kernels the number of rows takes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [2, 12])     # 24 rows; 144
@pytest.mark.parametrize("part", [(0, 2), (1, 3), (1, 1)])
def test_part_of_the_boundaries_is_refused(batch, part):
    import paper_2609_27396_b200 as dp
    j, bq, hq, hkv, d, hidden, inter = 3, 4, 4, 2, 64, 256, 512
    z = lambda *shape, dtype=torch.bfloat16: torch.zeros(*shape, dtype=dtype, device="cuda")  # noqa: E731
    y = torch.full((batch, j * bq, hidden), -7.0, device="cuda")
    io = dp.make_layer_io(x=z(batch, j * bq, hidden), w_qkv=z((hq + 2 * hkv) * d, hidden), w_o=z(hidden, hq * d), w_gate_up=z(2 * inter, hidden),
                          w_down=z(hidden, inter), y_f32=y, y_bf16=z(batch, j * bq, hidden))
    kc, vc = [z(9 * batch, hkv, d)], [z(9 * batch, hkv, d)]
    plan = dp.BackbonePlan(ctx_offsets=[9 * n for n in range(batch + 1)], n_boundaries=j, block=bq, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, layers=[io],
                           k_ctx=kc, v_ctx=vc, spine_queries=False)
    spine = z(batch, j, hkv, d)
    plan(k_spine=spine, v_spine=spine)  # the whole range: taken
    torch.cuda.synchronize()
    assert int(plan.status.item()) == 0 and not (y == -7.0).any()
    y.fill_(-7.0)
    plan.shape.boundary_lo, plan.shape.boundary_hi = part
    with pytest.raises(dp.DparaError) as e:
        plan(k_spine=spine, v_spine=spine)
    torch.cuda.synchronize()
    assert e.value.code == dp.ERR_UNSUPPORTED and (y == -7.0).all()
