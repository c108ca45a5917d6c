"""The C-ABI library loads, exports what include/dpara.h declares, and rejects bad arguments on the
host before any launch (no GPU needed)."""
import ctypes as C
import os
import re

import pytest

import paper_2609_27396_b200 as dp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    txt = open(os.path.join(ROOT, "include", "dpara.h")).read()
    txt = re.sub(r"/\*.*?\*/", "", txt, flags=re.S)
    return sorted(set(re.findall(r"\b(dpara_[a-z_0-9]+)\s*\(", txt)))


def test_every_declared_symbol_is_exported():
    names = _declared()
    assert "dpara_draft_all_boundaries" in names and "dpara_verify_select" in names
    for n in names:
        assert hasattr(dp.lib, n), n
    assert set(dp.EXPORTED) <= set(names)


def test_status_strings_and_version():
    assert dp.lib.dpara_version() >= 1000
    for code in (0, -1, -2, -3, -4, -5):
        assert len(dp.lib.dpara_status_string(code)) > 0


def _shape(**kw):
    d = dict(batch=1, n_boundaries=3, block=2, n_q_heads=4, n_kv_heads=2, head_dim=64, prefix_base=1, n_spine=3,
             boundary_lo=0, boundary_hi=3, softmax_scale=0.0, spine_queries=0)
    d.update(kw)
    return dp.Shape(*[d[f[0]] for f in dp.Shape._fields_])


def test_draft_argument_validation():
    off = (C.c_int64 * 2)(0, 5)
    io = dp.AttnIO()
    call = lambda s, i: dp.lib.dpara_draft_all_boundaries(C.byref(s), C.byref(i) if i is not None else None, None, None, 0, None, None)
    assert call(_shape(head_dim=96), io) == dp.ERR_UNSUPPORTED
    assert call(_shape(n_q_heads=3), io) == dp.ERR_UNSUPPORTED
    assert call(_shape(batch=0), io) == dp.ERR_INVALID_ARG
    assert call(_shape(boundary_hi=4), io) == dp.ERR_INVALID_ARG
    assert call(_shape(spine_queries=2), io) == dp.ERR_INVALID_ARG
    assert call(_shape(spine_queries=1, boundary_lo=1), io) == dp.ERR_UNSUPPORTED    # spine rows need the full boundary range
    assert call(_shape(), None) == dp.ERR_INVALID_ARG
    assert call(_shape(), io) == dp.ERR_INVALID_ARG                     # no host offsets
    io.host_ctx_offsets = C.cast(off, C.c_void_p).value
    assert call(_shape(), io) == dp.ERR_INVALID_ARG                     # null device pointers
    bad = (C.c_int64 * 2)(5, 0)
    io.host_ctx_offsets = C.cast(bad, C.c_void_p).value
    assert call(_shape(), io) == dp.ERR_INVALID_ARG                     # decreasing offsets
    assert dp.lib.dpara_draft_workspace_bytes(C.byref(_shape(head_dim=7)), C.cast(off, C.c_void_p), None, 0) == 0


def test_verify_argument_validation():
    io = dp.VerifyIO(2, 4, 100, 2, 8, 0)
    assert dp.lib.dpara_verify_workspace_bytes(C.byref(io)) > 0
    assert dp.lib.dpara_verify_select(C.byref(io), None, 0, None, None) == dp.ERR_INVALID_ARG      # null tensors
    assert dp.lib.dpara_verify_select(None, None, 0, None, None) == dp.ERR_INVALID_ARG
    io2 = dp.VerifyIO(2, 100, 100, 2, 8, 0)
    assert dp.lib.dpara_verify_workspace_bytes(C.byref(io2)) == 0                                   # J > 64
    io3 = dp.VerifyIO(2, 4, 100, 2, 8, 0, 16, None, 16, None, None, 16, 16, 16, None, None)
    assert dp.lib.dpara_verify_select(C.byref(io3), None, 0, None, None) == dp.ERR_WORKSPACE
    io4 = dp.VerifyIO(2, 4, 100, 2, 8, 1, 16, None, 16, None, None, 16, 16, 16, None, None)
    assert dp.lib.dpara_verify_select(C.byref(io4), None, 0, None, None) == dp.ERR_INVALID_ARG      # sampling needs uniforms
    io5 = dp.VerifyIO(2, 4, 100, 2, 8, 7)
    assert dp.lib.dpara_verify_workspace_bytes(C.byref(io5)) == 0                                   # bad mode


@pytest.mark.parametrize("kw", [
    dict(M=256, epilogue=1, n_groups=2),                      # one residual for all products
    dict(M=256, epilogue=2, n_groups=2),
    dict(M=256, epilogue=3, n_groups=2, row_order=True),
    dict(M=128, epilogue=3, split_k=2),                       # the kernel for few rows takes no planes
    dict(M=256, epilogue=0, split_k=2),
    dict(M=256, epilogue=3, split_k=2, row_order=True),
    dict(M=256, epilogue=3, split_k=9),                       # more parts than 64-column slabs of K
    dict(M=256, epilogue=0, n_groups=9),
])
def test_gemm_launches_that_are_refused(kw):
    with pytest.raises(dp.DparaError) as e:
        dp.gemm_route(N=512, K=512, **kw)
    assert e.value.code == dp.ERR_UNSUPPORTED


@pytest.mark.parametrize("kw", [dict(M=256, epilogue=3, n_groups=8, split_k=4), dict(M=8, epilogue=0, n_groups=8, one_chain=True), dict(M=256, epilogue=3, row_order=True)])
def test_gemm_launches_that_are_taken(kw):
    assert dp.gemm_route(N=512, K=512, **kw)["rounds"] >= 1


@pytest.mark.parametrize("M,rows", [(129, 144), (160, 160), (200, 208)])
def test_streamed_weights_are_read_by_one_pair(M, rows):
    """Many rounds of weights: tiles of all activation rows, since pairs that read the same weights do not fetch them once."""
    for N, K in ((151936, 2048), (151936, 5120), (75968, 4096)):
        r = dp.gemm_route(M, N, K, epilogue=3)
        assert r["few_rows"] == 0 and r["tile_rows"] == rows, r


def test_few_rounds_of_streamed_weights():
    """Two rounds of all 256 rows or three of half of them: the latter, as long as three rounds are enough."""
    assert dp.gemm_route(256, 12288, 4096, epilogue=2)["tile_rows"] == 128
    assert dp.gemm_route(256, 17408, 5120, epilogue=2)["tile_rows"] == 256


@pytest.mark.parametrize("M", [200, 256, 512, 1024])
def test_short_products_take_narrower_tiles(M):
    """K of one slab: the last tile's epilogue is most of the launch, so the activation rows are cut further than into tiles of 256."""
    r = dp.gemm_route(M, 264, 64)
    assert r["few_rows"] == 0 and r["tile_rows"] <= 176 and r["rounds"] == 1, r


def test_rings_of_the_kernel_for_few_rows():
    """Two slabs per stage leave a ring of three stages, of four above 64 activation rows, beside what lies behind the ring (at least 16 KB)."""
    two = 0
    for M in (1, 16, 17, 40, 64, 72, 100, 128):
        for N, K in ((264, 512), (6144, 4096), (5120, 17408), (20480, 8192), (151936, 5120), (151936, 64)):
            r = dp.gemm_route(M, N, K, epilogue=3)
            assert r["few_rows"] == 1 and r["slabs"] in (1, 2)
            two += r["slabs"] == 2
            stage = 2 * 128 * (r["operands"] * r["weight_rows"] + r["tile_rows"])
            assert r["slabs"] == 1 or (3 if M <= 64 else 4) * stage <= (227 - 16) * 1024, (M, N, K, r)
    assert two > 10


def _append_of_two_layers(**kw):
    """The host's answer to an append whose pointers are 4096 except for those given; without a workspace, so that nothing is launched."""
    n = 2
    d = dict(features=4096, w_kv=[4096] * n, norm=[4096] * n, knorm=[4096] * n, k=[4096] * n, v=[4096] * n)
    d.update(kw)
    tabs = [(C.c_void_p * n)(*d[k]) for k in ("w_kv", "norm", "knorm", "k", "v")]
    io = dp.CacheIO(1, 4, 128, 2, 64, n, d["features"], 4096, *[C.addressof(t) for t in tabs], 4096, 4096, 4096, 1e-6, 1e6, 1)
    return dp.lib.dpara_cache_append(C.byref(io), None, 0, None, None)


def test_append_refuses_misaligned_tensors():
    assert _append_of_two_layers() == dp.ERR_WORKSPACE                                  # nothing else is wrong
    assert _append_of_two_layers(norm=[None, 4096], knorm=[4096, None]) == dp.ERR_WORKSPACE
    for name in ("w_kv", "norm", "knorm", "k", "v"):
        for off in (2, 8):
            assert _append_of_two_layers(**{name: [4096, 4096 + off]}) == dp.ERR_INVALID_ARG, (name, off)
    assert _append_of_two_layers(features=4098) == dp.ERR_INVALID_ARG


@pytest.mark.parametrize("mode", [0, 1])
def test_workspace_of_a_larger_select_serves_a_smaller_one(mode):
    """A program that sizes one workspace for its largest batch calls with fewer requests and boundaries too."""
    need = lambda b, J, V: dp.lib.dpara_verify_workspace_bytes(C.byref(dp.VerifyIO(b, J, V, 2, 64, mode)))
    for V in (1, 1000, 20000, 60000, 151936):
        for J in (1, 2, 5, 16, 37, 64):
            for b in list(range(1, 80)) + [150, 444, 445]:
                most = need(b, J, V)
                assert need(b + 1, J, V) >= most and (J == 64 or need(b, J + 1, V) >= most) and need(b, J, V + 5000) >= most, (b, J, V)


@pytest.mark.parametrize("raw", [None, lambda device: 100 + device])
def test_stream_handle_with_and_without_the_raw_query(monkeypatch, raw):
    class Stream:
        cuda_stream = 103
    monkeypatch.setattr(dp, "_raw_stream", raw)
    monkeypatch.setattr(dp.torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(dp.torch.cuda, "current_stream", lambda: Stream)
    assert dp._stream_ptr(None) == 103
    Stream.cuda_stream = 7
    assert dp._stream_ptr(Stream) == 7


LAYER_POINTERS = ("x", "w_qkv", "w_o", "w_gate_up", "w_down", "rms1_w", "rms2_w", "qnorm_w", "knorm_w", "y_f32", "y_bf16")


def _blocks(n_layers, **at):
    """The host's answer to a block or a stack of blocks whose pointers are 4096 except the last block's given ones; without a workspace, so that nothing is launched."""
    off = (C.c_int64 * 2)(0, 0)
    io = dp.AttnIO(ctx_offsets=4096, host_ctx_offsets=C.addressof(off), k_spine=4096, v_spine=4096)
    ios = [dp.LayerIO(rms_eps=1e-6, rope_theta=1e6, use_rope=1, hidden=128, intermediate=128, **{k: 4096 for k in LAYER_POINTERS}) for _ in range(n_layers or 1)]
    for name, p in at.items():
        setattr(ios[-1 if name != "x" else 0], name, p)
    if not n_layers:
        return dp.lib.dpara_draft_all_boundaries(C.byref(_shape()), C.byref(io), C.byref(ios[0]), None, 0, None, None)
    layers, caches = (dp.LayerIO * n_layers)(*ios), (C.c_void_p * n_layers)(*[4096] * n_layers)
    bb = dp.BackboneIO(n_layers, C.addressof(layers), C.addressof(caches), C.addressof(caches))
    return dp.lib.dpara_draft_backbone(C.byref(_shape()), C.byref(io), C.byref(bb), None, 0, None, None)


@pytest.mark.parametrize("n_layers", [0, 1, 3])
def test_blocks_refuse_misaligned_tensors(n_layers):
    assert _blocks(n_layers) == dp.ERR_WORKSPACE                                        # nothing else is wrong
    assert _blocks(n_layers, rms1_w=None, rms2_w=None, qnorm_w=None, knorm_w=None, y_bf16=None) == dp.ERR_WORKSPACE
    for name in LAYER_POINTERS:
        assert _blocks(n_layers, **{name: 4098}) == dp.ERR_INVALID_ARG, name
    assert _blocks(n_layers, qnorm_w=4100, knorm_w=4104) == dp.ERR_WORKSPACE            # the row-wise kernel takes these


@pytest.mark.parametrize("hq,hkv,d,hidden,inter", [(40, 8, 128, 5120, 17408), (32, 8, 128, 4096, 12288), (16, 4, 64, 256, 512), (2, 2, 64, 64, 64), (64, 8, 128, 5184, 8192)])
def test_workspace_of_a_larger_batch_serves_a_smaller_one(hq, hkv, d, hidden, inter):
    """A serving loop's batch varies under one workspace.  The blocks' part of it (the attention's scratch is asked for by the same query, and not this test's)."""
    layers = (dp.LayerIO * 3)(*[dp.LayerIO(rms_eps=1e-6, rope_theta=1e6, use_rope=1, hidden=hidden, intermediate=inter) for _ in range(3)])
    bb = dp.BackboneIO(3, C.addressof(layers), None, None)
    for j, bq in ((8, 1), (5, 1), (1, 1), (3, 5), (8, 8)):
        for spine in (0, 1):
            most = [0, 0]
            for b in range(1, 140):
                shape = _shape(batch=b, n_boundaries=j, boundary_hi=j, n_spine=j, block=bq, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, spine_queries=spine)
                off = C.cast((C.c_int64 * (b + 1))(*[9 * n for n in range(b + 1)]), C.c_void_p)
                attn = dp.lib.dpara_draft_workspace_bytes(C.byref(shape), off, None, 0)
                need = [dp.lib.dpara_draft_workspace_bytes(C.byref(shape), off, C.byref(layers[0]), 1) - attn, dp.lib.dpara_backbone_workspace_bytes(C.byref(shape), off, C.byref(bb)) - attn]
                assert need[0] >= most[0] and need[1] >= most[1], (j, bq, spine, b, need, most)
                most = need
