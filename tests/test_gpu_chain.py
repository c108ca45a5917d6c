"""The few-row chain (everything between two attentions in one launch, up to 128 rows) against the kernels of their own that larger batches take.

The same requests run alone (at most 128 rows: the chain) and at the head of a batch with more requests behind them (more rows: kernels of their own); rows of
different requests never meet, so their outputs have to agree.  Bound: the two add a product's sums in different orders, so a bf16 rounding of an activation may flip; the layer
tests give what such flips do to a block's output, 4e-3 of its rms, and 1.6e-2 at most for a single element of ~1e5; held here to 1e-2 (2-norm) and 8e-2 of the rms."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _weights(g, hidden, inter, hq, hkv, d, norm):
    bf = lambda sigma, *shape: (sigma * torch.randn(*shape, device=DEV, generator=g)).to(torch.bfloat16)  # noqa: E731
    gain = lambda n: (1 + 0.1 * torch.randn(n, device=DEV, generator=g)).to(torch.bfloat16)  # noqa: E731
    w = dict(w_qkv=bf(hidden ** -0.5, (hq + 2 * hkv) * d, hidden), w_o=bf((hq * d) ** -0.5, hidden, hq * d), w_gate_up=bf(hidden ** -0.5, 2 * inter, hidden),
             w_down=bf(inter ** -0.5, hidden, inter))
    return dict(w, rms1_w=gain(hidden), rms2_w=gain(hidden), qnorm_w=gain(d), knorm_w=gain(d)) if norm else w


class _Stack:
    """A stack of blocks over `b` requests of (j * bq + j) rows each, or one block without spine rows."""

    def __init__(self, x, w, caches, lens, j, bq, heads, spine=None):
        import paper_2609_27396_b200 as dp
        b = x.shape[0]
        hq, hkv, d = heads
        off = [0]
        for n in lens[:b]:
            off.append(off[-1] + n)
        self.x, self.w = x.contiguous(), w
        self.y, self.y16 = torch.zeros(*x.shape, device=DEV), torch.zeros(*x.shape, device=DEV, dtype=torch.bfloat16)
        self.kc, self.vc = [c[0][: off[-1]] for c in caches], [c[1][: off[-1]] for c in caches]
        io = [dp.make_layer_io(x=self.x, **k, y_f32=self.y, y_bf16=self.y16) for k in w]
        shape = dict(ctx_offsets=off, n_boundaries=j, block=bq, n_q_heads=hq, n_kv_heads=hkv, head_dim=d)
        self.spine = [t[:b] for t in spine] if spine else None
        self.plan = dp.DraftPlan(**shape, layer=io[0]) if spine else dp.BackbonePlan(**shape, layers=io, k_ctx=self.kc, v_ctx=self.vc)

    def __call__(self):
        if self.spine:
            self.plan(k_ctx=self.kc[0], v_ctx=self.vc[0], k_spine=self.spine[0], v_spine=self.spine[1])
        else:
            self.plan()


def _case(seed, b, more, j, bq, heads, hidden, inter, layers, norm=True, spine_rows=True, rope=True):
    g = torch.Generator(device=DEV).manual_seed(seed)
    hq, hkv, d = heads
    rows = j * bq + (j if spine_rows else 0)
    lens = [int(n) for n in torch.randint(1, 90, (b + more,), generator=torch.Generator().manual_seed(seed))]
    x = torch.randn(b + more, rows, hidden, device=DEV, generator=g).to(torch.bfloat16)
    w = [dict(_weights(g, hidden, inter, hq, hkv, d, norm), use_rope=rope) for _ in range(layers)]
    kv = lambda *shape: torch.randn(*shape, device=DEV, generator=g).to(torch.bfloat16)  # noqa: E731
    caches = [(kv(sum(lens), hkv, d), kv(sum(lens), hkv, d)) for _ in range(layers)]
    spine = None if spine_rows else (kv(b + more, j, hkv, d), kv(b + more, j, hkv, d))
    few = _Stack(x[:b], w, caches, lens, j, bq, heads, spine)
    many = _Stack(x, w, caches, lens, j, bq, heads, spine)
    assert b * rows <= 128 < (b + more) * rows
    return few, many


def _agree(few, many):
    for a, r in ((few.y, many.y), (few.y16, many.y16)):
        a, r = a.double(), r[: a.shape[0]].double()
        rms = r.pow(2).mean().sqrt()
        assert ((a - r).norm() / r.norm()) <= 1e-2 and (a - r).abs().max() <= 8e-2 * rms


@pytest.mark.parametrize("b,more,j,bq,heads,hidden,inter,layers,norm,spine_rows,rope", [
    (1, 70, 1, 1, (2, 2, 64), 64, 64, 2, True, True, True),            # two rows, one slab of K, fewer tiles than SMs
    (1, 8, 4, 3, (8, 2, 128), 512, 1536, 3, True, True, True),         # exactly one multiple of 16
    (1, 8, 1, 16, (10, 2, 64), 320, 448, 2, False, True, False),       # 17 rows; odd numbers of slabs; no gains, no rotation
    (2, 1, 8, 7, (20, 4, 64), 896, 2432, 2, True, True, True),         # 128 rows: the most
    (1, 1, 8, 15, (8, 8, 128), 1088, 3136, 1, True, True, True),
    (1, 1, 10, 8, (16, 4, 128), 1024, 3072, 1, True, False, True),     # 80 rows (four stages of activations), block without spine rows
    (1, 1, 9, 9, (16, 2, 128), 1536, 4096, 1, True, False, True),      # 81 (three)
    (1, 1, 9, 8, (40, 8, 128), 5120, 17408, 1, True, True, True),      # the widest rows
])
def test_chain_against_kernels_of_their_own(b, more, j, bq, heads, hidden, inter, layers, norm, spine_rows, rope):
    import paper_2609_27396_b200 as dp
    few, many = _case(7, b, more, j, bq, heads, hidden, inter, layers, norm, spine_rows, rope)
    before = dp.lib.dpara_kernel_launches()
    few()
    assert dp.lib.dpara_kernel_launches() - before == 1 + layers + (layers + 1)      # a norm, attentions, chains
    many()
    torch.cuda.synchronize()
    assert int(few.plan.status.item()) == 0 and int(many.plan.status.item()) == 0
    _agree(few, many)
    first = few.y.clone()
    few()
    torch.cuda.synchronize()
    assert torch.equal(first, few.y)


def test_chain_takes_one_launch_between_attentions():
    import paper_2609_27396_b200 as dp
    few, many = _case(3, 1, 4, 4, 8, (8, 2, 64), 256, 512, 3)
    before = dp.lib.dpara_kernel_launches()
    few()
    alone = dp.lib.dpara_kernel_launches() - before
    many()
    torch.cuda.synchronize()
    assert alone == 1 + 3 + 4 and dp.lib.dpara_kernel_launches() - before - alone == 8 * 3


@pytest.mark.parametrize("j,bq,heads,hidden,inter,one", [
    (8, 8, (16, 4, 128), 1536, 4608, True),      # 72 rows, 58 MB of weights
    (8, 8, (16, 4, 128), 1600, 5120, False),     # 66
    (8, 3, (8, 2, 64), 768, 2304, True),         # 32 rows, 13 MB
    (8, 3, (8, 2, 64), 1024, 3072, False),       # 21
    (11, 2, (8, 2, 64), 1024, 3072, True),       # 33 rows
])
def test_one_block_goes_where_it_is_faster(j, bq, heads, hidden, inter, one):
    """One block of few rows takes the chain by its rows and weights; a stack of two such blocks takes it at all of these sizes."""
    import paper_2609_27396_b200 as dp
    for layers in (1, 2):
        few, many = _case(9, 1, 4, j, bq, heads, hidden, inter, layers)
        before = dp.lib.dpara_kernel_launches()
        few()
        assert dp.lib.dpara_kernel_launches() - before == (2 * layers + 2 if one or layers == 2 else 8)
        many()
        torch.cuda.synchronize()
        assert int(few.plan.status.item()) == 0
        _agree(few, many)


REFUSED = """
#define launch_chain launch_chain_as_it_is
#include "chain.cu"
#undef launch_chain
namespace dpara {
dpara_status launch_chain(const ChainShape &, const ChainArgs &, int32_t *, cudaStream_t) { return DPARA_ERR_UNSUPPORTED; }
}
"""


@pytest.mark.parametrize("spine_rows,layers", [(True, 3), (False, 1)])
def test_refused_cooperative_launch(tmp_path, monkeypatch, spine_rows, layers):
    """Where the grid of the chain cannot be held at once (here: the library with a launch that says so), the same call goes through kernels of their own."""
    import paper_2609_27396_b200 as dp
    from gpu_util import compile_native
    few, many = _case(5, 1, 4, 4, 8, (16, 4, 64), 256, 512, layers, spine_rows=spine_rows)
    many()
    lib = compile_native(tmp_path, REFUSED, without="chain")
    for name in dp.EXPORTED:
        getattr(lib, name).restype, getattr(lib, name).argtypes = getattr(dp.lib, name).restype, getattr(dp.lib, name).argtypes
    monkeypatch.setattr(dp, "_draft_packed", type(dp._draft_packed)(("dpara_draft_all_boundaries", lib)))
    monkeypatch.setattr(dp, "lib", lib)
    few()
    torch.cuda.synchronize()
    assert lib.dpara_kernel_launches() == 1 + 8 * layers      # (the norm ahead of the refused launch)
    assert int(few.plan.status.item()) == 0 and int(many.plan.status.item()) == 0
    _agree(few, many)


def test_chain_beside_other_streams():
    """The chain, whose CTAs wait for one another, beside streams that keep the SMs busy: the head loop (a cooperative launch too) behind its LM head, and grids of kernels that hold
    all SMs, a few of them, or come and go.  What the calls give alone, bit for bit."""
    import paper_2609_27396_b200 as dp
    few, _many = _case(21, 1, 2, 8, 7, (16, 4, 128), 1024, 3072, 3)
    g = torch.Generator(device=DEV).manual_seed(4)
    bf = lambda sigma, *shape: (sigma * torch.randn(*shape, device=DEV, generator=g)).to(torch.bfloat16)  # noqa: E731
    b, block, hidden, vocab, rank = 2, 6, 512, 30008, 256
    head, head_in = dp.HeadPlan(b, block, hidden, vocab, rank), (bf(1.0, b, block, hidden), bf(0.05, vocab, hidden), bf(0.3, vocab, rank), bf(0.3, vocab, rank),
                                                                 torch.zeros(b, dtype=torch.int32, device=DEV))
    wide, narrow, x = bf(0.02, 4096, 4096), bf(0.02, 256, 4096), bf(1.0, 512, 4096)
    few()
    head.run(*head_in)
    torch.cuda.synchronize()
    alone = [t.clone() for t in (few.y, few.y16, head.next_tokens)]
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(streams[0]):
            few()
        with torch.cuda.stream(streams[1]):
            head.run(*head_in)
        with torch.cuda.stream(streams[2]):
            for _ in range(4):
                x @ wide.T
        with torch.cuda.stream(streams[3]):
            for _ in range(10):
                x[:64] @ narrow.T
    torch.cuda.synchronize()
    assert int(few.plan.status.item()) == 0 and int(head.status.item()) == 0
    for got, want in zip((few.y, few.y16, head.next_tokens), alone):
        assert torch.equal(got, want)


def test_chains_on_two_streams_and_in_a_graph():
    """Two stacks of the chain in streams without order, then captured in a graph and replayed on other inputs."""
    pairs = [_case(s, 1, 2, 8, 7, (16, 4, 64), 640, 1984, 3) for s in (11, 12)]
    streams = [torch.cuda.Stream() for _ in pairs]
    torch.cuda.synchronize()
    for _ in range(10):
        for (few, _m), st in zip(pairs, streams):
            with torch.cuda.stream(st):
                few()
    torch.cuda.synchronize()
    for few, many in pairs:
        many()
        torch.cuda.synchronize()
        assert int(few.plan.status.item()) == 0
        _agree(few, many)
    few, many = pairs[0]
    with torch.cuda.stream(streams[0]):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=streams[0]):
            few()
    few.x.copy_(-few.x)
    many.x[:1].copy_(few.x)
    graph.replay()
    graph.replay()
    many()
    torch.cuda.synchronize()
    _agree(few, many)
