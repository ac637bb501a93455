"""How the library launches: every kernel is counted, and kernels that are placed while the one before them runs give the same results in
a replayed graph and beside those of another host thread."""
import threading

import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu
SEQ, ROW, BUDGET = vb.PER_SEQUENCE, vb.PER_QUERY, vb.PER_QUERY_BUDGET


class Layer:
    """A layer's handle with inputs; `one_pass`: the router gets scratch whatever the size (it asks for some only on large problems)."""

    def __init__(self, heads_q, heads_kv, dim, grid, topk, mode=ROW, flags=0, cube=(4, 4, 4), text=0, one_pass=False, seed=1, hidden=0):
        n = -(-grid[0] // cube[0]) * -(-grid[1] // cube[1]) * -(-grid[2] // cube[2])
        self.budgets, cap = None, 0
        gen = torch.Generator(device="cuda").manual_seed(seed)
        if mode == BUDGET:
            self.budgets = torch.randint(0, 30, (1, heads_q, n), device="cuda", generator=gen, dtype=torch.int32)
            cap = int(self.budgets.clamp(max=n).sum(-1).max())
        self.p = vb.make_params(1, heads_q, heads_kv, dim, grid, cube=cube, select_mode=mode, topk=topk, text_len=text, flags=flags,
                                nnz_cap=cap)
        self.attn, self.hidden, rows = vb.Vsa2Attention(self.p), hidden, grid[0] * grid[1] * grid[2]
        self.shapes = (heads_q, heads_kv, heads_kv, heads_q), rows + text, dim
        self.gate_shape = (1, heads_q, rows)
        tiles = -(-8 * n * (2 if cube[2] == 8 else 1) // 128)
        self.scratch = torch.empty(148 * tiles * 8192 + heads_q * (4 * 128 * tiles + 4 * n) + (2 << 20), dtype=torch.uint8,
                                   device="cuda") if one_pass else None
        if hidden:
            self.x = torch.randn(1, rows, hidden, device="cuda", generator=gen).bfloat16()
            self.w = (torch.randn(hidden, heads_q, device="cuda", generator=gen) / hidden ** 0.5).bfloat16()
            self.ws_gate = torch.empty(vb.vsa2_gate_bwd_workspace_bytes(self.p, hidden), dtype=torch.uint8, device="cuda")
        self.q, self.k, self.v, self.d_o, self.gate = self.inputs(seed)

    def inputs(self, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        heads, rows, dim = self.shapes
        x = [torch.randn(1, h, rows, dim, device="cuda", generator=gen).bfloat16() for h in heads]
        return x + [torch.rand(*self.gate_shape, device="cuda", generator=gen)]

    def __call__(self):
        a, out = self.attn, []
        if self.hidden:
            vb.vsa2_gate_fwd(self.p, self.hidden, self.x, self.w, self.gate)
        if self.scratch is None:
            a.route(self.q, self.k, self.budgets)
        else:
            vb.vsa2_route(self.p, self.q, self.k, self.budgets, a.map, a.ws_route, scratch=self.scratch)
        o, lse = a.forward(self.q, self.k, self.v, self.gate)
        out = [o, lse, *a.backward(self.q, self.k, self.v, self.gate, o, lse, self.d_o)]
        if self.hidden:
            out += [torch.empty(self.w.shape, dtype=torch.float32, device="cuda"), torch.empty_like(self.x)]
            vb.vsa2_gate_bwd(self.p, self.hidden, self.x, self.w, self.gate, out[5], out[6], out[7], self.ws_gate)
        return out


def _kernels(graph):
    """Kernel nodes of a captured graph."""
    from cuda.bindings import runtime as rt
    raw = rt.cudaGraph_t(graph.raw_cuda_graph())
    _, _, n = rt.cudaGraphGetNodes(raw)
    _, nodes, n = rt.cudaGraphGetNodes(raw, n)
    kinds = [rt.cudaGraphNodeGetType(x)[1] for x in nodes[:n]]
    return sum(k == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel for k in kinds)


LAYERS = [
    dict(heads_q=2, heads_kv=2, dim=64, grid=(4, 8, 8), topk=2),                                        # few blocks: no list is long
    dict(heads_q=4, heads_kv=2, dim=128, grid=(8, 16, 16), topk=9, hidden=64),                          # grouped heads, fp16 form
    dict(heads_q=4, heads_kv=2, dim=64, grid=(8, 16, 16), topk=3, mode=SEQ),                            # grouped heads, pair form
    dict(heads_q=2, heads_kv=2, dim=128, grid=(16, 40, 40), topk=5, mode=SEQ),                          # 400 blocks: long lists
    dict(heads_q=2, heads_kv=2, dim=128, grid=(8, 16, 16), topk=5, flags=vb.FLAG_FAST_BWD),
    dict(heads_q=2, heads_kv=2, dim=128, grid=(8, 16, 16), topk=5, flags=vb.FLAG_PRECISE_BWD),
    dict(heads_q=2, heads_kv=1, dim=64, grid=(5, 32, 64), topk=7, flags=vb.FLAG_GROUP_ROUTING, one_pass=True),   # packed query cubes
    dict(heads_q=2, heads_kv=2, dim=128, grid=(13, 30, 45), topk=9, mode=SEQ, one_pass=True),
    dict(heads_q=2, heads_kv=2, dim=128, grid=(9, 24, 40), topk=0, mode=BUDGET, text=70),
    dict(heads_q=3, heads_kv=3, dim=128, grid=(8, 16, 32), topk=5, cube=(4, 4, 8)),
    dict(heads_q=2, heads_kv=1, dim=64, grid=(12, 20, 40), topk=5, cube=(4, 4, 8), mode=SEQ),
]


def _name(layer):
    return "-".join(str(v) for v in layer.values()).replace(" ", "")


@pytest.mark.parametrize("layer", LAYERS, ids=_name)
def test_launch_count_is_the_number_of_kernels(layer):
    layer = Layer(**layer)
    layer()                                      # (what is looked up once per process)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    before = vb.vsa2_launch_count()
    with torch.cuda.graph(graph):
        layer()
    assert vb.vsa2_launch_count() - before == _kernels(graph)


REPLAYED = [
    dict(heads_q=9, heads_kv=9, dim=128, grid=(21, 30, 52), topk=16, mode=SEQ),              # one-pass router, packed query cubes, long lists
    dict(heads_q=12, heads_kv=4, dim=64, grid=(21, 30, 52), topk=12, flags=vb.FLAG_GROUP_ROUTING),
    dict(heads_q=3, heads_kv=3, dim=128, grid=(29, 30, 45), topk=9, cube=(4, 4, 8), one_pass=True),
    dict(heads_q=2, heads_kv=2, dim=64, grid=(4, 8, 8), topk=2, hidden=64),
]


@pytest.mark.parametrize("layer", REPLAYED, ids=_name)
def test_a_replayed_graph_gives_what_the_calls_give(layer):
    """A whole pass captured once (the edges between kernels are programmatic there too) and replayed on other inputs."""
    layer = Layer(**layer)
    layer()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = layer()
    for seed in (1, 7, 8):
        for x, y in zip((layer.q, layer.k, layer.v, layer.d_o, layer.gate), layer.inputs(seed)):
            x.copy_(y)
        for x in captured:
            x.zero_()
        graph.replay()
        graph.replay()
        got = [x.clone() for x in captured]
        layer.attn.check_status()
        want = layer()
        torch.cuda.synchronize()
        for i, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), (seed, i)
    if layer.attn.route_scratch_bytes or layer.scratch is not None:
        words = layer.attn.ws_route[:256].view(torch.int32)
        assert int(words[2]) == 0 and int(words[3]) > 0               # (the one-pass form, with pairs to settle)


def test_two_host_threads_on_two_streams():
    """Each thread's kernels are placed beside the other's, some with tensor memory for the whole SM."""
    layers = [Layer(**REPLAYED[0]), Layer(heads_q=4, heads_kv=2, dim=128, grid=(13, 30, 45), topk=9, one_pass=True, seed=2)]
    want = [layer() for layer in layers]
    torch.cuda.synchronize()
    results, errors = [None, None], []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(12):
                    results[i] = layers[i]()
            stream.synchronize()
        except Exception as e:                                          # noqa: BLE001 (handed to the test's thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for layer, got, ref in zip(layers, results, want):
        layer.attn.check_status()
        for x, y in zip(got, ref):
            assert torch.equal(x, y)
