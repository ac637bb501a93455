"""What a Vsa2Attention handle holds, and the scratch its backward takes for a call: a model keeps a handle per layer, so a handle holds
its maps, saved state and least workspaces, and the scratch of up to 7 GiB goes back after every call."""
import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


def make(seed, heads_q=4, heads_kv=2, grid=(8, 16, 16), topk=9):
    attn = vb.Vsa2Attention(vb.make_params(1, heads_q, heads_kv, 128, grid, select_mode=vb.PER_QUERY, topk=topk))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rows = grid[0] * grid[1] * grid[2]
    rnd = lambda h: torch.randn(1, h, rows, 128, device="cuda", generator=gen).bfloat16()
    return attn, (rnd(heads_q), rnd(heads_kv), rnd(heads_kv), torch.rand(1, heads_q, rows, device="cuda", generator=gen)), rnd(heads_q)


def passes(attn, qkvg, d_o, stream=None):
    q, k, v, gate = qkvg
    attn.route(q, k, stream=stream)
    o, lse = attn.forward(q, k, v, gate, stream=stream)
    return attn.backward(q, k, v, gate, o, lse, d_o, stream=stream)


def test_handles_hold_no_scratch():
    torch.cuda.empty_cache()
    p = vb.make_params(1, 12, 3, 128, (21, 30, 52), select_mode=vb.PER_QUERY, topk=78)      # 480p, grouped heads
    assert vb.vsa2_attn_bwd_scratch_bytes(p) > 4 << 30
    before = torch.cuda.memory_allocated()
    attn = vb.Vsa2Attention(p)
    s = attn.sizes
    held = torch.cuda.memory_allocated() - before
    state = 2 * 4 * (s.ptr_elems + s.idx_elems) + 4 * (2 * s.pooled_q_elems + 2 * s.pooled_kv_elems) + 4 * s.lse_c_elems + 2 * s.o_res_elems
    least = s.route_workspace_bytes + s.fwd_workspace_bytes + s.bwd_workspace_bytes
    assert held <= state + least + (8 << 20)                # (torch rounds its allocations up)


def test_scratch_is_given_back_and_done_without_when_there_is_no_room():
    attn, qkvg, d_o = make(5)
    want = passes(attn, qkvg, d_o)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    got = passes(attn, qkvg, d_o)
    assert attn.bwd_scratch_bytes > 1 << 20

    assert torch.cuda.memory_allocated() - before <= sum(t.numel() * t.element_size() for t in got) + 16 * 512
    attn.bwd_scratch_bytes = 1 << 50                         # more than any GPU has
    less = passes(attn, qkvg, d_o)
    assert attn.bwd_scratch_bytes == 0
    attn.check_status()
    for a, b, c in zip(want, got, less):
        assert torch.equal(a, b) and torch.equal(a, c)


def test_routes_without_scratch_when_there_is_no_room():
    attn, qkvg, _ = make(6, heads_q=9, heads_kv=9, grid=(21, 30, 52), topk=16)
    assert attn.route_scratch_bytes > 1 << 20
    attn.route(*qkvg[:2])
    want, scores = [x.clone() for x in attn.map_views()], attn.scores()
    attn.route_scratch_bytes = 1 << 50                       # more than any GPU has
    attn.route(*qkvg[:2])
    attn.check_status()
    assert attn.route_scratch_bytes == 0 and not torch.equal(attn.scores(), scores)
    for x, y in zip(want, attn.map_views()):
        assert torch.equal(x, y)


def test_handles_on_two_streams_and_in_a_graph():
    """Two handles whose backwards overlap on two streams (one given as a torch stream, one as its handle), and one whose passes
    are captured and replayed while the other runs."""
    (a1, x1, d1), (a2, x2, d2) = make(1), make(2, heads_q=2, heads_kv=2, grid=(12, 16, 20), topk=11)
    want1, want2 = passes(a1, x1, d1), passes(a2, x2, d2)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(5):
        with torch.cuda.stream(s1):
            got1 = passes(a1, x1, d1, stream=s1)
        with torch.cuda.stream(s2):
            got2 = passes(a2, x2, d2, stream=s2.cuda_stream)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want1 + want2, got1 + got2))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = passes(a1, x1, d1)
    for t in out:
        t.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        graph.replay()
    with torch.cuda.stream(s2):
        got2 = passes(a2, x2, d2)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want1 + want2, out + got2))
    del graph
