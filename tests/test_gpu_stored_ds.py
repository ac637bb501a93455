"""Backward with room for the stored score-gradient tiles of all KV groups, of some, and of none: the routes form
dQ from the same fp16 tiles and cubes in the same order, so the gradients must be the same bit for bit (the parity tests compare
the first with the oracle, through the scratch that a handle takes for the call)."""
import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads_q,heads_kv,dim,grid,topk,mode,text", [
    (2, 2, 64, (4, 8, 8), 2, vb.PER_QUERY, 0),
    (3, 3, 128, (5, 9, 13), 5, vb.PER_SEQUENCE, 0),          # ragged cubes, lists of any length, odd ones too
    (4, 2, 128, (8, 16, 16), 9, vb.PER_QUERY, 0),            # grouped heads, fp16 form
    (4, 2, 128, (8, 16, 16), 3, vb.PER_QUERY, 0),            # grouped heads, short lists: pair form
    (2, 2, 128, (8, 12, 16), 4, vb.PER_SEQUENCE, 77),        # text blocks, the last one ragged
    (8, 8, 64, (16, 20, 20), 3, vb.PER_SEQUENCE, 0),         # enough items for the pass to be drawn in order of length
])
def test_gradients_do_not_depend_on_the_scratch(heads_q, heads_kv, dim, grid, topk, mode, text):
    p = vb.make_params(1, heads_q, heads_kv, dim, grid, select_mode=mode, topk=topk, text_len=text)
    attn = vb.Vsa2Attention(p)
    gen = torch.Generator(device="cuda").manual_seed(7)
    rows = grid[0] * grid[1] * grid[2] + text
    rnd = lambda h: torch.randn(1, h, rows, dim, device="cuda", generator=gen).bfloat16()
    q, k, v, d_o = rnd(heads_q), rnd(heads_kv), rnd(heads_kv), rnd(heads_q)
    gate = torch.rand(1, heads_q, rows - text, device="cuda", generator=gen)
    attn.route(q, k)
    o, lse = attn.forward(q, k, v, gate)
    most, least = vb.vsa2_attn_bwd_preferred_workspace_bytes(p), attn.sizes.bwd_workspace_bytes
    assert most > least
    assert most - least - vb.vsa2_attn_bwd_scratch_bytes(p) in range(256)
    got = [attn.backward(q, k, v, gate, o, lse, d_o)]
    attn.check_status()
    attn.bwd_scratch_bytes = 0
    for size in (most, most - 256, least):
        attn.ws_bwd = torch.empty(size, dtype=torch.uint8, device="cuda")
        got.append(attn.backward(q, k, v, gate, o, lse, d_o))
        attn.check_status()
    for other in got[1:]:
        for name, x, y in zip(("dq", "dk", "dv", "dgate"), got[0], other):
            assert torch.equal(x, y), name


def test_a_score_gradient_at_the_fp16_limit_leaves_no_infinity_behind():
    """GQA groups, every product on fp16 copies: dS = P (dP - delta) with P = 1 and delta = 0 (q, o and lse are zero) lies at 65519.99
    with the bf16 tensors (fp16: 65504) and at 65520.01 with the copies, whose V elements of 1.0078 * 2^-25 have become 2^-24
    (fp16: infinite).  Whichever pass meets which, dK (dS times q = 0) must come out as zero, not as 0 times infinity."""
    heads_q, heads_kv, dim, grid = 4, 2, 64, (8, 8, 8)
    p = vb.make_params(1, heads_q, heads_kv, dim, grid, select_mode=vb.PER_QUERY, topk=8, flags=vb.FLAG_NO_COARSE, out_dtype=vb.F32)
    attn = vb.Vsa2Attention(p)
    rows = grid[0] * grid[1] * grid[2]
    q = torch.zeros(1, heads_q, rows, dim, device="cuda", dtype=torch.bfloat16)
    k = torch.ones(1, heads_kv, rows, dim, device="cuda", dtype=torch.bfloat16)
    v_row, do_row = torch.zeros(dim), torch.zeros(dim)
    v_row[:32], do_row[:32] = 1.0078125 * 2.0 ** -25, 2.0 ** 14             # 0.0158 in bf16, 0.0313 as copies, summed first
    v_row[32:46], do_row[32:46] = 1.0, 4096.0                                # 57344
    v_row[46], do_row[46] = 1.9921875, 4096.0                                # 8160
    v_row[47], do_row[47] = 1.0, 16.0
    v_row[48], do_row[48] = 1.0, -3 * 2.0 ** -7                              # 65519.977 in all
    v = v_row.expand(1, heads_kv, rows, dim).bfloat16().cuda().contiguous()
    d_o = do_row.expand(1, heads_q, rows, dim).bfloat16().cuda().contiguous()
    attn.route(q, k)
    o = torch.zeros(1, heads_q, rows, dim, device="cuda")
    lse = torch.zeros(1, heads_q, rows, device="cuda")
    for size in (vb.vsa2_attn_bwd_preferred_workspace_bytes(p), attn.sizes.bwd_workspace_bytes):
        attn.ws_bwd, attn.bwd_scratch_bytes = torch.zeros(size, dtype=torch.uint8, device="cuda"), 0
        dq, dk, dv, _ = attn.backward(q, k, v, None, o, lse, d_o)
        attn.check_status()
        assert (dk == 0).all()
        assert torch.isfinite(dq).all() and torch.isfinite(dv).all()
        assert ((dq / (rows * 65520.0 / dim ** 0.5) - 1).abs() < 2.0 ** -10).all()


@pytest.mark.parametrize("route", ["one_chunk", "group_by_group", "recomputed"])
@pytest.mark.parametrize("where", ["everywhere", "last_head"])
@pytest.mark.parametrize("batch,heads_q,heads_kv,dim,grid,topk,mode,factor", [
    (2, 3, 3, 128, (5, 9, 13), 5, vb.PER_SEQUENCE, 2.5e5),
    (2, 4, 2, 64, (8, 12, 12), 9, vb.PER_QUERY, 4e5),        # grouped heads: the fallback of dK/dV carries pairs for every list
    (2, 4, 2, 64, (8, 12, 12), 9, vb.PER_QUERY, 1e8),        # so large that the flag is up before the first pass
    (1, 2, 2, 64, (20, 32, 32), 256, vb.PER_QUERY, 3e6),     # lists on both sides of 256 entries: the fallback's two launches
])
def test_range_fallback_of_every_route(batch, heads_q, heads_kv, dim, grid, topk, mode, factor, where, route):
    """Score gradients beyond the fp16 range everywhere, or in the last head alone (with a chunk per KV group only the last chunk
    notices, when the others are through): all passes are redone by the forms that VSA2_FLAG_PRECISE_BWD and VSA2_FLAG_FAST_BWD run
    directly, bit for bit."""
    gen = torch.Generator(device="cuda").manual_seed(11)
    rows = grid[0] * grid[1] * grid[2]
    rnd = lambda h: torch.randn(batch, h, rows, dim, device="cuda", generator=gen).bfloat16()
    q, k, v, d_o = rnd(heads_q), rnd(heads_kv), rnd(heads_kv), rnd(heads_q).float()
    d_o[(slice(None), slice(None)) if where == "everywhere" else (-1, -1)] *= factor
    d_o = d_o.bfloat16()
    gate = torch.rand(batch, heads_q, rows, device="cuda", generator=gen)

    def run(flags, scratch=None):
        attn = vb.Vsa2Attention(vb.make_params(batch, heads_q, heads_kv, dim, grid, select_mode=mode, topk=topk, flags=flags, out_dtype=vb.F32))
        if scratch is not None:
            attn.bwd_scratch_bytes = scratch(attn)
        attn.route(q, k)
        o, lse = attn.forward(q, k, v, gate)
        out = attn.backward(q, k, v, gate, o, lse, d_o)
        attn.check_status()
        return attn, out

    def one_group(attn):
        # the whole, less all groups' tiles but one
        tiles = heads_q // heads_kv * attn.sizes.nnz_cap * 64 * 64 * 2
        return attn.bwd_scratch_bytes - (batch * heads_kv - 1) * tiles

    attn, got = run(0, {"one_chunk": None, "group_by_group": one_group, "recomputed": lambda a: 0}[route])
    _, pair = run(vb.FLAG_PRECISE_BWD)
    assert all(torch.isfinite(t).all() for t in got)
    assert torch.equal(got[0], pair[0]) and torch.equal(got[3], pair[3])
    if heads_q != heads_kv:
        assert torch.equal(got[1], pair[1]) and torch.equal(got[2], pair[2])
        return
    _, fast = run(vb.FLAG_FAST_BWD)
    col_ptr = attn.map_views()[2]
    long = ((col_ptr[..., 1:] - col_ptr[..., :-1]) > 256)                     # [B, H, N]
    if topk == 256:
        assert long.any() and not long.all()
    # cube of every token: grids of whole cubes along each edge where lists can be long
    t, h, w = (torch.arange(n, device="cuda") // 4 for n in grid)
    n_h, n_w = -(-grid[1] // 4), -(-grid[2] // 4)
    cube = ((t[:, None, None] * n_h + h[None, :, None]) * n_w + w[None, None, :]).reshape(-1)
    is_long = long[:, :, cube][..., None]
    for i in (1, 2):
        assert torch.equal(got[i], torch.where(is_long, pair[i], fast[i]))


@pytest.mark.parametrize("factor", [1.0, 2.5e5, 1e8])        # in range; found by the dQ pass; found before the first pass
@pytest.mark.parametrize("heads,dim,grid,topk,mode", [
    (2, 64, (4, 8, 16), 2, vb.PER_QUERY),
    (3, 128, (5, 9, 9), 3, vb.PER_SEQUENCE),         # ragged cubes, trailing half-cubes without a token, lists of any length
    (8, 64, (16, 20, 40), 3, vb.PER_SEQUENCE),       # enough items for the pass to be drawn in order of length
    (2, 128, (8, 16, 32), 11, vb.PER_QUERY),
])
def test_gradients_of_128_token_cubes_do_not_depend_on_the_scratch(heads, dim, grid, topk, mode, factor):
    """The same on 128 x 128 tiles: dQ from stored tiles (one chunk, a head at a time) against the pass that recomputes them; out of
    range both end in the forms without fp16."""
    p = vb.make_params(1, heads, heads, dim, grid, cube=(4, 4, 8), select_mode=mode, topk=topk)
    attn = vb.Vsa2Attention(p)
    gen = torch.Generator(device="cuda").manual_seed(7)
    rows = grid[0] * grid[1] * grid[2]
    rnd = lambda: torch.randn(1, heads, rows, dim, device="cuda", generator=gen).bfloat16()
    q, k, v, d_o = rnd(), rnd(), rnd(), rnd().float()
    d_o[:, -1] *= factor                             # (the last head alone: a head at a time, only the last chunk meets it)
    d_o = d_o.bfloat16()
    gate = torch.rand(1, heads, rows, device="cuda", generator=gen)
    attn.route(q, k)
    o, lse = attn.forward(q, k, v, gate)
    all_heads, least = vb.vsa2_attn_bwd_scratch_bytes(p), attn.sizes.bwd_workspace_bytes
    one_head = all_heads - (heads - 1) * attn.sizes.nnz_cap * 128 * 128 * 2
    attn.bwd_scratch_bytes, attn.ws_bwd = 0, torch.empty(least, dtype=torch.uint8, device="cuda")
    got = [attn.backward(q, k, v, gate, o, lse, d_o)]
    for size in (all_heads, one_head):
        attn.bwd_scratch_bytes = size
        got.append(attn.backward(q, k, v, gate, o, lse, d_o))
        attn.check_status()
    for other in got[1:]:
        for name, x, y in zip(("dq", "dk", "dv", "dgate"), got[0], other):
            assert torch.isfinite(x.float()).all() and torch.equal(x, y), name
