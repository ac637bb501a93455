"""Backward on grids whose last layer of cubes is cut to one or two frames: with scratch the dK/dV pass packs four or two such query
cubes into a tile (and dQ reads only their rows of the stored dS), without it nothing is packed.  Sixteen rows are one step of a
product's contraction and their order stays, so the gradients are the same bit for bit.  Out of range both end in the same forms."""
import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu
SEQ, ROW, BUDGET = vb.PER_SEQUENCE, vb.PER_QUERY, vb.PER_QUERY_BUDGET


@pytest.mark.parametrize("factor", [1.0, 2.5e5])
@pytest.mark.parametrize("batch,heads_q,heads_kv,dim,grid,topk,mode,text", [
    (1, 2, 2, 64, (5, 32, 64), 7, ROW, 0),             # one frame: four cubes a tile
    (1, 3, 3, 128, (9, 30, 45), 9, SEQ, 0),            # cubes cut along the other edges too, lists of any length
    (2, 2, 2, 128, (5, 29, 47), 5, ROW, 77),           # text blocks behind the packed cubes, the last one ragged
    (1, 4, 2, 128, (5, 32, 64), 9, ROW, 0),            # grouped heads, fp16 form
    (1, 6, 2, 64, (6, 30, 61), 3, SEQ, 130),           # grouped heads, pair form; two frames: two cubes a tile; text
    (1, 8, 2, 128, (9, 24, 40), 0, BUDGET, 0),
    (1, 2, 2, 64, (6, 32, 64), 150, ROW, 0),           # long lists
    (1, 2, 2, 128, (7, 32, 64), 6, ROW, 0),            # three frames: nothing to pack
])
def test_gradients_of_packed_query_cubes(batch, heads_q, heads_kv, dim, grid, topk, mode, text, factor):
    rows = grid[0] * grid[1] * grid[2]
    gen = torch.Generator(device="cuda").manual_seed(12)
    budgets, cap = None, 0
    if mode == BUDGET:
        n = -(-grid[0] // 4) * -(-grid[1] // 4) * -(-grid[2] // 4)
        budgets = torch.randint(0, 30, (batch, heads_q, n), device="cuda", generator=gen, dtype=torch.int32)
        cap = int(budgets.sum(-1).max())
    p = vb.make_params(batch, heads_q, heads_kv, dim, grid, select_mode=mode, topk=topk, text_len=text, nnz_cap=cap, out_dtype=vb.F32)
    attn = vb.Vsa2Attention(p)
    rnd = lambda h: torch.randn(batch, h, rows + text, dim, device="cuda", generator=gen).bfloat16()
    q, k, v, d_o = rnd(heads_q), rnd(heads_kv), rnd(heads_kv), rnd(heads_q).float()
    d_o[-1, -1] *= factor
    d_o = d_o.bfloat16()
    gate = torch.rand(batch, heads_q, rows, device="cuda", generator=gen)
    attn.route(q, k, budgets)
    o, lse = attn.forward(q, k, v, gate)
    assert attn.bwd_scratch_bytes > 0
    got = attn.backward(q, k, v, gate, o, lse, d_o)
    attn.check_status()
    attn.bwd_scratch_bytes, attn.ws_bwd = 0, torch.empty(attn.sizes.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
    want = attn.backward(q, k, v, gate, o, lse, d_o)
    attn.check_status()
    for name, x, y in zip(("dq", "dk", "dv", "dgate"), got, want):
        assert torch.isfinite(x).all(), name
        # (grouped heads with fp16 passes: dQ's dP comes from the fp16 copies with stored tiles, 2^-25 off where V is below 2^-17)
        assert torch.equal(x, y) or (heads_q != heads_kv and name == "dq" and (x - y).norm() <= 1e-6 * y.norm()), name
