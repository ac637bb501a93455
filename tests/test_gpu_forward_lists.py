"""The 64-row kernels, forward and backward, on lists of every small length: empty, one block, odd and even, all of them, one after the other, with more items than
SMs (several items per CTA: its double buffers change over, empty items between them) on a grid that cuts cubes in every dimension."""
import numpy as np
import pytest
import torch

from oracle import vsa2_oracle as orc
from paper_2609_32882_b200 import binding as vb
from vsa2_testlib import assert_close, assert_lse_close, csr_to_mask, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("out_dtype", [vb.BF16, vb.F32])
@pytest.mark.parametrize("grid", [(5, 9, 13), (4, 8, 24)])
def test_lists_of_every_small_length(dim, out_dtype, grid):
    torch.manual_seed(dim)
    heads = 24
    tok = grid[0] * grid[1] * grid[2]
    geo = orc.Geometry(grid, (4, 4, 4), (2, 2, 2))
    q, k, v = (torch.randn(1, heads, tok, dim, device="cuda", dtype=torch.bfloat16) for _ in range(3))
    gate = torch.tanh(torch.randn(1, heads, tok, device="cuda"))
    n = geo.N
    lengths = torch.tensor([0, 1, 2, 3, 0, 0, n, 4, 5, 1, 1, 0, 7], dtype=torch.int32, device="cuda")
    budgets = lengths[(torch.arange(heads * n, device="cuda") * 5) % len(lengths)].view(1, heads, n).contiguous()
    p = vb.make_params(1, heads, heads, dim, grid, select_mode=vb.PER_QUERY_BUDGET, out_dtype=out_dtype, nnz_cap=int(budgets.sum(-1).max()))
    attn = vb.Vsa2Attention(p)
    attn.route(q, k, budgets)
    o, lse = attn.forward(q, k, v, gate)
    attn.check_status()
    rp, ci, _, _ = (t.cpu().numpy() for t in attn.map_views())
    mask = csr_to_mask(rp, ci, n)
    want, want_lse = orc.forward(to_f64(q), to_f64(k), to_f64(v), to_f64(gate), mask, geo, 1.0 / np.sqrt(dim))
    assert_close("O", to_f64(o), want, bf16_storage=out_dtype == vb.BF16)
    assert_lse_close(to_f64(lse), want_lse)
    d_o = torch.randn_like(q)
    got = attn.backward(q, k, v, gate, o, lse, d_o)
    attn.check_status()
    ref = orc.backward(to_f64(q), to_f64(k), to_f64(v), to_f64(gate), mask, geo, 1.0 / np.sqrt(dim), to_f64(d_o))
    for name, x, y in zip(("dQ", "dK", "dV", "dgate"), got, ref):
        assert_close(name, to_f64(x), y, bf16_storage=x.dtype == torch.bfloat16)


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("out_dtype", [vb.BF16, vb.F32])
@pytest.mark.parametrize("kind", ["cubes_of_128", "shared_map"])
def test_pairs_of_blocks_on_lists_of_every_small_length(dim, out_dtype, kind):
    """The same for the 128-row forward: cubes of 128 tokens (some of whose second halves are empty), and query heads that share a map."""
    torch.manual_seed(dim)
    wide = kind == "cubes_of_128"
    heads, heads_kv = (24, 24) if wide else (32, 8)
    grid, cube = ((5, 9, 26), (4, 4, 8)) if wide else ((5, 9, 13), (4, 4, 4))
    tok = grid[0] * grid[1] * grid[2]
    geo = orc.Geometry(grid, cube, (2, 2, 2))
    q = torch.randn(1, heads, tok, dim, device="cuda", dtype=torch.bfloat16)
    k, v = (torch.randn(1, heads_kv, tok, dim, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    gate = torch.tanh(torch.randn(1, heads, tok, device="cuda"))
    n = geo.N
    if wide:
        lengths = torch.tensor([0, 1, 2, 3, 0, 0, n, 4, 5, 1, 1, 0, 7], dtype=torch.int32, device="cuda")
        budgets = lengths[(torch.arange(heads * n, device="cuda") * 5) % len(lengths)].view(1, heads, n).contiguous()
        p = vb.make_params(1, heads, heads_kv, dim, grid, cube=cube, select_mode=vb.PER_QUERY_BUDGET, out_dtype=out_dtype,
                           nnz_cap=int(budgets.sum(-1).max()))
    else:                                    # (kept per sequence: lists of any length)
        budgets = None
        p = vb.make_params(1, heads, heads_kv, dim, grid, select_mode=vb.PER_SEQUENCE, topk=3, out_dtype=out_dtype, flags=vb.FLAG_GROUP_ROUTING)
    attn = vb.Vsa2Attention(p)
    attn.route(q, k, budgets)
    o, lse = attn.forward(q, k, v, gate)
    attn.check_status()
    rp, ci, _, _ = (t.cpu().numpy() for t in attn.map_views())
    mask = csr_to_mask(rp, ci, n)
    want, want_lse = orc.forward(to_f64(q), to_f64(k), to_f64(v), to_f64(gate), mask, geo, 1.0 / np.sqrt(dim))
    assert_close("O", to_f64(o), want, bf16_storage=out_dtype == vb.BF16)
    assert_lse_close(to_f64(lse), want_lse)
