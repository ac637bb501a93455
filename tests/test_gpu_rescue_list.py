"""Forward calls in which every query block leaves the safe range of the fixed-reference softmax: each block is handed to the exact kernel once, also
where a CTA has a hundred of them one after the other and its epilogue warps are at different ones."""
import math

import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("kind", ["cubes_of_64", "cubes_of_128", "shared_map"])
def test_every_block_is_listed_once(dim, kind):
    wide = kind == "cubes_of_128"
    heads, grid, cube = 600, (4, 4, 96 if wide else 100), (4, 4, 8 if wide else 4)
    heads_kv = 150 if kind == "shared_map" else heads
    rows, last = grid[0] * grid[1] * grid[2], grid[2] // cube[2] - 1
    # A key scores 100 nats more than one of the cube before it, so the first tile's maximum says nothing about the last cube
    step = 100 / (math.sqrt(dim) * 4)
    k = (torch.arange(grid[2], device="cuda") // cube[2] * step).bfloat16().view(1, 1, 1, grid[2], 1)
    k = k.expand(1, heads_kv, 16, grid[2], dim).reshape(1, heads_kv, rows, dim).contiguous()
    q = torch.full((1, heads, rows, dim), 4.0, device="cuda", dtype=torch.bfloat16)
    v = torch.randn(1, heads_kv, rows, dim, device="cuda", dtype=torch.bfloat16)
    p = vb.make_params(1, heads, heads_kv, dim, grid, cube=cube, select_mode=vb.PER_QUERY, topk=3, out_dtype=vb.F32,
                       flags=vb.FLAG_NO_COARSE | (vb.FLAG_GROUP_ROUTING if kind == "shared_map" else 0))
    attn = vb.Vsa2Attention(p)
    attn.route(q, k)
    lists = attn.map_views()[1][0].view(heads, last + 1, 3)
    assert (lists[:, :, 0] == 0).all() and (lists[:, :, 2] == last).all()      # (the others' scores are 0: the lowest come first)
    blocks = heads * rows // 64
    for _ in range(3):
        o, lse = attn.forward(q, k, v, None)
        assert int(attn.ws_fwd[8:12].view(torch.int32).item()) == blocks <= 16384
        attn.check_status()
        # every row is the mean of the last cube's values (weights of 2^-6 or 2^-7, which 16 bits hold)
        want = v.view(heads_kv, 16, grid[2], dim)[:, :, last * cube[2]:].double().flatten(1, 2)
        top = 4.0 * math.sqrt(dim) * k[0, 0, -1, 0].double().item()
        assert (o.view(heads, rows, dim) - want.mean(1).repeat_interleave(heads // heads_kv, 0)[:, None]).abs().max() <= 1e-5
        assert (lse - (top + math.log(want.shape[1]))).abs().max() <= 1e-3
