"""Cube and sub-cube means of 64-token cubes of every shape that 2 x 2 x 2 sub-cubes fill, on grids that cut them in each dimension by an odd and an even
number of tokens: the cube means, and the block scores as what the sub-cubes' means lead to."""
import numpy as np
import pytest
import torch

from oracle import vsa2_oracle as orc
from paper_2609_32882_b200 import binding as vb
from vsa2_testlib import to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("cube", [(4, 4, 4), (2, 2, 16), (2, 16, 2), (16, 2, 2), (2, 4, 8), (8, 2, 4), (4, 8, 2)])
@pytest.mark.parametrize("cut", [(1, 2, 1), (2, 1, 0), (0, 1, 2)])
def test_means_of_cut_cubes(dim, cube, cut):
    grid = tuple(2 * c - x for c, x in zip(cube, cut))
    geo = orc.Geometry(grid, cube, (2, 2, 2))
    rows = grid[0] * grid[1] * grid[2]
    gen = torch.Generator(device="cuda").manual_seed(dim)
    q, k, v = (torch.randn(1, 2, rows, dim, device="cuda", generator=gen).bfloat16() for _ in range(3))
    p = vb.make_params(1, 2, 2, dim, grid, cube=cube, select_mode=vb.PER_QUERY, topk=2)
    attn = vb.Vsa2Attention(p)
    attn.route(q, k)
    scores = to_f64(attn.scores())
    attn.forward(q, k, v, torch.ones(1, 2, rows, device="cuda"))
    attn.check_status()
    for x, got in ((q, attn.qc), (k, attn.kc), (v, attn.vc)):
        want = np.stack([orc.mean_pool_cube(to_f64(x)[0, h], geo) for h in range(2)])
        # 64 terms of at most 4.5 in fp32: 6 roundings on a path, each of a partial sum
        assert np.abs(to_f64(got).reshape(want.shape) - want).max() <= 6 * 2.0 ** -24 * 4.5
    _, want = orc.route(to_f64(q), to_f64(k), geo, 1 / np.sqrt(dim), vb.PER_QUERY, 2, return_scores=True)
    # (scores as in the router's own test: 2e-4 for |s| <= 60; a mean that is one bf16 step off would show at 2^-9)
    assert (np.abs(scores - want) <= 2e-4 * np.abs(want) + 1e-30).all()
