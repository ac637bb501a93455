"""The coarse forward with one group of warps per row block (more row blocks than SMs) and with two (each takes every other tile of 32 keys): the
same heads, all in one call and in calls of a quarter, at numbers of cubes around the tiles' and groups' edges."""
import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("grid,cubes", [((4, 16, 32), 32), ((4, 12, 44), 33), ((4, 16, 64), 64), ((4, 20, 52), 65), ((4, 12, 128), 96), ((4, 4, 388), 97),
                                        ((3, 18, 111), 140)])
def test_two_groups_of_warps_give_what_one_gives(dim, grid, cubes):
    heads, parts = 160, 4
    rows = grid[0] * grid[1] * grid[2]
    gen = torch.Generator(device="cuda").manual_seed(cubes)
    # (cube means of the order of one, so that the weights are not all alike)
    q, k, v = (3 * torch.randn(1, heads, rows, dim, device="cuda", generator=gen).bfloat16() for _ in range(3))
    gate = torch.rand(1, heads, rows, device="cuda", generator=gen)

    def coarse(part):
        n = part.stop - part.start
        p = vb.make_params(1, n, n, dim, grid, select_mode=vb.PER_QUERY, topk=1)
        attn = vb.Vsa2Attention(p)
        assert attn.sizes.n_cubes == cubes
        t = [x[:, part].contiguous() for x in (q, k, v, gate)]
        attn.route(t[0], t[1])
        attn.forward(*t)
        attn.check_status()
        return attn.oc_hat.view(n, cubes, dim).clone(), attn.lse_c.view(n, cubes).clone(), attn.vc.view(n, cubes, dim).clone()

    o, lse, vc = coarse(slice(0, heads))
    step = heads // parts
    for i in range(parts):
        part = slice(i * step, (i + 1) * step)
        o2, lse2, _ = coarse(part)
        # the scores are the same TF32 products; a weight is rounded to TF32 against its group's running maximum: 2^-12 of it either way,
        # once in each form, and the sums' order differs
        bound = 2.0 ** -11 * vc[part].abs().amax(1, keepdim=True) + 1e-6
        assert ((o2 - o[part]).abs() <= bound).all()
        assert (lse2 - lse[part]).abs().max() <= 1e-5
