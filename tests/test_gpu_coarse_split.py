"""The coarse forward does not depend on who shares the call: a head alone, with others, or in a batch gives the same bits (calls with more row
blocks than SMs and with fewer are placed differently), at numbers of cubes around the edges of its tiles of 32 keys and 64 rows."""
import math

import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


def _coarse(grid, q, k, v, gate):
    """(oc_hat, lse_c, O) of a call, each [heads of all batches, ...]"""
    batch, heads, _, dim = q.shape
    p = vb.make_params(batch, heads, heads, dim, grid, select_mode=vb.PER_QUERY, topk=1)
    attn = vb.Vsa2Attention(p)
    q, k, v, gate = (x.contiguous() for x in (q, k, v, gate))
    attn.route(q, k)
    o, _ = attn.forward(q, k, v, gate)
    attn.check_status()
    n = attn.sizes.n_cubes
    return attn.oc_hat.view(batch * heads, n, dim).clone(), attn.lse_c.view(batch * heads, n).clone(), o.flatten(0, 1)


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("grid,cubes", [((4, 16, 32), 32), ((4, 12, 44), 33), ((4, 16, 64), 64), ((4, 20, 52), 65), ((4, 12, 128), 96), ((4, 4, 388), 97),
                                        ((3, 18, 111), 140)])
def test_a_head_is_the_same_whatever_shares_its_call(dim, grid, cubes):
    heads, parts = 160, 4
    rows = grid[0] * grid[1] * grid[2]
    gen = torch.Generator(device="cuda").manual_seed(cubes)
    # (cube means of the order of one, so that the weights are not all alike)
    x = [3 * torch.randn(1, heads, rows, dim, device="cuda", generator=gen).bfloat16() for _ in range(3)]
    x.append(torch.rand(1, heads, rows, device="cuda", generator=gen))
    want = _coarse(grid, *x)
    assert want[0].shape[1] == cubes
    step = heads // parts
    for i in range(parts):
        part = slice(i * step, (i + 1) * step)
        for a, b in zip(_coarse(grid, *(t[:, part] for t in x)), want):
            assert torch.equal(a, b[part])
    for a, b in zip(_coarse(grid, *(t[:, :step].unflatten(1, (2, step // 2)).squeeze(0) for t in x)), want):      # as a batch of two
        assert torch.equal(a, b[:step])


@pytest.mark.parametrize("dim", [64, 128])
def test_a_tile_of_keys_without_weight(dim):
    """A run of 32 cubes whose means lie below the range of fp32 (every score -infinity) takes no weight."""
    cubes, grid = 97, (4, 4, 388)
    gen = torch.Generator(device="cuda").manual_seed(dim)
    q, k, v = (torch.randn(1, 1, 64 * cubes, dim, device="cuda", generator=gen).bfloat16() for _ in range(3))
    q = q.abs() + 0.5
    # tokens run through the rows of the grid: those of cubes 32 .. 63 have w in [128, 256)
    k.view(4, 4, 388, dim)[:, :, 128:256] = -3e38
    gate = torch.ones(1, 1, 64 * cubes, device="cuda")
    p = vb.make_params(1, 1, 1, dim, grid, select_mode=vb.PER_QUERY, topk=1)
    attn = vb.Vsa2Attention(p)
    attn.route(q, k)
    attn.forward(q, k, v, gate)
    attn.check_status()
    qc, kc, vc = (t.view(cubes, dim).double() for t in (attn.qc, attn.kc, attn.vc))
    assert torch.isinf(kc[32:64]).all() and torch.isfinite(kc[:32]).all() and torch.isfinite(kc[64:]).all()
    keep = torch.ones(cubes, dtype=torch.bool, device="cuda")
    keep[32:64] = False
    s = qc @ kc[keep].T / math.sqrt(dim)
    got = attn.oc_hat.view(cubes, dim).double()
    # TF32 operands, 2^-11 each: of a score |s| <= |q_c| |k_c| / sqrt(D), of a weight and of a value
    bound = 2.0 ** -11 * (2 + 2 * (qc.norm(dim=1).max() * kc[keep].norm(dim=1).max()).item() / math.sqrt(dim)) * vc.abs().max()
    assert torch.isfinite(got).all()
    assert (got - torch.softmax(s, -1) @ vc[keep]).abs().max() <= bound
