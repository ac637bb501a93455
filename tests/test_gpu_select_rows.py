"""Per-query TopK at the row lengths where the kernel takes another form (row held in 8, 20, 32, 48 or 64 registers a lane, or
histograms of a whole block), with and without ties: the map must be exactly the k largest of the block scores the
library computed, ties to the lower column, in both its CSR and its CSC form."""
import numpy as np
import pytest
import torch

from paper_2609_32882_b200 import binding as vb
from vsa2_testlib import csr_to_mask

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 256, 257, 640, 641, 1024, 1025, 1536, 1537, 2048, 2049])
@pytest.mark.parametrize("budget", [False, True])
def test_rows_of_every_register_count(n, budget):
    torch.manual_seed(n)
    k = min(n, 13)
    grid = (4, 4, 4 * n)
    p = vb.make_params(1, 1, 1, 64, grid, select_mode=vb.PER_QUERY_BUDGET if budget else vb.PER_QUERY, topk=0 if budget else k,
                       nnz_cap=n * (n // 2 + 1) if budget else 0)
    attn = vb.Vsa2Attention(p)
    q = torch.randn(1, 1, 16 * 4 * n, 64, device="cuda", dtype=torch.bfloat16)
    kk = torch.randn_like(q)
    if n > 1:
        kk[:, :, : 16 * 4 * n // 2] = 0.0        # equal scores in half of the sub-cube columns: ties in every row
        kk = kk.contiguous()
    budgets = torch.randint(0, n // 2 + 1, (1, 1, n), dtype=torch.int32, device="cuda") if budget else None
    attn.route(q, kk, budgets)
    attn.check_status()
    score = attn.scores()[0, 0].cpu().numpy()
    rp, ci, cp, ri = (t[0, 0].cpu().numpy() for t in attn.map_views())
    got = csr_to_mask(rp, ci, n)
    assert np.array_equal(got, csr_to_mask(cp, ri, n).T)
    take = budgets[0, 0].cpu().numpy() if budget else np.full(n, k)
    order = np.argsort(-score, axis=1, kind="stable")
    want = np.zeros_like(got)
    for i in range(n):
        want[i, order[i, : take[i]]] = True
    assert np.array_equal(got, want)


@pytest.mark.parametrize("n", [32, 33, 64, 65, 127, 128, 129, 160])
@pytest.mark.parametrize("mode", ["row", "budget", "sequence"])
def test_maps_around_the_one_block_form(n, mode):
    """Up to 128 cubes one block per head builds both maps, in words of 32; ties in every row, one head whose scores all tie, and budgets
    that are zero here and everything there."""
    torch.manual_seed(n)
    heads, k = 3, min(n, 7)
    sel = {"row": vb.PER_QUERY, "budget": vb.PER_QUERY_BUDGET, "sequence": vb.PER_SEQUENCE}[mode]
    budgets = None
    if mode == "budget":
        budgets = torch.randint(0, n + 1, (1, heads, n), dtype=torch.int32, device="cuda")
        budgets[0, 0, ::3], budgets[0, 1, ::4] = 0, n
    cap = int(budgets.sum(dim=-1).max()) if mode == "budget" else 0
    p = vb.make_params(1, heads, heads, 64, (4, 4, 4 * n), select_mode=sel, topk=0 if mode == "budget" else k, nnz_cap=cap)
    attn = vb.Vsa2Attention(p)
    q = torch.randn(1, heads, 64 * n, 64, device="cuda", dtype=torch.bfloat16)
    kk = torch.randn_like(q)
    kk[:, :, : 32 * n] = 0.0                       # equal scores in half of the sub-cube columns
    kk[:, 1] = 0.0                                 # and everywhere
    attn.route(q, kk, budgets)
    attn.check_status()
    score = attn.scores()[0].cpu().numpy()
    rp, ci, cp, ri = (t[0].cpu().numpy() for t in attn.map_views())
    for h in range(heads):
        got = csr_to_mask(rp[h], ci[h], n)
        assert np.array_equal(got, csr_to_mask(cp[h], ri[h], n).T)
        want = np.zeros_like(got)
        if mode == "sequence":
            want.reshape(-1)[np.argsort(-score[h].reshape(-1), kind="stable")[: n * k]] = True
        else:
            take = budgets[0, h].cpu().numpy() if mode == "budget" else np.full(n, k)
            order = np.argsort(-score[h], axis=1, kind="stable")
            for i in range(n):
                want[i, order[i, : take[i]]] = True
        assert np.array_equal(got, want), h


@pytest.mark.parametrize("n", [1, 7, 9, 128, 129, 136, 161, 255, 288, 471, 480, 481])
@pytest.mark.parametrize("ties", [False, True])
def test_heads_whose_selection_runs_in_a_cluster(n, ties):
    """Up to 480 cubes, per sequence: eight parts of the rows (the last one shorter, words of 32 columns cut), from two-pass scores, from
    one-pass scores, and with a capacity that the selection exceeds."""
    torch.manual_seed(n)
    heads, k = 3, min(9, n)
    q = torch.randn(1, heads, 64 * n, 64, device="cuda", dtype=torch.bfloat16)
    kk = torch.randn_like(q)
    if ties:
        kk[:, 0, : 32 * n] = 0.0                   # equal scores in half of the columns, at the threshold or not
        q[:, 1] = 0.0                              # a head whose scores all tie: the first n * k entries
    scratch = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    for cap in (0, max(1, n * k - 4 * n - 3)):
        p = vb.make_params(1, heads, heads, 64, (4, 4, 4 * n), select_mode=vb.PER_SEQUENCE, topk=k, nnz_cap=cap)
        attn = vb.Vsa2Attention(p)
        vb.vsa2_route(p, q, kk, None, attn.map, attn.ws_route)
        score = attn.scores()[0].cpu().numpy()
        keep = cap or n * k
        assert vb.vsa2_device_status(attn.ws_route) == (vb.ERR_MAP_OVERFLOW if keep < n * k else vb.OK)
        maps = [t[0].cpu().numpy() for t in attn.map_views()]
        for h in range(heads):
            want = np.zeros((n, n), dtype=bool)
            want.reshape(-1)[np.argsort(-score[h].reshape(-1), kind="stable")[: n * k]] = True
            want.reshape(-1)[np.flatnonzero(want)[keep:]] = False        # entries past the capacity, in row order
            got = csr_to_mask(maps[0][h], maps[1][h], n)
            assert maps[0][h][n] == keep and maps[2][h][n] == keep
            assert np.array_equal(got, want), h
            assert np.array_equal(got, csr_to_mask(maps[2][h], maps[3][h], n).T), h
        one = vb.Vsa2Attention(p)
        vb.vsa2_route(p, q, kk, None, one.map, one.ws_route, scratch=scratch)
        for a, b in zip(maps, one.map_views()):
            assert np.array_equal(a[:, :keep], b[0].cpu().numpy()[:, :keep])


@pytest.mark.parametrize("n", [1, 128, 129, 288, 480])
@pytest.mark.parametrize("ties", [False, True])
def test_selection_without_room_for_clusters(n, ties):
    """Contexts without room for a cluster of eight CTAs take the launches over all heads: the same maps, from two-pass and one-pass scores, and
    within the capacity or not.  (An ordinary context has the room: it needs fewer launches.)"""
    torch.manual_seed(n)
    heads, k = 3, min(9, n)
    q = torch.randn(1, heads, 64 * n, 64, device="cuda", dtype=torch.bfloat16)
    kk = torch.randn_like(q)
    if ties:
        kk[:, 0, : 32 * n] = 0.0
        q[:, 1] = 0.0
    scratch = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    for cap in (0, max(1, n * k - 4 * n - 3)):
        for extra in (None, scratch):
            maps, launches, status = [], [], []
            for flags in (0, vb.FLAG_SELECT_NO_CLUSTERS):
                p = vb.make_params(1, heads, heads, 64, (4, 4, 4 * n), select_mode=vb.PER_SEQUENCE, topk=k, nnz_cap=cap, flags=flags)
                attn = vb.Vsa2Attention(p)
                before = vb.vsa2_launch_count()
                vb.vsa2_route(p, q, kk, None, attn.map, attn.ws_route, scratch=extra)
                launches.append(vb.vsa2_launch_count() - before)
                status.append(vb.vsa2_device_status(attn.ws_route))
                keep = int(attn.map_views()[0].max())
                maps.append([t[..., : keep if i % 2 else None].clone() for i, t in enumerate(attn.map_views())])
            assert launches[0] < launches[1] and status[0] == status[1]
            assert all(torch.equal(a, b) for a, b in zip(*maps))


@pytest.mark.parametrize("n", [40, 128, 129, 300, 1100, 2100])
@pytest.mark.parametrize("one_pass", [False, True])
def test_rows_that_keep_nothing_whatever_their_scores(n, one_pass):
    """Rows with a budget of none stay empty where their scores are not numbers, and leave the other rows' lists alone."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    q, k = (torch.randn(1, 1, 64 * n, 64, device="cuda", generator=gen).bfloat16() for _ in range(2))
    none = torch.rand(n, device="cuda", generator=gen) < 0.3
    none[:2] = torch.tensor([True, False], device="cuda")
    budgets = torch.randint(1, 9, (1, 1, n), device="cuda", generator=gen, dtype=torch.int32)
    budgets[0, 0, none] = 0
    cap = int(budgets.sum())
    p = vb.make_params(1, 1, 1, 64, (4, 4, 4 * n), select_mode=vb.PER_QUERY_BUDGET, nnz_cap=cap)
    scratch = torch.empty(1 << 29, dtype=torch.uint8, device="cuda") if one_pass else None
    maps = []
    for value in (None, float("nan")):
        if value is not None:
            q.view(4, 4, n, 4, 64)[:, :, none] = value
        attn = vb.Vsa2Attention(p)
        vb.vsa2_route(p, q, k, budgets, attn.map, attn.ws_route, scratch=scratch)
        assert vb.vsa2_device_status(attn.ws_route) == vb.OK
        maps.append([t.clone() for t in attn.map_views()])
    assert int(maps[0][0][0, 0, n]) == cap and int(maps[0][2][0, 0, n]) == cap
    assert all(torch.equal(a, b) for a, b in zip(*maps))
