"""The router that forms every exponential once (with scratch) against the one that forms them twice (without): the same maps bit
for bit, the same scores but for their last bits, and at the thresholds the very scores -- for every way to select, shared maps,
cubes of 128 tokens, grids that are ragged in every dimension, and inputs on which the one-pass form stands back (ties by the
thousand, scores that climb beyond the range of a parked sum, thresholds next to zero)."""
import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu
SEQ, ROW, BUDGET = vb.PER_SEQUENCE, vb.PER_QUERY, vb.PER_QUERY_BUDGET
WIDE = dict(cube=(4, 4, 8))

# heads_q, heads_kv, D, grid, cube, mode, topk, flags, kind of input
CASES = [
    (2, 1, 64, (4, 8, 8), {}, SEQ, 2, 0, "random"),                              # one tile, one block builds the map
    (3, 3, 128, (9, 30, 45), {}, SEQ, 16, 0, "random"),                          # 288 cubes, ragged
    (12, 4, 64, (13, 27, 47), {}, ROW, 24, 0, "random"),
    (4, 2, 128, (21, 30, 52), {}, BUDGET, 0, 0, "random"),
    (12, 3, 128, (13, 30, 33), {}, ROW, 9, vb.FLAG_GROUP_ROUTING, "random"),     # scores summed over the heads of a group
    (4, 2, 128, (21, 30, 52), {}, SEQ, 40, vb.FLAG_GROUP_ROUTING, "random"),
    (3, 3, 128, (20, 18, 68), WIDE, SEQ, 12, 0, "random"),                       # trailing half-cubes without a token
    (2, 1, 64, (24, 44, 88), WIDE, ROW, 30, 0, "random"),
    (1, 1, 64, (40, 60, 60), {}, ROW, 100, 0, "random"),                         # rows of more than 2048 entries
    (2, 2, 64, (16, 32, 32), {}, SEQ, 10, 0, "constant"),                        # every score ties
    (2, 2, 64, (16, 32, 32), {}, ROW, 10, 0, "constant"),
    (2, 2, 64, (16, 32, 32), {}, ROW, 7, 0, "halves"),                           # ties by the row, some at the threshold
    (2, 2, 64, (28, 28, 28), {}, SEQ, 20, 0, "growing"),
    (2, 2, 128, (28, 28, 32), WIDE, ROW, 20, 0, "growing"),
    (2, 2, 64, (16, 32, 32), {}, SEQ, 200, 0, "peaked"),                         # thresholds below 2^-60
    (2, 2, 64, (16, 32, 32), {}, ROW, 256, 0, "random"),                         # everything is kept
    (2, 1, 128, (8, 32, 32), {}, SEQ, 7, 0, "random"),                           # eight tiles, one block builds the map of what was settled
    (3, 3, 64, (8, 32, 32), {}, ROW, 9, 0, "random"),
    (2, 2, 128, (16, 16, 64), WIDE, SEQ, 11, 0, "random"),                       # the same with cubes of 128 tokens
    (2, 2, 64, (16, 32, 32), {}, ROW, 7, 0, "few"),                              # ties by the row, few enough to be settled
    (2, 2, 64, (16, 32, 32), {}, SEQ, 10, 0, "region"),                          # 4096 ties at the threshold
    (2, 2, 64, (16, 32, 32), {}, ROW, 10, 0, "region"),
]


def _inputs(heads_q, heads_kv, dim, grid, kind):
    gen = torch.Generator(device="cuda").manual_seed(5)
    rows = grid[0] * grid[1] * grid[2]
    q = torch.randn(1, heads_q, rows, dim, device="cuda", generator=gen)
    k = torch.randn(1, heads_kv, rows, dim, device="cuda", generator=gen)
    if kind == "random":
        return (2.0 * q).bfloat16(), (2.0 * k).bfloat16()
    if kind == "constant":
        k = torch.ones_like(k)
    elif kind == "halves":       # the second half of the frames repeats the first
        half = rows // 2
        k[:, :, half:] = k[:, :, :half]
        q, k = 2.0 * q, 2.0 * k
    elif kind == "growing":      # scores climb by 60 nats from the first frame to the last
        t = torch.arange(rows, device="cuda") // (grid[1] * grid[2]) / (grid[0] - 1)
        q[..., 0] = 4.0
        k[..., 0] = (60.0 * dim ** 0.5 / 4.0 * t)[None, None, :]
    elif kind == "few":          # an eighth of the cubes repeat others
        v = k.view(1, heads_kv, *grid, dim)
        v[:, :, 12:, :16] = v[:, :, :4, :16]
        q, k = 2.0 * q, 2.0 * k
    elif kind == "region":       # a quarter of the rows without content
        for x in (q, k):
            x.view(1, -1, *grid, dim)[:, :, :, :grid[1] // 4] = 1.0
    elif kind == "peaked":
        q, k = 24.0 * q, 24.0 * k
    return q.bfloat16(), k.bfloat16()


def _state(attn):
    """(flag that sends a call back to the two-pass form, pairs settled on two-pass scores) of the last route call."""
    words = attn.ws_route[:256].view(torch.int32)
    return int(words[2]), int(words[3])


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}x{c[1]}_d{c[2]}_{'x'.join(map(str, c[3]))}_mode{c[5]}_{c[8]}_{c[7]}")
def test_one_pass_maps_are_the_two_pass_maps(case):
    heads_q, heads_kv, dim, grid, cube, mode, topk, flags, kind = case
    n = -(-grid[0] // 4) * -(-grid[1] // 4) * -(-grid[2] // (8 if cube else 4))
    gen = torch.Generator(device="cuda").manual_seed(6)
    budgets = torch.randint(0, 120, (1, heads_q, n), device="cuda", generator=gen, dtype=torch.int32) if mode == BUDGET else None
    cap = int(budgets.clamp(max=n).sum(-1).max()) if mode == BUDGET else 0
    p = vb.make_params(1, heads_q, heads_kv, dim, grid, select_mode=mode, topk=topk, flags=flags, nnz_cap=cap, **cube)
    q, k = _inputs(heads_q, heads_kv, dim, grid, kind)
    attn = vb.Vsa2Attention(p)
    sub = 8 * n * (2 if cube else 1)
    tiles = -(-sub // 128)
    scratch = torch.empty(148 * tiles * 8192 + heads_q * (4 * sub + 4 * n) + (1 << 20) + 4096, dtype=torch.uint8, device="cuda")
    scratch.fill_(0xff)                                          # (NaN wherever something is read before it is written)
    out = []
    for s in (None, scratch):
        vb.vsa2_route(p, q, k, budgets, attn.map, attn.ws_route, scratch=s)
        attn.check_status()
        views = attn.map_views()
        nnz = int(views[0][..., -1].max())
        out.append(([views[0].clone(), views[1][..., :nnz].clone(), views[2].clone(), views[3][..., :nnz].clone()], attn.scores()))
    (two_map, two), (one_map, one) = out
    redo, pairs = _state(attn)
    if tiles < 8:
        assert torch.equal(one, two)
    elif kind in ("growing", "peaked") and topk < n:             # seen by the router: nothing is listed
        assert (redo, pairs) == (1, 0) and torch.equal(one, two)
    elif mode == SEQ and kind in ("constant", "region"):         # a head has more ties at its threshold than are ranked
        assert redo == 1 and pairs > 0 and torch.equal(one, two)
    else:                        # the one-pass form's scores but for the pairs that are settled, and its map
        assert redo == 0 and (kind == "constant" or not torch.equal(one, two))
        assert pairs > 0 or topk == n or (mode != SEQ and kind == "random")
    for name, x, y in zip(("row_ptr", "col_idx", "col_ptr", "row_idx"), two_map, one_map):
        if mode != BUDGET or "ptr" in name:
            assert torch.equal(x, y), name
    if mode == BUDGET:                                           # (heads keep different numbers of entries)
        for h in range(heads_q):
            e = int(two_map[0][0, h, -1])
            assert torch.equal(two_map[1][0, h, :e], one_map[1][0, h, :e]) and torch.equal(two_map[3][0, h, :e], one_map[3][0, h, :e])
    # the bound derived in select.cu (from 2^-52 on; on these inputs it holds from 2^-60 on)
    counted = two >= 2.0 ** -60
    assert ((one - two).abs() <= 1.4e-5 * two)[counted].all()
    if mode == SEQ and kind == "random":
        # the band of a head: its two-pass scores
        tau = two.flatten(2).topk(n * topk, dim=-1).values[..., -1].view(torch.int32)[..., None, None]
        band = (two.view(torch.int32) - tau).abs() <= 128        # (well inside the 512 units of the one-pass threshold)
        assert band.sum() >= heads_q and torch.equal(one[band], two[band])


@pytest.mark.parametrize("heads,dim,grid,cube", [
    (1, 64, (16, 32, 32), {}),            # one item a CTA: every tile is fetched behind the loop
    (2, 128, (20, 18, 68), WIDE),
    (7, 128, (13, 30, 33), {}),           # two or three items a CTA
])
def test_parked_sums_come_back_whole(heads, dim, grid, cube):
    """Every parked sum is read after it was written, those of a CTA's last item too: NaN wherever one is not, run after run."""
    p = vb.make_params(1, heads, heads, dim, grid, topk=9, **cube)
    q, k = _inputs(heads, heads, dim, grid, "random")
    attn = vb.Vsa2Attention(p)
    n = -(-grid[0] // 4) * -(-grid[1] // 4) * -(-grid[2] // (8 if cube else 4))
    tiles = -(-8 * n * (2 if cube else 1) // 128)
    scratch = torch.empty(148 * tiles * 8192 + heads * (4 * 128 * tiles + 4 * n) + (1 << 20) + 4096, dtype=torch.uint8, device="cuda")
    first = None
    for _ in range(12):
        scratch.fill_(0xff)
        vb.vsa2_route(p, q, k, None, attn.map, attn.ws_route, scratch=scratch)
        attn.check_status()
        scores = attn.scores().clone()
        assert torch.isfinite(scores).all()
        first = scores if first is None else first
        assert torch.equal(scores, first)


def test_pairs_whose_flat_index_is_beyond_32_bits_are_settled():
    """48,400 cubes: row * cubes + column passes 2^31 in the last rows, of which some entries lie in the band of the threshold."""
    grid = (16, 440, 440)
    p = vb.make_params(1, 1, 1, 64, grid, topk=4)
    q, k = _inputs(1, 1, 64, grid, "random")
    attn = vb.Vsa2Attention(p)
    n, tiles = 48400, 3025
    scratch = torch.empty(148 * tiles * 8192 + 4 * 128 * tiles + 4 * n + (1 << 20) + 4096, dtype=torch.uint8, device="cuda")
    maps = []
    for s in (None, scratch):
        vb.vsa2_route(p, q, k, None, attn.map, attn.ws_route, scratch=s)
        attn.check_status()
        maps.append([x.clone() for x in attn.map_views()])
    redo, pairs = _state(attn)
    assert redo == 0 and pairs > 0
    for name, x, y in zip(("row_ptr", "col_idx", "col_ptr", "row_idx"), *maps):
        assert torch.equal(x, y), name


def _levels(kind):
    """256 cubes, 16 key tiles of 16 cubes; a thread has the cubes 4 part .. 4 part + 3 of every tile.  Scores of the key cubes in nats below a
    dominant key in cube 0, by query sub-cube (0; the others)."""
    cube = torch.arange(256, device="cuda")
    tile, part = cube // 16, cube % 16 // 4
    if kind == "tail":          # parts 1 - 3: the first tile 124 octaves down, the later ones 76; part 0: from 101 octaves on, cube by cube
        k0 = torch.where(tile == 0, -86.0, -53.0)
        in0 = part == 0
        k0[in0] = -70.0 - 0.5 * torch.arange(int(in0.sum()), device="cuda")
        k1 = k0
        k2 = torch.zeros(256, device="cuda")
    else:                       # "rows": part 0 leads by a 16th of a nat where sub-cube 0 asks, parts 1 - 3 by a tenth with the other sub-cubes
        k0 = torch.where((part > 0) & (tile == 0), -38.0, -37.0)
        k1 = torch.where(part == 0, -100.0, torch.where(tile == 0, -85.5, -41.25))
        k2 = torch.where(part == 0, 0.5, 0.0)
    k0, k1, k2 = k0.clone(), k1.clone(), k2.clone()
    k0[0] = k1[0] = k2[0] = 0.0
    return k0, k1, k2


@pytest.mark.parametrize("kind,mode,topk", [("tail", ROW, 4), ("tail", SEQ, 4), ("tail", BUDGET, 4), ("rows", ROW, 4),
                                            ("tail", ROW, 256), ("tail", SEQ, 256), ("tail", BUDGET, 300)])
def test_thresholds_far_below_the_row_maximum(kind, mode, topk):
    """A thread's parked sums are lost where its first scores lie 2^126 below the row's denominator, the scores it has later (up to 2^48
    more) with them: a threshold so low must not be taken from one-pass scores, however clear of its neighbours it is -- unless
    everything is kept."""
    grid = (16, 32, 32)
    k0, k1, k2 = _levels(kind)
    t, h, w = (x.reshape(-1) for x in torch.meshgrid(*(torch.arange(n, device="cuda") for n in grid), indexing="ij"))
    of = (t // 4 * 8 + h // 4) * 8 + w // 4
    first = ((t % 4 < 2) & (h % 4 < 2) & (w % 4 < 2)).float()                 # tokens of sub-cube 0
    gen = torch.Generator(device="cuda").manual_seed(3)
    noise = 0.25 if kind == "tail" else 0.0
    q = noise * torch.randn(1, 1, 16384, 64, device="cuda", generator=gen)
    k = noise * 4 * torch.randn(1, 1, 16384, 64, device="cuda", generator=gen)
    q[..., 0], q[..., 1], q[..., 2] = 8.0 * first, 8.0 * (1.0 - first), 1.0
    k[..., 0], k[..., 1], k[..., 2] = k0[of], k1[of], k2[of]
    q, k = q.bfloat16(), k.bfloat16()
    budgets = torch.full((1, 1, 256), topk, device="cuda", dtype=torch.int32) if mode == BUDGET else None
    p = vb.make_params(1, 1, 1, 64, grid, select_mode=mode, topk=0 if mode == BUDGET else topk,
                       nnz_cap=256 * min(topk, 256))
    attn = vb.Vsa2Attention(p)
    scratch = torch.empty(16 << 20, dtype=torch.uint8, device="cuda")
    maps = []
    for s in (None, scratch):
        vb.vsa2_route(p, q, k, budgets, attn.map, attn.ws_route, scratch=s)
        attn.check_status()
        maps.append([x.clone() for x in attn.map_views()])
    assert _state(attn)[0] == (topk < 256)
    for name, x, y in zip(("row_ptr", "col_idx", "col_ptr", "row_idx"), *maps):
        assert torch.equal(x, y), name


@pytest.mark.parametrize("mode", [SEQ, ROW])
@pytest.mark.parametrize("kind", ["key nan", "key inf", "key -inf", "query nan", "query inf"])
def test_scores_that_are_not_finite(kind, mode):
    """Rows whose denominator is not a number keep their scores as they are: 2^144 at the cubes of the first key tile of parts 1 - 3, 2^-86
    at their others (beyond the fp32 range of what is parked against the first), 1 in part 0."""
    grid, topk = (16, 32, 32), 200
    cube = torch.arange(256, device="cuda")
    level = torch.where(cube % 16 < 4, 0.0, torch.where(cube < 16, 100.0, -60.0))
    t, h, w = (x.reshape(-1) for x in torch.meshgrid(*(torch.arange(n, device="cuda") for n in grid), indexing="ij"))
    q, k = (x.float() * 0.1 for x in _inputs(1, 1, 64, grid, "random"))
    q[..., 0], k[..., 0] = 8.0, level[(t // 4 * 8 + h // 4) * 8 + w // 4]
    x, value = (q if kind.startswith("query") else k), float(kind.split()[1])
    x[0, 0, 2048 + 128, 3] = value                       # (of cube 8, of part 2, or of query cube 8)
    if kind == "key nan":
        k[0, 0, 2048, 3] = value                         # (of cube 0, of part 0)
    p = vb.make_params(1, 1, 1, 64, grid, select_mode=mode, topk=topk)
    attn = vb.Vsa2Attention(p)
    scratch = torch.empty(16 << 20, dtype=torch.uint8, device="cuda")
    out = []
    for s in (None, scratch):
        vb.vsa2_route(p, q.bfloat16(), k.bfloat16(), None, attn.map, attn.ws_route, scratch=s)
        attn.check_status()
        out.append(([x.clone() for x in attn.map_views()], attn.scores()))
    (two_map, two), (one_map, one) = out
    for name, x, y in zip(("row_ptr", "col_idx", "col_ptr", "row_idx"), two_map, one_map):
        assert torch.equal(x, y), name
    assert torch.equal(one.isnan(), two.isnan())
    counted = two >= 2.0 ** -40
    assert (((one - two).abs() <= 1.4e-5 * two) | (one == two))[counted].all()


@pytest.mark.parametrize("heads_q,heads_kv,dim,grid,cube,mode", [
    (9, 9, 128, (21, 30, 52), {}, SEQ),
    (12, 12, 64, (21, 30, 52), {}, ROW),
    (2, 2, 128, (61, 30, 52), WIDE, ROW),
])
def test_scratch_of_the_size_asked_for_is_enough_and_one_byte_less_is_none(heads_q, heads_kv, dim, grid, cube, mode):
    p = vb.make_params(1, heads_q, heads_kv, dim, grid, select_mode=mode, topk=16, **cube)
    q, k = _inputs(heads_q, heads_kv, dim, grid, "random")
    attn = vb.Vsa2Attention(p)
    size = vb.vsa2_route_scratch_bytes(p)
    assert size == attn.route_scratch_bytes > 0
    guarded = torch.full((size + 4096,), 0xa5, dtype=torch.uint8, device="cuda")
    scores, settled = [], []
    for scratch in (None, guarded[:size - 1], guarded[:size]):
        vb.vsa2_route(p, q, k, None, attn.map, attn.ws_route, scratch=scratch)
        attn.check_status()
        scores.append(attn.scores())
        settled.append(_state(attn))
    assert (guarded[size:] == 0xa5).all()
    assert torch.equal(scores[0], scores[1]) and not torch.equal(scores[0], scores[2])
    assert settled[1] == (0, 0) and settled[2][0] == 0 and settled[2][1] > 0
