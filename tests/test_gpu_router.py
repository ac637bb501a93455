"""GPU parity of the block scores P_r of the tensor-core router: one and several items per CTA, one and many key tiles, a last
tile of one cube, 128-token cubes whose scores the kernel folds from half-cubes (empty second halves among them), and scores that
climb along a row."""
import numpy as np
import pytest

from oracle import vsa2_oracle as orc
from paper_2609_32882_b200 import inputs as syn

pytestmark = pytest.mark.gpu

WIDE = dict(cube=(4, 4, 8), rpool=(2, 2, 2))
# name, heads_q, heads_kv, D, grid, cube kind, growth of the scores along the frames
CASES = [
    ("one_tile", 2, 1, 64, (4, 8, 8), {}, 0.0),
    ("one_cube_over", 3, 3, 128, (3, 4, 65), {}, 0.0),
    ("several_items_per_cta", 16, 4, 64, (11, 18, 57), {}, 0.0),
    ("wide_7_tiles", 2, 2, 128, (8, 20, 37), WIDE, 0.0),
    ("wide_empty_half", 2, 1, 128, (20, 18, 68), WIDE, 0.0),
    ("wide_16_per_half", 2, 1, 64, (8, 12, 40), dict(cube=(4, 4, 8), rpool=(1, 2, 2)), 0.0),
    ("growing", 2, 2, 64, (28, 28, 28), {}, 60.0),
    ("growing_wide", 2, 2, 128, (40, 20, 40), WIDE, 60.0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
def test_block_scores(case):
    import vsa2_testlib as tl
    name, hq, hk, dim, grid, cube, growth = case
    wl = syn.Workload(name, 1, hq, hk, dim, grid, select_mode=syn.PER_QUERY, topk=4, seed=90, **cube)
    data = syn.make_inputs(wl, with_grad=False)
    if growth:
        # a direction shared by every query that the keys follow more and more along t: the scores of a row climb by
        # up to `growth` nats from its first key tile to its last
        q, k = (data[n].astype(np.uint32) << 16 for n in "qk")
        q, k = q.view(np.float32).copy(), k.view(np.float32).copy()
        t = (np.arange(q.shape[2]) // (grid[1] * grid[2])) / (grid[0] - 1)
        q[..., 0] = 4.0
        k[..., 0] = (growth * np.sqrt(dim) / 4.0 * t)[None, None, :]
        data["q"], data["k"] = ((x.view(np.uint32) >> 16).astype(np.uint16) for x in (q, k))
    run = tl.CudaPath(wl, data)
    run.route()
    got = tl.to_f64(run.attn.scores())
    a = tl.oracle_arrays({**data})
    _, want = orc.route(a["q"], a["k"], orc.Geometry(wl.grid, wl.cube, wl.rpool), 1.0 / np.sqrt(dim), wl.select_mode, wl.topk,
                        return_scores=True)
    # a score s carries the rounding of a D-term fp32 sum and of the exponent's multiply-add: |s| log2(e) (1 + D / 8) 2^-24 at
    # most, i.e. under 1.3e-4 relative in exp(s) for |s| <= 60 and D = 128; sums of positive terms add 2^-22 or so
    scale = np.abs(want)
    bad = np.abs(got - want) > 2e-4 * scale + 1e-30
    assert not bad.any(), (name, float((np.abs(got - want) / np.maximum(scale, 1e-30)).max()))
