"""Gradients of a loss that is a mean over many elements: dO far below one, or V far below one.  The fp16 forms of the backward
passes round dS to fp16, whose subnormals end at 2^-24; dQ, dK and dV scale with dO (dQ and dK with V too), so they must meet the
stated bounds scaled by the same factors -- with the score gradients kept between the passes and with them formed twice."""
import numpy as np
import pytest

from oracle import vsa2_oracle as orc
from paper_2609_32882_b200 import binding as vb
from paper_2609_32882_b200 import inputs as syn
from vsa2_testlib import TOL_ABS, CudaPath, assert_close, oracle_arrays, to_f64

pytestmark = pytest.mark.gpu

WORKLOADS = [
    syn.Workload("small_mha", 1, 2, 2, 128, (8, 12, 12), select_mode=syn.PER_QUERY, topk=12, seed=301),
    syn.Workload("small_gqa", 2, 4, 2, 128, (8, 12, 9), select_mode=syn.PER_QUERY, topk=10, seed=302),       # four fp16 copies
    syn.Workload("small_gqa_pairs", 1, 4, 1, 64, (8, 12, 12), select_mode=syn.PER_QUERY, topk=6, seed=303),  # bf16 pairs in dK/dV
    syn.Workload("small_wide", 1, 2, 2, 128, (8, 12, 20), select_mode=syn.PER_QUERY, topk=9, cube=(4, 4, 8), rpool=(2, 2, 2), seed=304),
    syn.Workload("small_ragged", 1, 3, 3, 64, (5, 11, 13), select_mode=syn.PER_SEQUENCE, topk=7, seed=305),
]


@pytest.mark.parametrize("least", [False, True], ids=["stored", "recomputed"])
@pytest.mark.parametrize("tensor,factor", [("do", 1e-4), ("do", 1e-7), ("do", 1e-20), ("v", 1e-3), ("v", 1e-6)])
@pytest.mark.parametrize("wl", WORKLOADS, ids=lambda w: w.name)
def test_small_gradients_keep_their_bits(wl, tensor, factor, least):
    data = syn.make_inputs(wl)
    data[tensor] = syn.f32_to_bf16_bits(syn.bf16_bits_to_f32(data[tensor]) * np.float32(factor))
    if tensor == "do":
        # one head a thousand times below the others (heads of a KV group share a scale)
        d = syn.bf16_bits_to_f32(data["do"]).copy()
        d[:, -1] *= np.float32(1e-3)
        data["do"] = syn.f32_to_bf16_bits(d)
    run = CudaPath(wl, data, out_dtype=vb.F32, flags=vb.FLAG_NO_COARSE)
    if least:
        run.attn.bwd_scratch_bytes = 0
    run.route()
    run.forward()
    run.backward()
    a = oracle_arrays(data)
    want = orc.backward(a["q"], a["k"], a["v"], np.zeros_like(a["gate"]), run.mask, orc.Geometry(wl.grid, wl.cube, wl.rpool),
                        1.0 / np.sqrt(wl.head_dim), a["do"])
    rep = wl.heads_q // wl.heads_kv
    for name, got, ref in zip(("dQ", "dK", "dV"), (run.dq, run.dk, run.dv), want):
        got = to_f64(got)
        for h in range(ref.shape[1]):
            last = h == ref.shape[1] - 1 and (name == "dQ" or rep == 1)
            unit = factor if tensor == "do" or name != "dV" else 1.0
            if tensor == "do" and last:
                # a head that shares its group's scale may lose to it what a dS 1000 times smaller than the group's loses
                if rep > 1:
                    continue
                unit *= 1e-3
            assert_close(f"{name} head {h}", got[:, h], ref[:, h], tol_abs=TOL_ABS * unit)
