"""The library in several CUDA contexts of one device: what it remembers about a kernel belongs to a context."""
import subprocess
import sys
import os

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import ctypes as C
from paper_2609_32882_b200 import binding as vb

cu = C.CDLL("libcuda.so.1")
def ok(code, what):
    assert code == 0, (what, code)
ok(cu.cuInit(0), "cuInit")
dev = C.c_int()
ok(cu.cuDeviceGet(C.byref(dev), 0), "cuDeviceGet")
p = vb.make_params(1, 2, 2, 64, (4, 8, 8), select_mode=vb.PER_QUERY, topk=2)
s = vb.vsa2_query_sizes(p)

def mem(nbytes):
    ptr = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(ptr), C.c_size_t(max(256, nbytes))), "cuMemAlloc")
    ok(cu.cuMemsetD8_v2(ptr, C.c_ubyte(0), C.c_size_t(max(256, nbytes))), "cuMemsetD8")
    return ptr.value

def one_pass():
    tok, n = 2 * 256, 2 * 256 * 64
    q, k, v, o, d_o, dq, dk, dv = (mem(2 * n) for _ in range(8))
    gate, lse, dgate = (mem(4 * tok) for _ in range(3))
    vmap = vb.Map(mem(4 * s.ptr_elems), mem(4 * s.idx_elems), mem(4 * s.ptr_elems), mem(4 * s.idx_elems))
    saved = vb.Saved(mem(4 * s.pooled_q_elems), mem(4 * s.pooled_kv_elems), mem(4 * s.pooled_kv_elems), mem(4 * s.pooled_q_elems),
                     mem(4 * s.lse_c_elems), mem(2 * s.o_res_elems))
    ws = [mem(x) for x in (s.route_workspace_bytes, s.fwd_workspace_bytes, s.bwd_workspace_bytes)]
    vb.vsa2_route(p, q, k, None, vmap, ws[0], s.route_workspace_bytes, stream=0)
    vb.vsa2_attn_fwd(p, q, k, v, gate, vmap, o, lse, saved, ws[1], s.fwd_workspace_bytes, stream=0)
    vb.vsa2_attn_bwd(p, q, k, v, gate, vmap, o, lse, saved, d_o, dq, dk, dv, dgate, ws[2], s.bwd_workspace_bytes, stream=0)
    assert [vb.vsa2_device_status(w, 0) for w in ws] == [0, 0, 0]

contexts = []
for _ in range(2):
    ctx = C.c_void_p()
    ok(cu.cuCtxCreate_v2(C.byref(ctx), 0, dev), "cuCtxCreate")
    contexts.append(ctx)
for i in (0, 1, 0, 1):
    ok(cu.cuCtxSetCurrent(contexts[i]), "cuCtxSetCurrent")
    one_pass()
for ctx in contexts:
    ok(cu.cuCtxDestroy_v2(ctx), "cuCtxDestroy")
print("both contexts")
"""


def test_two_contexts_of_a_device():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and "both contexts" in run.stdout, run.stdout + run.stderr
