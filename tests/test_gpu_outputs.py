"""Output tensors that a handle allocates: contiguous, in the output type and on the queries' device, whatever kind of tensor the inputs are, and on the
stream that is current for the calling thread."""
import threading

import pytest
import torch

from paper_2609_32882_b200 import binding as vb

pytestmark = pytest.mark.gpu


class Labelled(torch.Tensor):
    pass


@pytest.mark.parametrize("out_dtype", [vb.BF16, vb.F32])
@pytest.mark.parametrize("kind", ["tensor", "parameter", "subclass"])
def test_outputs(out_dtype, kind):
    p = vb.make_params(1, 2, 1, 64, (4, 8, 8), select_mode=vb.PER_QUERY, topk=2, out_dtype=out_dtype)
    attn = vb.Vsa2Attention(p)
    wrap = {"tensor": lambda x: x, "parameter": torch.nn.Parameter, "subclass": lambda x: x.as_subclass(Labelled)}[kind]
    q, k, v = (wrap(torch.randn(1, h, 256, 64, device="cuda").bfloat16()) for h in (2, 1, 1))
    gate = torch.rand(1, 2, 256, device="cuda")
    attn.route(q, k)
    o, lse = attn.forward(q, k, v, gate)
    dq, dk, dv, dgate = attn.backward(q, k, v, gate, o, lse, torch.randn_like(q).detach())
    attn.check_status()
    kind_out = torch.float32 if out_dtype == vb.F32 else torch.bfloat16
    for x, shape, dtype in ((o, q.shape, kind_out), (lse, q.shape[:-1], torch.float32), (dq, q.shape, kind_out), (dk, k.shape, kind_out),
                            (dv, v.shape, kind_out), (dgate, (1, 2, 256), torch.float32)):
        assert type(x) is torch.Tensor and not x.requires_grad
        assert x.shape == shape and x.dtype == dtype and x.is_contiguous() and x.device == q.device


def test_stream_of_the_calling_thread():
    """The handle that a call without a stream runs on is the one of torch.cuda.current_stream(), in each thread and inside a stream context."""
    seen = []

    def look():
        side = torch.cuda.Stream()
        for _ in range(3):
            assert vb._stream(None) == torch.cuda.current_stream().cuda_stream == 0
            with torch.cuda.stream(side):
                assert vb._stream(None) == side.cuda_stream != 0
        seen.append(side.cuda_stream)

    torch.cuda.init()
    threads = [threading.Thread(target=look) for _ in range(2)]
    for t in threads:
        t.start()
    look()
    for t in threads:
        t.join()
    assert len(seen) == 3
