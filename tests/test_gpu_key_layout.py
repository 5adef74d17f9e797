"""The key layout is finished when the call that made it returns: the next
call may come on another stream, which nothing orders after the first.

Keys are laid out by a modulus switch on one stream (the call that shares
neither scratch nor data with a key switch); the key switch then runs at once
on another non-blocking stream and is compared, word for word, with its
definition (Sec. 3.2) in numpy.  Once with the matrix-product key switch,
whose operand blocks are built on the device, and once with the SIMT one
(t = 7), which reads the uploaded rows."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W
from test_gpu_keyswitch import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [dict(W.full_params(2), n=170), dict(W.toy_params(2), t=7)], ids=["product", "simt"])
@pytest.mark.parametrize("first", ["default", "other"])
def test_key_switch_on_another_stream_right_after_the_layout(P, first):
    import torch
    from paper_2205_05825_gb300 import binding as B
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = B.Context(P, W.CRS_SEED, device=0, stream=a.cuda_stream if first == "other" else None)
    ext = np.random.default_rng(17).integers(0, 1 << 32, size=(3, ctx.E), dtype=np.uint32)
    ext_d = torch.from_numpy(ext.view(np.int32)).cuda()
    out = torch.full((3, ctx.W), -1, dtype=torch.int32, device="cuda")
    rows, abar = (torch.zeros((1, ctx.W), dtype=torch.int32, device="cuda") for _ in range(2))
    lin = torch.from_numpy(B.lin_records([0])).cuda()
    torch.cuda.synchronize()
    for again in range(3):  # other keys, laid out anew, each time
        for p, s in enumerate(W.party_seeds(2)):
            ctx.keygen(p, s + 100 * again)
        ks = [ctx.export_party(p, ("ks",))["ks"] for p in range(2)]
        out.fill_(-1)
        torch.cuda.synchronize()
        ctx.set_stream(a.cuda_stream if first == "other" else 0)
        ctx.stage_modswitch(lin, rows, rows, abar)
        ctx.set_stream(b.cuda_stream)
        ctx.stage_keyswitch(ext_d, out)
        ctx.sync()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), reference(P, ks, ext))
    ctx.set_stream(0)
    ctx.close()
