"""The key switch of more rows than a grid has y blocks for groups of 256
(16,776,960): rows around that limit and the last one, word for word against
the definition (Sec. 3.2) in numpy.  17 GB of extracted samples."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W
from test_gpu_keyswitch import reference

pytestmark = pytest.mark.gpu


def test_more_groups_than_grid_y():
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.toy_params(1), n=4)
    ctx = B.Context(P, W.CRS_SEED, device=0)
    ctx.keygen(0, W.party_seeds(1)[0])
    ks = [ctx.export_party(0, ("ks",))["ks"]]
    limit = 65535 * 256
    count = limit + 300
    ext = torch.empty((count, ctx.E), dtype=torch.int32, device="cuda").random_(-(1 << 31), 1 << 31)
    out = torch.full((count, ctx.W), -1, dtype=torch.int32, device="cuda")
    ctx.stage_keyswitch(ext, out)
    ctx.sync()
    rows = torch.tensor([0, 255, 256, limit - 1, limit, limit + 255, limit + 256, count - 1], device="cuda")
    got, sample = (t[rows].cpu().numpy().view(np.uint32) for t in (out, ext))
    ctx.close()
    assert np.array_equal(got, reference(P, ks, sample))
