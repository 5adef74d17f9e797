"""An operator's captured graph is captured again when the latency mode
changes, also where the mode is all that differs: at k = 8 the cluster kernel
does not exist, so the threshold it was chosen by is 0 in every mode.

The two modes' kernels are told apart by the fault hook: with variant 0, OFF
runs the variant's own kernel, which waits for nothing, and AUTO the team
kernel, whose wait for the withheld products runs out."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_latency_mode_change_recaptures():
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.full_params(8), n=24)
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(8)):
        ctx.keygen(p, s)
    a, b = (torch.from_numpy(ctx.encrypt_joint(np.array([1, 0], np.uint8), 70 + j).view(np.int32)).cuda().reshape(1, 2, -1)
            for j in range(2))
    off, out = (torch.zeros((1, 2, ctx.W), dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.set_variant(0)
    ctx.set_graphs(True)
    ctx.debug_fault("skip_key_step", 0, 20_000_000)
    ctx.set_cluster("off")
    ctx.add_kbit(2, a, b, off)
    ctx.sync()
    assert ctx.route(1) == [(1, "variant")]
    ctx.set_cluster("auto")
    assert ctx.route(1) == [(1, "team")]
    ctx.add_kbit(2, a, b, out)
    with pytest.raises(B.MkError, match="MK_ETIMEOUT"):
        ctx.sync()
    ctx.debug_fault("none")
    ctx.add_kbit(2, a, b, out)
    ctx.sync()
    assert torch.equal(out, off)
    ctx.close()
