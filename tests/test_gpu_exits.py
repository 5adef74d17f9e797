"""Kernels whose wait for matrix products runs out near their end: the step
whose products are withheld is the last but one, so the last step's products
are issued and never waited for by the abandoned loop, and only the exit's own
wait stands between them and the release of TMEM.  The launch is followed, on
the same stream, by one that allocates the same TMEM at once.  Checked:
mk_sync reports MK_ETIMEOUT once, and the next launch is right word for word.
(On the CPU: tests/test_shared_protocol.py.)"""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def check(k, count, cluster):
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.full_params(k), n=24)
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(k)):
        ctx.keygen(p, s)
    ctx.set_cluster(cluster)
    abar = np.random.default_rng(k + count).integers(1, 2 * P["N"], size=(count, k * P["n"] + 1))
    dev = torch.from_numpy(abar.astype(np.int32)).cuda()
    good, bad, acc = (torch.zeros((count, (k + 1) * P["N"]), dtype=torch.int32, device="cuda") for _ in range(3))
    ctx.stage_blind_rotate(dev, -1, good)
    ctx.sync()
    for _ in range(3):
        ctx.debug_fault("skip_key_step", k * P["n"] - 2, 20_000_000)
        ctx.stage_blind_rotate(dev, -1, bad)
        ctx.stage_blind_rotate(dev, k * P["n"] - 2, acc)  # ends before the withheld step
        with pytest.raises(B.MkError, match="MK_ETIMEOUT"):
            ctx.sync()
        ctx.sync()
        ctx.debug_fault("none")
        ctx.stage_blind_rotate(dev, -1, acc)
        ctx.sync()
        assert torch.equal(acc, good)
    ctx.close()


@pytest.mark.parametrize("k,count", [(1, 1), (2, 3), (2, 60), (2, 152), (4, 2), (8, 1), (8, 40)])
def test_latency_form(k, count):
    check(k, count, "on")


@pytest.mark.parametrize("k,count", [(4, 100), (8, 304)])
def test_one_cta_a_gate(k, count):
    check(k, count, "auto")
