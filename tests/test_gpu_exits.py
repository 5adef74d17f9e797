"""Kernels whose wait for matrix products or key tiles runs out, which then
have to leave with nothing in flight.  The blind rotations near their end: the step
whose products are withheld is the last but one, so the last step's products
are issued and never waited for by the abandoned loop, and only the exit's own
wait stands between them and the release of TMEM.  The launch is followed, on
the same stream, by one that allocates the same TMEM at once.  Checked:
mk_sync reports MK_ETIMEOUT once, and the next launch is right word for word.
Also with the first step's products withheld (every later one is issued and
not waited for), and the key switch with its first, middle or last key tile.
(On the CPU: tests/test_shared_protocol.py, tests/test_keyswitch_protocol.py.)"""
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
    for step in (k * P["n"] - 2, k * P["n"] - 2, 0):
        ctx.debug_fault("skip_key_step", step, 20_000_000)
        ctx.stage_blind_rotate(dev, -1, bad)
        ctx.stage_blind_rotate(dev, step, acc)  # ends before the withheld step
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


@pytest.mark.parametrize("k,count", [(1, 1), (2, 5), (2, 305), (2, 700), (8, 310)])
def test_warp_kernel(k, count):
    check(k, count, "off")


@pytest.mark.parametrize("count,pair", [(1, 0), (1, 511), (130, 255), (300, 0), (4096, 511)])
def test_key_switch(count, pair):
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.full_params(2), n=170)
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(2)):
        ctx.keygen(p, s)
    ext = torch.from_numpy(np.random.default_rng(count).integers(0, 1 << 32, size=(count, ctx.E), dtype=np.uint32)
                           .view(np.int32)).cuda()
    good, out = (torch.zeros((count, ctx.W), dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.stage_keyswitch(ext, good)
    ctx.sync()
    for _ in range(3):
        ctx.debug_fault("skip_key_tile", pair, 20_000_000)
        ctx.stage_keyswitch(ext, out)
        with pytest.raises(B.MkError, match="MK_ETIMEOUT"):
            ctx.sync()
        ctx.sync()
        ctx.debug_fault("none")
        ctx.stage_keyswitch(ext, out)
        ctx.sync()
        assert torch.equal(out, good)
    ctx.close()
