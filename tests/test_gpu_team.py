"""The team kernel (latency form of the two-prime blind rotation at N = 1024,
base 2^8) against the general kernel, word for word, with the form forced on.

Party counts from one team a cluster to nine polynomials on three CTAs with
idle teams, batches that pick one, two and three teams a CTA, step limits
inside a party, skipped steps, and the bounded wait."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _ctx(P):
    from paper_2205_05825_gb300 import binding as B
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(P["k"])):
        ctx.keygen(p, s)
    return ctx


def _abar(P, count, seed):
    r = np.random.default_rng(seed)
    abar = r.integers(0, 2 * P["N"], size=(count, P["k"] * P["n"] + 1))
    abar[r.random(abar.shape) < 0.1] = 0
    abar[0, :4] = [0, 1, P["N"], 2 * P["N"] - 1]
    if count > 1:
        abar[1, :P["n"]] = 0  # a party whose steps are all skipped
    return abar.astype(np.int32)


@pytest.mark.parametrize("k,count,steps", [(1, 1, -1), (2, 1, -1), (2, 3, 30), (2, 60, -1), (2, 100, 40), (2, 160, 30),
                                           (3, 2, -1), (4, 1, -1), (4, 40, 60), (5, 4, -1), (6, 1, -1), (7, 1, -1),
                                           (7, 30, 40), (8, 1, -1), (8, 40, 50)])
def test_accumulators_equal_the_general_kernel(k, count, steps):
    import torch
    P = dict(W.full_params(k), n=24)
    ctx = _ctx(P)
    dev = torch.from_numpy(_abar(P, count, 10 * k + count)).cuda()
    accs = []
    for mode, variant in (("on", 2), ("off", 0)):
        acc = torch.full((count, (k + 1) * P["N"]), -1, dtype=torch.int32, device="cuda")
        ctx.set_cluster(mode)
        ctx.set_variant(variant)
        ctx.stage_blind_rotate(dev, steps, acc)
        ctx.sync()
        accs.append(acc)
    assert torch.equal(*accs)
    ctx.close()


def test_products_wait_runs_out_and_the_context_recovers():
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.full_params(2), n=24)
    ctx = _ctx(P)
    ctx.set_cluster("on")
    dev = torch.from_numpy(_abar(P, 2, 5)).cuda()
    good, acc = (torch.zeros((2, 3 * P["N"]), dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.stage_blind_rotate(dev, -1, good)
    ctx.sync()
    step = int(np.flatnonzero(dev[0, :24].cpu().numpy())[3])
    ctx.debug_fault("skip_key_step", step, 20_000_000)
    ctx.stage_blind_rotate(dev, -1, acc)
    with pytest.raises(B.MkError, match="MK_ETIMEOUT"):
        ctx.sync()
    ctx.debug_fault("none")
    ctx.stage_blind_rotate(dev, -1, acc)
    ctx.sync()
    assert torch.equal(acc, good)
    ctx.close()
