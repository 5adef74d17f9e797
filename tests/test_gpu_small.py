"""The N = 256 kernel of the two-prime form (variant 2, base 2^8) against the
general kernel (variant 0), word for word: party counts on both register
builds, batches of one gate per SM and more, step limits inside a party,
skipped steps, rotations at the ends of the range."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,count,steps", [(1, 1, -1), (2, 24, -1), (2, 153, 100), (2, 700, 20), (3, 5, -1), (3, 200, 70),
                                           (4, 3, -1), (5, 160, 40), (8, 2, -1)])
def test_accumulators_equal_the_general_kernel(k, count, steps):
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = W.toy_params(k)
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(k)):
        ctx.keygen(p, s)
    r = np.random.default_rng(k + count)
    abar = r.integers(0, 2 * P["N"], size=(count, k * P["n"] + 1))
    abar[r.random(abar.shape) < 0.1] = 0
    abar[0, :4] = [0, 1, P["N"], 2 * P["N"] - 1]
    abar[-1, -1] = 2 * P["N"] - 1
    if count > 1:
        abar[1, :P["n"]] = 0
    dev = torch.from_numpy(abar.astype(np.int32)).cuda()
    accs = []
    for mode, variant in (("auto", 2), ("off", 2), ("off", 0)):
        acc = torch.full((count, (k + 1) * P["N"]), -1, dtype=torch.int32, device="cuda")
        ctx.set_cluster(mode)
        ctx.set_variant(variant)
        ctx.stage_blind_rotate(dev, steps, acc)
        ctx.sync()
        accs.append(acc)
    assert torch.equal(accs[0], accs[2]) and torch.equal(accs[1], accs[2])
    ctx.close()
