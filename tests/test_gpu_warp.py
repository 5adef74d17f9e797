"""The warp kernel of the two-prime form (variant 2 at N = 1024, base 2^8)
against the general kernel (variant 0), word for word: both are exact, so
every accumulator coefficient has to be equal.

Cases sit where the kernel can go wrong: party counts with no, one and many
other polynomials (and fewer gates per CTA), batches around one and several
gates per CTA and past one pass of the grid, step limits in the middle of a
party, rotations 0, 1, N, 2N - 1 and runs of skipped steps."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _ctx(P):
    from paper_2205_05825_gb300 import binding as B
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(P["k"])):
        ctx.keygen(p, s)
    ctx.set_cluster("off")
    return ctx


def _rotate(ctx, variant, abar, steps):
    import torch
    k, N = ctx.params["k"], ctx.params["N"]
    acc = torch.full((abar.shape[0], (k + 1) * N), -1, dtype=torch.int32, device="cuda")
    ctx.set_variant(variant)
    ctx.stage_blind_rotate(abar, steps, acc)
    ctx.sync()
    return acc


# n = 24 keeps the keys and the runs small; everything else is the full set.
@pytest.mark.parametrize("k,count,steps", [(1, 5, -1), (2, 1, -1), (2, 153, 30), (2, 305, 25), (2, 470, 26), (3, 7, -1),
                                           (4, 160, 50), (5, 3, 70), (6, 2, 100), (8, 310, 28), (8, 2, -1)])
def test_accumulators_equal_the_general_kernel(k, count, steps):
    import torch
    P = dict(W.full_params(k), n=24)
    ctx = _ctx(P)
    r = np.random.default_rng(7 * k + count)
    abar = r.integers(0, 2 * P["N"], size=(count, k * P["n"] + 1))
    abar[r.random(abar.shape) < 0.1] = 0
    special = np.array([0, 1, P["N"] - 1, P["N"], P["N"] + 1, 2 * P["N"] - 1])
    abar[0, :len(special)] = special
    abar[-1, -1] = 2 * P["N"] - 1
    if count > 1:
        abar[1, :P["n"]] = 0  # a party whose steps are all skipped
    dev = torch.from_numpy(abar.astype(np.int32)).cuda()
    assert torch.equal(_rotate(ctx, 2, dev, steps), _rotate(ctx, 0, dev, steps))
    ctx.close()


@pytest.mark.parametrize("k,count", [(2, 9), (3, 4)])
def test_gates_equal_the_general_kernel(k, count):
    """Linear part, sample extraction and key switch around it, per-gate types."""
    import torch
    P = dict(W.full_params(k), n=24)
    ctx = _ctx(P)
    types, b1, b2 = W.random_gates(count, config_id=40 + k)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()
    a, b = dev(ctx.encrypt_joint(b1, 1)), dev(ctx.encrypt_joint(b2, 2))
    ty = torch.from_numpy(types.astype(np.uint8)).cuda()
    outs = []
    for variant in (2, 0):
        out = torch.zeros((count, ctx.W), dtype=torch.int32, device="cuda")
        ctx.set_variant(variant)
        ctx.gates(ty, a, b, out)
        ctx.sync()
        outs.append(out)
    assert torch.equal(*outs)
    ctx.close()
