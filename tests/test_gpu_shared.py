"""The shared kernel (two-prime blind rotation at N = 1024, base 2^8: a gate a
CTA, its polynomials shared out among three teams) against the general
kernel, word for word, at counts where the launch rule takes it, and batches
that run as two launches.

Every party count it can take, a part-filled and an over-filled chip, step
limits inside a party, skipped steps and a party whose steps are all skipped;
gates whose last pass has one gate, some, and nearly all of the chip; and the
bounded wait."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _abar(P, count, seed):
    r = np.random.default_rng(seed)
    abar = r.integers(0, 2 * P["N"], size=(count, P["k"] * P["n"] + 1))
    abar[r.random(abar.shape) < 0.1] = 0
    abar[0, :4] = [0, 1, P["N"], 2 * P["N"] - 1]
    abar[1, :P["n"]] = 0
    return abar.astype(np.int32)


def _ctx(P):
    from paper_2205_05825_gb300 import binding as B
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(P["k"])):
        ctx.keygen(p, s)
    return ctx


@pytest.mark.parametrize("k,count,steps", [(3, 150, -1), (4, 100, -1), (4, 152, 61), (5, 100, -1), (6, 100, 37), (7, 100, -1),
                                           (8, 96, -1), (8, 304, 50), (2, 153, -1), (4, 200, 40), (4, 480, 30)])
def test_accumulators_equal_the_general_kernel(k, count, steps):
    import torch
    P = dict(W.full_params(k), n=24)
    ctx = _ctx(P)
    dev = torch.from_numpy(_abar(P, count, 10 * k + count)).cuda()
    accs = []
    for mode, variant in (("auto", 2), ("off", 0)):
        acc = torch.full((count, (k + 1) * P["N"]), -1, dtype=torch.int32, device="cuda")
        ctx.set_cluster(mode)
        ctx.set_variant(variant)
        ctx.stage_blind_rotate(dev, steps, acc)
        ctx.sync()
        accs.append(acc)
    assert torch.equal(*accs)
    ctx.close()


@pytest.mark.parametrize("k,count", [(2, 153), (2, 457), (4, 301), (4, 465)])
def test_gates_of_two_launches_equal_the_general_kernel(k, count):
    import torch
    P = dict(W.full_params(k), n=24)
    ctx = _ctx(P)
    r = np.random.default_rng(count)
    bits = r.integers(0, 2, size=(2, count)).astype(np.uint8)
    a, b = (torch.from_numpy(ctx.encrypt_joint(bits[j], 30 + j).view(np.int32)).cuda() for j in range(2))
    types = torch.from_numpy(r.integers(0, 6, count).astype(np.uint8)).cuda()
    outs = []
    for mode, variant in (("auto", 2), ("off", 0)):
        out = torch.zeros((count, ctx.W), dtype=torch.int32, device="cuda")
        ctx.set_cluster(mode)
        ctx.set_variant(variant)
        ctx.gates(types, a, b, out)
        ctx.sync()
        outs.append(out)
    assert torch.equal(*outs)
    ctx.close()


def test_products_wait_runs_out_and_the_context_recovers():
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = dict(W.full_params(4), n=24)
    ctx = _ctx(P)
    dev = torch.from_numpy(_abar(P, 100, 5)).cuda()
    good, acc = (torch.zeros((100, 5 * P["N"]), dtype=torch.int32, device="cuda") for _ in range(2))
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
