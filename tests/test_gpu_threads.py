"""Two threads, each with its own context and stream, launch the same kernel
with different amounts of shared memory (gates a CTA, or party counts):
neither thread's limit may refuse the other's launches, and the results are
those of one thread alone."""
import threading

import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _ctx(P):
    import torch
    from paper_2205_05825_gb300 import binding as B
    stream = torch.cuda.Stream()
    ctx = B.Context(P, W.CRS_SEED, device=0, stream=stream.cuda_stream)
    for p, s in enumerate(W.party_seeds(P["k"])):
        ctx.keygen(p, s)
    ctx._keep = stream
    return ctx


@pytest.mark.parametrize("base,jobs,cluster", [("full", ((2, 1), (2, 400)), "off"), ("full", ((1, 2), (3, 2)), "on"),
                                               ("full", ((3, 150), (7, 150)), "auto"), ("toy", ((1, 2), (3, 2)), "auto")])
def test_launches_of_two_threads(base, jobs, cluster):
    import torch
    runs = []
    for k, count in jobs:
        P = dict((W.full_params if base == "full" else W.toy_params)(k), n=8)
        ctx = _ctx(P)
        ctx.set_cluster(cluster)
        abar = np.random.default_rng(k).integers(0, 2 * P["N"], size=(count, ctx.W)).astype(np.int32)
        dev = torch.from_numpy(abar).cuda()
        good, acc = (torch.zeros((count, (k + 1) * P["N"]), dtype=torch.int32, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        ctx.stage_blind_rotate(dev, 2, good)
        ctx.sync()
        runs.append((ctx, dev, good, acc))
    errors = []

    def work(ctx, dev, acc):
        try:
            for _ in range(1500):
                ctx.stage_blind_rotate(dev, 2, acc)
            ctx.sync()
        except Exception as e:  # reported by the main thread
            errors.append(str(e))
    threads = [threading.Thread(target=work, args=(ctx, dev, acc)) for ctx, dev, _, acc in runs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for ctx, _, good, acc in runs:
        assert torch.equal(acc, good)
        ctx.close()
