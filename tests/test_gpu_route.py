"""Which kernel a launch gets, at the counts where tests/test_gpu_shared.py,
_warp, _team and _small compare kernels with the general one: a change of the
launch rule that takes a count elsewhere would leave those comparisons (and
the shared kernel's bounded wait) without their kernel, and fails here.

The counts have a margin that does not depend on how many clusters fit on the
GPU at hand: fewer make the team kernel dearer.  Also: the query refuses a
context whose keys are not laid out."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def contexts():
    import torch
    from paper_2205_05825_gb300 import binding as B
    made = {}

    def get(k, params=W.full_params):
        if (k, params) not in made:
            P = dict(params(k), n=24)
            ctx = B.Context(P, W.CRS_SEED, device=0)
            for p, s in enumerate(W.party_seeds(k)):
                ctx.keygen(p, s)
            with pytest.raises(B.MkError, match="MK_ESTATE"):
                ctx.route(1)
            ab = torch.zeros((1, ctx.W), dtype=torch.int32, device="cuda")
            ctx.stage_blind_rotate(ab, 0, torch.zeros((1, (k + 1) * P["N"]), dtype=torch.int32, device="cuda"))
            ctx.sync()
            made[k, params] = ctx
        ctx = made[k, params]
        ctx.set_cluster("auto")
        ctx.set_variant(2)
        return ctx
    yield get
    for ctx in made.values():
        ctx.close()


@pytest.mark.parametrize("k,count", [(3, 150), (4, 100), (4, 152), (5, 100), (6, 100), (7, 100), (8, 96), (8, 304)])
def test_shared(contexts, k, count):
    assert {name for _, name in contexts(k).route(count)} == {"shared"}


@pytest.mark.parametrize("k,count", [(2, 457), (4, 465), (4, 480)])
def test_two_launches(contexts, k, count):
    route = contexts(k).route(count)
    assert len(route) == 2 and sum(g for g, _ in route) == count and route[0][0] % 152 == 0


@pytest.mark.parametrize("k,count,cluster,variant,name",
                         [(2, 1, "auto", 2, "team"), (4, 5, "auto", 2, "team"), (8, 1, "auto", 2, "team"),
                          (2, 1, "auto", 0, "team"), (2, 4096, "auto", 2, "warp"), (4, 4096, "auto", 0, "variant"),
                          (2, 1, "off", 2, "warp"), (8, 310, "off", 2, "warp"), (2, 5, "off", 0, "variant"),
                          (2, 160, "on", 2, "team"), (8, 40, "on", 0, "team")])
def test_other_routes(contexts, k, count, cluster, variant, name):
    ctx = contexts(k)
    ctx.set_cluster(cluster)
    ctx.set_variant(variant)
    assert ctx.route(count)[0][1] == name


@pytest.mark.parametrize("cluster,variant,name", [("auto", 2, "small"), ("off", 2, "small"), ("off", 0, "variant"),
                                                  ("on", 2, "cluster")])
def test_n256(contexts, cluster, variant, name):
    ctx = contexts(2, W.toy_params)
    ctx.set_cluster(cluster)
    ctx.set_variant(variant)
    assert ctx.route(24) == [(24, name)]
