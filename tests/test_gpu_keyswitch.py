"""The key switch against its definition (Sec. 3.2) in numpy, word for word.

Counts around the matrix-product kernel's groups of 128 and 256 gates, mask
dimensions around its 85-word column tiles, one and many parties, digit words
at their extremes; and the SIMT kernels on parameters the product kernel does
not take (t = 7 digits), below and above their batch threshold."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def reference(P, ks, ext):
    """ext [count][k N + 1] -> [count][k n + 1]: round to t digits of 2 bits, add the selected rows."""
    n, N, k, t = P["n"], P["N"], P["k"], P["t"]
    out = np.zeros((len(ext), k * n + 1), np.uint32)
    out[:, -1] = ext[:, -1]
    for i in range(k):
        a = ext[:, i * N:(i + 1) * N] + np.uint32(1 << (31 - 2 * t))
        for g in range(len(ext)):
            acc = np.zeros(n + 1, np.uint32)
            for lv in range(t):
                d = (a[g] >> np.uint32(30 - 2 * lv)) & 3
                for v in (1, 2, 3):
                    acc += ks[i][d == v, lv, v - 1].sum(axis=0, dtype=np.uint32)
            out[g, i * n:(i + 1) * n] = acc[:-1]
            out[g, -1:] += acc[-1:]
    return out


def run(P, count, seed):
    import torch
    from paper_2205_05825_gb300 import binding as B
    ctx = B.Context(P, W.CRS_SEED, device=0)
    for p, s in enumerate(W.party_seeds(P["k"])):
        ctx.keygen(p, s)
    ks = [ctx.export_party(p, ("ks",))["ks"] for p in range(P["k"])]
    r = np.random.default_rng(seed)
    ext = r.integers(0, 1 << 32, size=(count, ctx.E), dtype=np.uint32)
    ext[0] = 0xFFFFFFFF  # rounds up past the last digit: every digit 0
    ext[-1, ::2] = 0xFFFF7FFF  # every digit 3
    ext[-1, 1::2] = 0x55550000  # every digit 1
    out = torch.full((count, ctx.W), -1, dtype=torch.int32, device="cuda")
    ctx.stage_keyswitch(torch.from_numpy(ext.view(np.int32)).cuda(), out)
    ctx.sync()
    rows = sorted({0, count // 2, count - 1, min(count - 1, 127), min(count - 1, 128), min(count - 1, 255)})
    got = out.cpu().numpy().view(np.uint32)[rows]
    ctx.close()
    assert np.array_equal(got, reference(P, ks, ext[rows]))


@pytest.mark.parametrize("n,k,count", [(24, 1, 1), (24, 2, 128), (24, 2, 129), (24, 3, 256), (24, 2, 257), (84, 2, 3),
                                       (85, 2, 130), (169, 1, 2), (170, 1, 300), (560, 2, 37), (24, 8, 96), (24, 2, 4096)])
def test_product_kernel(n, k, count):
    run(dict(W.full_params(k), n=n), count, n + count)


@pytest.mark.parametrize("count", [1, 130])
def test_product_kernel_toy(count):
    run(W.toy_params(2), count, count)


@pytest.mark.parametrize("count", [3, 63, 64, 70])
def test_simt_kernels(count):
    run(dict(W.toy_params(2), t=7), count, count)
