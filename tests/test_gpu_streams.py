"""A context on a non-blocking stream, which does not wait for the legacy
stream on which plans are uploaded: the first call of each operator, by
levels, by one persistent launch and by the server, gives the words that a
context on the default stream does."""
import numpy as np
import pytest

from paper_2205_05825_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_first_calls_on_a_non_blocking_stream():
    import torch
    from paper_2205_05825_gb300 import binding as B
    P = W.toy_params(2)
    stream = torch.cuda.Stream()
    plain, other = (B.Context(P, W.CRS_SEED, device=0, stream=s) for s in (None, stream.cuda_stream))
    for p, s in enumerate(W.party_seeds(2)):
        plain.keygen(p, s)
    other.load_keys(plain.save_keys())
    r = np.random.default_rng(3)
    for bits in (2, 3, 4):
        a, b = (torch.from_numpy(plain.encrypt(j, r.integers(0, 2, 5 * bits).astype(np.uint8), 90 + j).view(np.int32)
                                 .reshape(5, bits, -1)).cuda() for j in range(2))
        want, got, again, served = (torch.zeros_like(a) for _ in range(4))
        torch.cuda.synchronize()
        plain.add_kbit(bits, a, b, want)
        plain.sync()
        other.set_circuit_exec("levels")
        other.add_kbit(bits, a, b, got)
        other.sync()
        other.set_circuit_exec("persistent")
        other.set_circuit_style("shallow")  # a plan of its own
        other.add_kbit(bits, a, b, again)
        other.sync()
        plain.set_circuit_style("shallow")
        want_s = torch.zeros_like(a)
        plain.add_kbit(bits, a, b, want_s)
        plain.sync()
        server = B.Server(other, wave_gates=64, pool_rows=4096)
        server.submit("add", bits, a, b, served)
        while not server.step():
            pass
        other.sync()
        server.close()
        for c in (plain, other):
            c.set_circuit_style("array")
        assert torch.equal(got, want) and torch.equal(again, want_s) and torch.equal(served, want_s)
    other.close()
    plain.close()
