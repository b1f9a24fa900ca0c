"""The forms of a delivery (one cluster kernel, or a thread per synapse or per four, also
replayed from a graph) give the oracle's integers at the edges of the rules that choose them
and at every remainder of four."""
import numpy as np
import pytest

import oracle
from gpu_common import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()
    oracle.build()


# capacity: four synapses per thread from 3,072 per SM on (466,944 on 152 SMs)
@pytest.mark.parametrize("n,synapses,capacity", [
    (1, 2, 64), (1024, 3001, 9000), (1025, 3002, 9000), (1025, 0, 9000), (9000, 60003, 327680),
    (9000, 60003, 327681), (40960, 100000, 300000), (40961, 100001, 300000),
    (40961, 100001, 700000), (50000, 100002, 700000), (50000, 100003, 700000),
    (50000, 100004, 700000)])
def test_direct_and_replayed_deliveries_match_the_oracle(n, synapses, capacity):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    rng = np.random.default_rng(n + synapses)
    src, tgt = (rng.integers(0, n, synapses).astype(np.int32) for _ in range(2))
    sign = rng.choice(np.array([-1, 1], np.int8), synapses)
    spiked, rate = (rng.random(n) < 0.4).astype(np.uint8), rng.random(n).astype(np.float32)
    ctx = R.relearn_create(n, capacity, capacity)
    R.relearn_build_octree(ctx, *(dev(rng.random(n).astype(np.float32)) for _ in range(3)))
    R.relearn_set_synapses(ctx, src, tgt, sign)
    syn = oracle.Synapses(max(synapses, 1), src, tgt, sign)
    want = (oracle.deliver_spikes(n, syn, spiked), oracle.deliver_rates(n, syn, rate, 9, 4))
    d_spiked, d_rate = dev(spiked), dev(rate)
    out = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)]

    def deliver():
        R.relearn_deliver_spikes(ctx, d_spiked, out[0])
        R.relearn_deliver_rates(ctx, d_rate, 9, 4, out[1])

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        deliver()
    for form in (deliver, graph.replay, deliver, graph.replay):
        for o in out:
            o.fill_(-5)
        form()
        for o, w in zip(out, want):
            assert np.array_equal(o.cpu().numpy(), w)
    ctx.close()
