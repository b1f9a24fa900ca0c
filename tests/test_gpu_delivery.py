"""Spike and firing-rate delivery read four synapses per thread and compare rates in whole
numbers: the same integers as the oracle's FP64 comparison, at every remainder of four, on
both sides of a rate's decision and for rates outside [0, 1]."""
import numpy as np
import pytest

import oracle
from gpu_common import dev

pytestmark = pytest.mark.gpu

SEED, STEP = 77, 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()
    oracle.build()


def _least_firing_rates(n, tgt):
    """Per source s (with the one synapse s -> tgt[s]) the least float that fires, by
    bisection over the bit patterns of the positive floats up to 1."""
    src = np.arange(n, dtype=np.int32)
    lo = np.zeros(n, np.int64)  # never fires
    hi = np.full(n, np.float32(1.0).view(np.int32), np.int64)
    syn = oracle.Synapses(n, src, np.arange(n, dtype=np.int32), np.ones(n, np.int8))
    syn.tgt[:n] = tgt  # a permutation: one synapse per target, too
    for _ in range(31):
        mid = (lo + hi) // 2
        rate = mid.astype(np.int32).view(np.float32)
        fires = oracle.deliver_rates(n, syn, rate, SEED, STEP)[tgt] == 1
        hi, lo = np.where(fires, mid, hi), np.where(fires, lo, mid)
    return hi.astype(np.int32).view(np.float32)


# 40,960 neurons and fewer run the cluster kernel, more the general one
@pytest.mark.parametrize("n", [1, 3, 1001, 40961, 50002, 50003, 50004])
def test_delivery_matches_oracle(n):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    rng = np.random.default_rng(n)
    tgt = rng.permutation(n).astype(np.int32)
    least = _least_firing_rates(n, tgt)
    below = np.nextafter(least, np.float32(0.0))
    odd = rng.choice(np.array([0.0, -0.0, -1.0, 1.0, 2.0, np.inf, -np.inf, np.nan, 1e-45,
                               1e-38, 1 - 2.0 ** -24, 2.0 ** -32, 3e38], np.float32), n)
    sign = rng.choice(np.array([-1, 1], np.int8), n)
    spiked = (rng.random(n) < 0.3).astype(np.uint8)
    ctx = R.relearn_create(n, 8 * n + 64, 8 * n + 64)
    pos = [dev(rng.random(n).astype(np.float32)) for _ in range(3)]
    R.relearn_build_octree(ctx, *pos)
    syn = oracle.Synapses(n, np.arange(n, dtype=np.int32), tgt, sign)
    R.relearn_set_synapses(ctx, *syn.arrays())
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    R.relearn_deliver_spikes(ctx, dev(spiked), out)
    assert np.array_equal(out.cpu().numpy(), oracle.deliver_spikes(n, syn, spiked))
    for rate in (least, below, odd):
        R.relearn_deliver_rates(ctx, dev(rate), SEED, STEP, out)
        assert np.array_equal(out.cpu().numpy(),
                              oracle.deliver_rates(n, syn, rate, SEED, STEP))
    ctx.close()
