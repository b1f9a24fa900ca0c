"""What a pass of the differentiable form sets up (active sources, family order) is one
cluster kernel up to 16,384 neurons and a chain of kernels above: values and gradients at
the sizes around its tiles, its blocks and that line, against the FP64 oracle.

theta = 0 (every candidate a leaf: no criterion ties). Tolerance: a source's length and a
gradient's rounding errors are a few FP32 roundings of its terms, 1e-5 of the sum of their
magnitudes, as derived in test_gpu_length.py."""
import numpy as np
import pytest

import oracle
from gpu_common import dev
from paper_2509_26193_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("n", [2, 31, 511, 8193, 16384, 16385])
def test_setup_matches_oracle(n):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    net = workloads.differentiable_cube(n=n, seed=n)
    net.vac_ax[1::3] = 0  # sources and targets with gaps
    net.vac_de[::5] = 0
    net.vac_ax[0], net.vac_de[-1] = 1, 1
    ctx = R.relearn_create(n, 64)
    va, vd = dev(net.vac_ax), dev(net.vac_de)
    prm = R.params(net.sigma, 0.0, 0, 0)
    t = oracle.Tree(net.x, net.y, net.z)
    t.reduce(net.vac_de)
    o = oracle.mean_length(t, net.sigma, 0.0, net.vac_ax, net.vac_de, grad=True, threads=16)
    t.close()
    mean = torch.empty(1, dtype=torch.float64, device="cuda")
    ell = torch.empty(n, dtype=torch.float32, device="cuda")
    gs = torch.empty(1, dtype=torch.float64, device="cuda")
    R.relearn_build_octree(ctx, *(dev(a) for a in (net.x, net.y, net.z)))
    for _ in range(2):  # the second pass meets the first one's scratch
        R.relearn_mean_length(ctx, prm, va, vd, mean, ell)
        g = [torch.full((n,), 7.0, dtype=torch.float32, device="cuda") for _ in range(3)]
        R.relearn_mean_length_backward(ctx, va, vd, *g, gsigma=gs)
        assert abs(float(mean.item()) - o["mean"]) <= 1e-5 * o["mean"]
        e = ell.cpu().numpy().astype(np.float64)
        ok = np.isfinite(o["ell"])
        assert np.array_equal(np.isfinite(e), ok)
        assert (np.abs(e[ok] - o["ell"][ok]) <= 1e-5 * o["ell"][ok]).all()
        gg = np.stack([a.cpu().numpy() for a in g], 1).astype(np.float64)
        assert (np.abs(gg - o["g"]) <= 1e-5 * np.maximum(o["g_abs"], 1e-300)).all()
        # (a single candidate has dsigma = 0: a covariance of rounding errors)
        assert abs(float(gs.item()) - o["dsigma"]) <= 1e-5 * (abs(o["dsigma"])
                                                              + o["mean"] / net.sigma)
    ctx.close()
