"""The group walk of the differentiable form (length.cu) at the sizes where it can go
wrong: groups of one warp and less, shared groups, families of more than eight children
(buckets), exponents that underflow. Against the FP64 oracle with the tolerances of
test_gpu_length.py (1e-5 of each source's length, and of each gradient element's terms)."""
import numpy as np
import pytest

import oracle
from paper_2509_26193_gb300 import workloads
from test_gpu_length import _compare_forward, _compare_gradient, _gpu, _orc, _tie_free

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()
    oracle.build()


def _buckets(n):
    """Three of four neurons on seven points (families of many leaves), the rest uniform."""
    net = workloads.differentiable_cube(n=n, seed=41)
    rng = np.random.default_rng(42)
    at = rng.random((7, 3)) * 700.0
    own = rng.integers(0, 28, n)
    for k, a in enumerate((net.x, net.y, net.z)):
        a[own < 21] = at[own[own < 21] % 7, k].astype(np.float32)
    return net


@pytest.mark.parametrize("theta", [0.0, 0.3])
@pytest.mark.parametrize("n", [3, 31, 33, 70, 257, 1025, 5003])
def test_ragged_sizes(n, theta):
    net = workloads.differentiable_cube(n=n, seed=40 + n)
    if theta > 0:
        net, _ = _tie_free(net, theta)
    g, o = _gpu(net, theta), _orc(net, theta)
    _compare_forward(g, o, theta)
    _compare_gradient(g, o, n, floor_rule=False)


@pytest.mark.parametrize("theta", [0.0, 0.5])
@pytest.mark.parametrize("n", [60, 1500])
def test_buckets_of_many_leaves(n, theta):
    net = _buckets(n)
    if theta > 0:
        net, _ = _tie_free(net, theta)
    g, o = _gpu(net, theta), _orc(net, theta)
    _compare_forward(g, o, theta)
    _compare_gradient(g, o, n, floor_rule=False)


def test_underflowing_attractions():
    """Every attraction of a distant group underflows FP32 (its sums are redone with the
    exponents shifted): 40 sources 20 sigma from the nearest candidate."""
    net = workloads.differentiable_cube(n=600, seed=43)
    net.sigma = 40.0
    net.x[:40] += 2000.0
    net.vac_de[:40] = 0
    net.vac_ax[:40] = 2
    _compare_forward(_gpu(net, 0.0, grad=False), _orc(net, 0.0, grad=False), 0.0)
