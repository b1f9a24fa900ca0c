"""Sources whose every attraction underflows FP32 have their sums redone by two more walks of
their group (length.cu): forward and adjoint against the FP64 oracle, with about a tenth of
the sources redone, at every number of warps that share a group (8 to 34,000 neurons, 4 to
68,000, 2 to 135,000, then 1), and with all of them redone.

Tolerance: an attraction's exponent D / sigma^2 carries the relative rounding errors of D
(three roundings, 3 x 2^-24). The most isolated sources have D / sigma^2 of about 270, so an
attraction is off by up to 270 x 3 x 2^-24 = 4.8e-5, a ratio of sums of them by twice that:
1e-4 of a source's length, of the mean, of its derivative by sigma and of the position
gradient's norm. (Not of each gradient element: with sigma far below the distances, the two
parts of a term, 2 (d - l) / sigma^2 and 1 / d, nearly cancel in some elements.)"""
import numpy as np
import pytest

import oracle
from paper_2509_26193_gb300 import workloads
from test_gpu_length import _gpu, _orc

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()
    oracle.build()


def _check(net, theta):
    if theta > 0:  # without the sources that lie near a tie of the criterion
        near = _orc(net, theta, grad=False)["margin_ac"] < 1e-4
        net.vac_ax = np.where(near, 0, net.vac_ax).astype(np.int32)
    g, o = _gpu(net, theta), _orc(net, theta)
    ok = np.isfinite(o["ell"])
    assert np.array_equal(np.isfinite(g["ell"]), ok)
    assert np.abs(g["ell"][ok] / o["ell"][ok] - 1.0).max() <= TOL
    assert abs(g["mean"] / o["mean"] - 1.0) <= TOL
    assert abs(g["dsigma"] / o["dsigma"] - 1.0) <= TOL
    assert np.linalg.norm(g["g"] - o["g"]) <= TOL * np.linalg.norm(o["g"])
    return o


@pytest.mark.parametrize("n,theta", [(40, 0.0), (1000, 0.0), (1000, 0.3), (5003, 0.3),
                                     (40001, 0.3), (100003, 0.3), (150001, 0.3)])
def test_some_sources_underflow(n, theta):
    net = workloads.differentiable_cube(n=n, seed=90)
    net.sigma = 8.0  # 62 um between neighbours
    _check(net, theta)


@pytest.mark.parametrize("n", [300, 5003])
def test_all_sources_underflow(n):
    """Two slabs 800 um apart, sources in one, targets in the other, sigma 55 um: D / sigma^2
    between 211 and 270."""
    net = workloads.differentiable_cube(n=n, seed=91)
    half = n // 2
    net.x = (net.x * np.float32(100.0 / max(net.x.max(), 1.0))).astype(np.float32)
    net.y = (net.y * np.float32(30.0 / max(net.y.max(), 1.0))).astype(np.float32)
    net.z = (net.z * np.float32(30.0 / max(net.z.max(), 1.0))).astype(np.float32)
    net.x[half:] += np.float32(800.0)
    net.vac_ax[half:] = 0
    net.vac_de[:half] = 0
    net.sigma = 55.0
    net.vac_ax[:half] = 1
    _check(net, 0.0)
