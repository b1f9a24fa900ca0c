"""Group walks whose pending list runs nearly full: the subtrees without room are walked by
each source alone (walk_pending in length.cu). Few sources far apart, or many at a small
theta, lead there: a forward call of the cases below counts 7,392, 1,278 and 45,117 such
subtrees. Forward and adjoint against the FP64 oracle, with the tolerances of
test_gpu_length.py."""
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


# one source in `every` takes part: they are few, far apart, and share a group
@pytest.mark.parametrize("n,theta,every", [(140007, 0.0, 50), (200003, 0.0, 1000),
                                           (1 << 18, 0.2, 1)])
def test_crowded_pending_lists(n, theta, every):
    net = workloads.differentiable_cube(n=n, seed=95)
    net.vac_ax = np.where(np.arange(n) % every == 0, net.vac_ax, 0).astype(np.int32)
    if theta > 0:
        net, _ = _tie_free(net, theta)
    g, o = _gpu(net, theta), _orc(net, theta)
    _compare_forward(g, o, theta)
    _compare_gradient(g, o, n, floor_rule=False)
