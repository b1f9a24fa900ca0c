"""An update whose synapses do not fit reports CAPACITY and changes nothing, in both forms
(one cluster kernel, general kernels): the vacancies, the store (empty, or with synapses in
it) and the count stay, and a later update that fits works."""
import numpy as np
import pytest

from gpu_common import dev
from paper_2509_26193_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("filled", [False, True])
def test_overflowing_update_changes_nothing(filled, general):
    from paper_2509_26193_gb300 import relearn as R
    net = workloads.uniform_cube(n=900, seed=62)
    n = net.n
    few = np.zeros(n, np.int32)
    few[::9] = 1  # 100 searches
    cap = 300
    ctx = R.relearn_create(n, cap, 8 * n)
    R.relearn_debug_no_clusters(ctx, general)
    R.relearn_build_octree(ctx, dev(net.x), dev(net.y), dev(net.z))
    typ = dev(net.type)

    def update(ax, de, step):
        R.relearn_update_connectivity(ctx, R.params(net.sigma, net.theta, net.seed, step), ax, de,
                                      typ)

    ax, de = dev(few), dev(net.vac_de + 1)
    if filled:
        update(ax, de, 0)
    before = R.relearn_get_synapses(ctx)
    assert (len(before[0]) > 0) == filled
    big_ax, big_de = dev(net.vac_ax + 1), dev(net.vac_de + 1)
    update(big_ax, big_de, 1)
    status, _ = R.relearn_last_error(ctx)
    assert status == R.ERR_CAPACITY
    assert np.array_equal(big_ax.cpu().numpy(), net.vac_ax + 1)
    assert np.array_equal(big_de.cpu().numpy(), net.vac_de + 1)
    after = R.relearn_get_synapses(ctx)
    assert all(np.array_equal(a, b) for a, b in zip(after, before))
    # one that fits, in the same context
    ax, de = dev(few), dev(net.vac_de + 1)
    update(ax, de, 2)
    st = R.relearn_get_last_stats(ctx)
    src, tgt, sign = R.relearn_get_synapses(ctx)
    assert st["formed"] > 0 and st["synapses"] == len(src) == len(before[0]) + st["formed"]
    assert few.sum() - ax.cpu().numpy().sum() == st["formed"]
    assert (net.vac_de + 1).sum() - de.cpu().numpy().sum() == st["formed"]
    ctx.close()
