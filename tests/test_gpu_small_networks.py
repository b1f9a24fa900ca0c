"""Networks of at most 40,960 neurons run each pass as one cluster kernel (cluster.cuh).
The same calls on a context whose capacity for searches keeps it on the general kernels
give the same integers, at the edges of the cluster's tiles and of the rule."""
import numpy as np
import pytest

from gpu_common import dev
from paper_2509_26193_gb300 import workloads

pytestmark = pytest.mark.gpu

SMALL = 40960


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()


def _run(net, general, max_synapses=0, offsets=None, typed=False):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    n = net.n
    q = int(net.vac_ax.sum())
    searches = 8 * SMALL + 1 if general else min(2 * q + 64, 8 * SMALL)
    cap = max_synapses or 2 * q + 64
    ctx = (R.relearn_create_batched(n, cap, len(offsets) - 1, searches) if offsets is not None
           else R.relearn_create(n, cap, searches))
    x, y, z, typ = dev(net.x), dev(net.y), dev(net.z), dev(net.type)
    ax, de = dev(net.vac_ax), dev(net.vac_de)
    di = dev(net.vac_de[::-1].copy())
    inp = torch.zeros(n, dtype=torch.int32, device="cuda")
    rate = dev(np.linspace(0.0, 1.0, n).astype(np.float32))
    out = []
    if offsets is not None:
        R.relearn_build_octree_batch(ctx, offsets, x, y, z)
    else:
        R.relearn_build_octree(ctx, x, y, z)
    for step in range(3):
        p = R.params(net.sigma, net.theta, net.seed, step)
        if typed:
            st = R.relearn_update_connectivity_typed(ctx, p, ax, de, di, typ, stats=True)
        else:
            st = R.relearn_update_connectivity(ctx, p, ax, de, typ, stats=True)
        out += [st[k] for k in ("searches", "failed", "requests_declined", "formed", "synapses")]
        out += list(R.relearn_get_requests(ctx))
        R.relearn_deliver_spikes(ctx, dev(workloads.spikes(n, net.seed, step, 0.3)), inp)
        out.append(inp.cpu().numpy())
        R.relearn_deliver_rates(ctx, rate, net.seed, step, inp)
        out.append(inp.cpu().numpy())
        if step == 1:
            out += list(R.relearn_get_synapses(ctx))  # the store is canonical from here on
        ra, rd = workloads.retractions(n, net.seed, step, 1.5)
        out.append(R.relearn_delete_synapses(ctx, p, dev(ra), dev(rd), ax, de, count=True))
        out += list(R.relearn_get_synapses(ctx)) + [ax.cpu().numpy(), de.cpu().numpy()]
    tree = R.relearn_get_tree(ctx)
    out += [tree[k] for k in sorted(tree)]
    ctx.close()
    return out


def _same(a, b):
    assert len(a) == len(b)
    for u, v in zip(a, b):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("n", [1, 2, 33, 511, 513, 8192, 8193, 16385, SMALL, SMALL + 1])
def test_cluster_kernels_equal_the_general_ones(n):
    net = workloads.gaussian_clusters(n=n, clusters=min(n, 3), side=1500.0, std=120.0, seed=60 + n,
                                      sigma=300.0)
    _same(_run(net, False), _run(net, True))


@pytest.mark.parametrize("typed", [False, True])
def test_networks_of_one_batch_and_typed_pools(typed):
    net = workloads.uniform_cube(n=2500, seed=61)
    _same(_run(net, False, offsets=[0, 1, 700, 2500], typed=typed),
          _run(net, True, offsets=[0, 1, 700, 2500], typed=typed))


@pytest.mark.parametrize("general", [False, True])
def test_overflowing_store_applies_nothing(general):
    from paper_2509_26193_gb300 import relearn as R
    net = workloads.uniform_cube(n=900, seed=62)
    with pytest.raises(R.RelearnError) as e:
        _run(net, general, max_synapses=50)
    assert e.value.status == R.ERR_CAPACITY
