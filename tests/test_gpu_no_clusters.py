"""Where no cluster of 16 blocks can be placed, small networks run the general kernels
(relearn_debug_no_clusters stands in for such a GPU): every call gives the same result with
and without the cluster kernels, also when the form changes from call to call."""
import numpy as np
import pytest

from gpu_common import dev
from paper_2509_26193_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()


def _updates(net, off):
    """off(k): whether call k runs without cluster kernels."""
    import torch
    from paper_2509_26193_gb300 import relearn as R
    n, k = net.n, iter(range(100))
    q = int(net.vac_ax.sum())
    ctx = R.relearn_create(n, 2 * q + 64, 2 * q + 64)

    def call(f, *args, **kw):
        R.relearn_debug_no_clusters(ctx, off(next(k)))
        return f(ctx, *args, **kw)

    ax, de, typ = dev(net.vac_ax), dev(net.vac_de), dev(net.type)
    inp = torch.zeros(n, dtype=torch.int32, device="cuda")
    call(R.relearn_build_octree, dev(net.x), dev(net.y), dev(net.z))
    out = []
    for step in range(2):
        p = R.params(net.sigma, net.theta, net.seed, step)
        st = call(R.relearn_update_connectivity, p, ax, de, typ, stats=True)
        out += [st[s] for s in ("searches", "failed", "requests_declined", "formed", "synapses")]
        out += list(R.relearn_get_requests(ctx))
        call(R.relearn_deliver_spikes, dev(workloads.spikes(n, net.seed, step, 0.3)), inp)
        out.append(inp.cpu().numpy())
        ra, rd = workloads.retractions(n, net.seed, step, 1.5)
        out.append(call(R.relearn_delete_synapses, p, dev(ra), dev(rd), ax, de, count=True))
        call(R.relearn_deliver_rates, dev(np.linspace(0, 1, n).astype(np.float32)), 5, step, inp)
        out += [inp.cpu().numpy(), ax.cpu().numpy(), de.cpu().numpy()]
        out += list(R.relearn_get_synapses(ctx))
    tree = R.relearn_get_tree(ctx)
    out += [tree[s] for s in sorted(tree)]
    ctx.close()
    return out


@pytest.mark.parametrize("n", [2, 700, 9001])
def test_update_delivery_and_deletion(n):
    net = workloads.gaussian_clusters(n=n, clusters=min(n, 3), side=1500.0, std=120.0, seed=80 + n,
                                      sigma=300.0)
    want = _updates(net, lambda k: True)
    for off in (lambda k: False, lambda k: k % 2 == 0, lambda k: k % 3 != 0):
        got = _updates(net, off)
        assert len(got) == len(want)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("n", [3, 700, 9001])
def test_differentiable_form(n):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    net = workloads.differentiable_cube(n=n, seed=81)
    va, vd = dev(net.vac_ax), dev(net.vac_de)
    res = []
    for off in (True, False):
        ctx = R.relearn_create(n, 64)
        R.relearn_debug_no_clusters(ctx, off)
        R.relearn_build_octree(ctx, dev(net.x), dev(net.y), dev(net.z))
        mean = torch.empty(1, dtype=torch.float64, device="cuda")
        ell, *g = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(4))
        gs = torch.empty(1, dtype=torch.float64, device="cuda")
        R.relearn_mean_length(ctx, R.params(net.sigma, 0.3, 0, 0), va, vd, mean, ell)
        R.relearn_mean_length_backward(ctx, va, vd, *g, gsigma=gs)
        res.append([t.cpu().numpy() for t in (ell, mean, gs, *g)])
        ctx.close()
    a, b = res
    assert np.array_equal(a[0], b[0], equal_nan=True)  # each source's own sums
    # the sums over sources and the nodes' adjoints are FP64 atomics in any order (a few
    # 2^-53 of the largest), the gradient is their FP32 rounding
    for u, v in zip(a[1:3], b[1:3]):
        assert np.allclose(u, v, rtol=1e-12, atol=0.0, equal_nan=True)
    scale = max(float(np.abs(u).max()) for u in a[3:])
    for u, v in zip(a[3:], b[3:]):
        assert np.abs(u - v).max() <= 2.0 ** -23 * scale


def test_hook_needs_a_context():
    from paper_2509_26193_gb300 import relearn as R
    assert R.lib().relearn_debug_no_clusters(None, 1) == R.ERR_INVALID_ARG
