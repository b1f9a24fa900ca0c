"""Hubs in small networks: the cluster kernels rank rows of more than 256 requests or
synapses by sorted runs of 512 entries. The same integers as the general kernels, at the
edges of the rule and of the runs, with duplicates and mixed signs in a row."""
import numpy as np
import pytest

from gpu_common import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()


def _context(n, cap, general, seed):
    from paper_2509_26193_gb300 import relearn as R
    rng = np.random.default_rng(seed)
    ctx = R.relearn_create(n, cap, cap)
    R.relearn_debug_no_clusters(ctx, general)
    R.relearn_build_octree(ctx, *(dev((rng.random(n) * 900.0).astype(np.float32))
                                  for _ in range(3)))
    return R, ctx


@pytest.mark.parametrize("n,hubs", [(257, [1]), (258, [100]), (2000, [1, 255, 256, 257]),
                                    (3000, [513, 900, 2999]), (9000, [40, 3000, 5000]),
                                    (40960, [700, 20000])])
def test_acceptance_at_over_requested_hubs(n, hubs):
    def run(general):
        R, ctx = _context(n, 2 * n + 64, general, n)
        ax = dev(np.full(n, 2 if n <= 9000 else 1, np.int32))
        de = np.zeros(n, np.int32)
        de[np.linspace(3, n - 1, len(hubs)).astype(int)] = hubs
        de = dev(de)
        st = R.relearn_update_connectivity(ctx, R.params(5000.0, 0.5, 7, 1), ax, de,
                                           dev((np.arange(n) % 5 == 0).astype(np.uint8)),
                                           stats=True)
        out = [st[k] for k in ("searches", "failed", "requests_declined", "formed")]
        out += [*R.relearn_get_requests(ctx), *R.relearn_get_synapses(ctx), ax.cpu().numpy(),
                de.cpu().numpy()]
        ctx.close()
        return out

    got, want = run(False), run(True)
    assert want[2] > 0 and want[3] > 0
    assert all(np.array_equal(a, b) for a, b in zip(got, want))


def _store(degrees, n, inward, seed):
    """Rows of the given degrees around distinct hubs (targets drawn with repeats), the rest
    sparse; the sign follows the target's parity, so that a row holds both."""
    rng = np.random.default_rng(seed)
    hub = np.repeat(np.linspace(5, n - 2, len(degrees)).astype(int), degrees)
    other = rng.integers(0, n, len(hub))
    a, b = np.concatenate([hub, rng.integers(0, n, n // 2)]), np.concatenate(
        [other, rng.integers(0, n, n // 2)])
    src, tgt = (b, a) if inward else (a, b)
    order = rng.permutation(len(src))
    src, tgt = src[order].astype(np.int32), tgt[order].astype(np.int32)
    return src, tgt, np.where(tgt & 1, 1, -1).astype(np.int8)


@pytest.mark.parametrize("inward", [False, True])
@pytest.mark.parametrize("n,degrees", [(50, [255, 256, 257, 511, 512, 513]),
                                       (3000, [1023, 1024, 1025, 1500]), (40960, [9000, 300])])
def test_order_and_deletion_of_hub_rows(n, degrees, inward):
    src, tgt, sign = _store(degrees, n, inward, n)
    m = len(src)
    rng = np.random.default_rng(n + 1)
    ra, rd = rng.integers(0, 3, n).astype(np.int32), rng.integers(0, 3, n).astype(np.int32)
    for h in np.linspace(5, n - 2, len(degrees)).astype(int):
        ra[h] = rd[h] = 100

    def run(general):
        R, ctx = _context(n, m + 64, general, n)
        zero = lambda: dev(np.zeros(n, np.int32))
        ax, de = zero(), zero()
        R.relearn_set_synapses(ctx, src, tgt, sign)
        out = []
        for step in range(2):  # an update that forms nothing: the order is formed anew
            prm = R.params(5000.0, 0.5, 7, step)
            R.relearn_update_connectivity(ctx, prm, zero(), zero(), dev(np.zeros(n, np.uint8)))
            out.append(R.relearn_delete_synapses(ctx, prm, dev(ra), dev(rd), ax, de, count=True))
        out += [*R.relearn_get_synapses(ctx), ax.cpu().numpy(), de.cpu().numpy()]
        ctx.close()
        return out

    got, want = run(False), run(True)
    assert want[0] > 0
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
