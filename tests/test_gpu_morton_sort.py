"""Morton codes and their stable order at the edges of the sort's forms (one cluster up to
40,960 neurons, 32,768 in a build; tiles of 2,048 keys beyond) against the oracle's codes
and a stable host sort: through the allocation-free entry point and the octree build."""
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


def _positions(n, kind):
    rng = np.random.default_rng(1000 + n)
    p = (rng.random((3, n)) * 900.0).astype(np.float32)
    if kind == "equal":        # one code: the order is the ids'
        p[:] = 250.0
        p[:, 0] = 0.0
    elif kind == "few":        # nine codes, in runs
        p[:] = np.repeat(rng.integers(0, 9, (n + 63) // 64), 64)[:n].astype(np.float32) * 100.0
    elif kind == "nan":        # coordinates that are not numbers fall into the first cell
        p[1, ::7] = np.nan
    return p


def _codes_with_nan(p):
    """The quantisation of relearn_build_octree in NumPy float32: coordinates that are not
    numbers are left out of the box and become 0 (the oracle does not define them)."""
    code = np.zeros(p.shape[1], np.uint32)
    for a in range(3):
        lo, hi = np.nanmin(p[a]), np.nanmax(p[a])
        inv = np.float32(1.0) / np.float32(hi - lo)
        t = ((p[a] - lo) * inv) * np.float32(1024.0)
        q = np.where(np.isnan(t), 0.0, np.clip(t, 0.0, 1023.0)).astype(np.uint32)
        for b in range(10):
            code |= ((q >> b) & 1) << (3 * b + a)
    return code


@pytest.mark.parametrize("n,kind", [(1, "any"), (2, "any"), (33, "any"), (513, "any"),
                                    (2047, "few"), (2049, "any"), (8193, "equal"),
                                    (32768, "any"), (32769, "nan"), (40960, "few"),
                                    (40961, "any"), (40961, "equal"), (100003, "few"),
                                    (300007, "nan"), (1 << 20, "any")])
def test_order_is_stable_by_code_then_id(n, kind):
    import torch
    from paper_2509_26193_gb300 import relearn as R
    p = _positions(n, kind)
    want = _codes_with_nan(p) if kind == "nan" else oracle.morton(p[0], p[1], p[2])[0]
    perm = np.argsort(want, kind="stable").astype(np.int32)
    x, y, z = (dev(a) for a in p)
    codes = torch.empty(n, dtype=torch.int32, device="cuda")
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    for _ in range(2):  # the second call on the first one's scratch
        R.relearn_morton_order_noalloc(x, y, z, codes, order)
        assert np.array_equal(order.cpu().numpy(), perm)
        assert np.array_equal(codes.cpu().numpy().view(np.uint32), want[perm])
    ctx = R.relearn_create(n, 16)
    R.relearn_build_octree(ctx, x, y, z)
    assert np.array_equal(R.relearn_get_tree(ctx)["perm"], perm)
    ctx.close()
