"""The bounding boxes of a batch are folded in chunks that cross network borders: every
network of a batch has the tree of its own single build, at sizes around a chunk's rows
and with chunks that hold several networks or lie inside one."""
import numpy as np
import pytest

from gpu_common import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2509_26193_gb300 import build
    build.build()


@pytest.mark.parametrize("sizes", [[1, 2, 31, 32, 33, 127, 128, 129, 5, 1, 1],
                                   [70001, 3, 40000, 1, 90000, 64],
                                   [200, 1500000, 7]])
def test_batch_trees_are_the_single_ones(sizes):
    from paper_2509_26193_gb300 import relearn as R
    rng = np.random.default_rng(sum(sizes))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    # boxes of different places and sizes, of either sign
    at = rng.uniform(-5e3, 5e3, (3, len(sizes)))
    edge = rng.uniform(10.0, 4e3, (3, len(sizes)))
    p = (rng.random((3, n)) * np.repeat(edge, sizes, 1) + np.repeat(at, sizes, 1))
    p = p.astype(np.float32)
    if sizes[0] > 1:
        p[1, off[1] - 1] = np.nan  # left out of its network's box
    ctx = R.relearn_create_batched(n, 64, len(sizes), 64)
    R.relearn_build_octree_batch(ctx, off, *(dev(a) for a in p))
    batch = R.relearn_get_tree(ctx)
    ctx.close()
    nodes = 0
    for b, k in enumerate(sizes):
        one = R.relearn_create(k, 64, 64)
        R.relearn_build_octree(one, *(dev(a[off[b]:off[b + 1]].copy()) for a in p))
        t = R.relearn_get_tree(one)
        one.close()
        m = len(t["depth"])
        for key in ("depth", "size", "is_leaf"):
            assert np.array_equal(batch[key][nodes:nodes + m], t[key]), (b, key)
        assert np.array_equal(batch["perm"][off[b]:off[b + 1]] - off[b], t["perm"]), b
        nodes += m
    assert nodes == len(batch["depth"])
