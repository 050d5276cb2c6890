"""A call that is walked in Morton order against the same queries in calls too small to be sorted, on both
sides of the line between them (2^19 queries) and past a sort's tile and a warp there, on a tree of many
clustered sources: the same sums in the same order, so the same bits."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [(1 << 19) - 1, 1 << 19, (1 << 19) + 31, (1 << 20) + 17])
@pytest.mark.parametrize("kind", ["coulomb", "winding", "smoothdist"])
def test_sorted_walk_of_a_clustered_tree(sbh, kind, nq):
    import torch
    rng = np.random.default_rng(nq)
    n = 1 << 18
    centre = rng.random((300, 3))
    p = (centre[rng.integers(0, 300, n)] + rng.normal(size=(n, 3)) * rng.choice([1e-1, 1e-2, 1e-4], (n, 1))).astype(np.float32)
    p[::7] = p[rng.integers(0, n, p[::7].shape[0])]  # some of them twice
    w = rng.uniform(0.5, 1.5, n).astype(np.float32)
    v = rng.normal(size=(n, 3)).astype(np.float32) if kind == "winding" else None
    tree = sbh.sbh_build(dev(p), dev(w), dev(v), leaf_size=2)
    q = (p[rng.integers(0, n, nq)] + rng.normal(size=(nq, 3)) * rng.choice([0.0, 1e-3, 1.0], (nq, 1))).astype(np.float32)
    q = dev(q)
    whole = sbh.sbh_eval_bh(tree, q, kind, 0.9, False)
    step = 1 << 18
    parts = torch.cat([sbh.sbh_eval_bh(tree, q[a:a + step], kind, 0.9, False) for a in range(0, nq, step)])
    assert torch.equal(whole, parts)
