"""The terms of the Barnes-Hut walk: with one source a sum is one term, which brute force forms by the same
operations on the same differences (their squares in one fused sum), so both give the same bits."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vote", [False, True])
@pytest.mark.parametrize("normals", [False, True])  # other records of the nodes
@pytest.mark.parametrize("nq", [5000, 1 << 19])
def test_coulomb_term(sbh, nq, normals, vote):
    import torch
    rng = np.random.default_rng(nq)
    p, w, v = dev(rng.random((1, 3))), dev(rng.random(1) + 0.5), dev(rng.normal(size=(1, 3)))
    q = dev(rng.random((nq, 3)) * 4 - 2)
    tree = sbh.sbh_build(p, w, v if normals else None)
    for softening in (0.0, 1e-3, 0.3):
        assert torch.equal(sbh.sbh_eval_bh(tree, q, "coulomb", 0.5, vote, softening=softening),
                           sbh.sbh_eval_brute(p, w, q, "coulomb", softening=softening))


@pytest.mark.parametrize("vote", [False, True])
@pytest.mark.parametrize("kind,normals", [("coulomb", False), ("coulomb", True), ("winding", True), ("smoothdist", False),
                                          ("affine", True)])
def test_few_queries_walk_as_many_do(sbh, kind, normals, vote):
    """Up to 512 queries to an SM a walk asks for its nodes ahead: the same sums as in a larger call."""
    import torch
    rng = np.random.default_rng(8)
    n = 20000
    p = rng.random((n, 3)).astype(np.float32)
    p[15000:] = p[15000]  # a leaf of 5,000 points
    w, v = rng.random(n) + 0.5, rng.normal(size=(n, 3))
    tree = sbh.sbh_build(dev(p), dev(w), dev(v) if normals else None, leaf_size=3)
    few = 512 * torch.cuda.get_device_properties(0).multi_processor_count
    q = dev(rng.random((few + 32, 3)) * 3 - 1)
    for theta in (0.0, 0.4, 1.1):
        m = 2048 if theta == 0.0 else few
        many = sbh.sbh_eval_bh(tree, q if m == few else q[:m].repeat(41, 1), kind, theta, vote)
        for a, b in ((0, 1), (0, 33), (0, m)):
            if vote and b % 32:  # a vote's queries are a warp's: none left out of the last one
                continue
            assert torch.equal(sbh.sbh_eval_bh(tree, q[a:b], kind, theta, vote), many[a:b])
