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
