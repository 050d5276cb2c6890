"""Many coincident points beside others: the leaf of the coincident ones takes one warp seconds, during
which every other block of the build waits for it. The wait must not give up on it.

2^23 points in one cell, half of what a cell may hold. Their leaf's FP64 sums are exact (24-bit coordinates
times at most 2^23), so it has the records of one point with all the mass, and so have the nodes above
it: Barnes-Hut, which takes so small a cell whole, must give the very results of a tree over that
point and the others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("normals", [False, True])
def test_millions_of_points_in_one_cell(sbh, normals):
    import torch
    m, others = 1 << 23, 1000
    g = torch.Generator(device="cuda").manual_seed(7)
    p = torch.rand(m + others, 3, generator=g, device="cuda")
    p[others:] = p[others].clone()
    w = torch.ones(m + others, device="cuda")
    v = torch.randn(m + others, 3, generator=g, device="cuda") if normals else None
    tree = sbh.sbh_build(p, w, v)
    q = torch.rand(64, 3, generator=g, device="cuda") + torch.tensor([2.0, 0.0, 0.0], device="cuda")
    few = w[: others + 1].clone()
    few[others] = m
    one = sbh.sbh_build(p[: others + 1].contiguous(), few)
    assert torch.equal(sbh.sbh_eval_bh(tree, q, "coulomb", 0.05, False), sbh.sbh_eval_bh(one, q, "coulomb", 0.05, False))
    for which in (0, 1):
        ex, small = sbh.sbh_tree_export(tree, which), sbh.sbh_tree_export(one, which)
        leaf = int(ex["nchild"].argmax())
        f, nc = int(ex["first_child"][leaf]), int(ex["nchild"][leaf])
        assert nc == m
        c = torch.arange(1, nc + 1, dtype=torch.float64)
        assert torch.equal(torch.from_numpy(ex["cdf"][f:f + nc]), (c / nc).float())
        # without the leaf's points the breadth-first order of nodes is that of the other tree
        assert np.array_equal(np.delete(ex["com_mass"], np.arange(f, f + nc), axis=0), small["com_mass"])
