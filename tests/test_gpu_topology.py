"""Tree topology at sizes around a block's tile (4,096 points), a warp's share (256) and their remainders,
for point sets whose nodes cross those edges: every integer array and every link equals the oracle's tree,
for both trees and leaf sizes up to the largest."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _points(kind, n, rng):
    if kind == "two":  # two far clusters: one boundary at level 0, the rest collapses deep
        p = 1e-4 * rng.random((n, 3))
        p[n // 2:] += 1.0
    elif kind == "runs":  # many points in few cells, long runs of one code
        p = (rng.integers(0, 3, (n, 3)) / 2.0) + 1e-7 * rng.integers(0, 2, (n, 3))
    elif kind == "line":  # every level populated along a line
        p = np.stack([2.0 ** -rng.uniform(0, 22, n)] * 3, 1)
    else:
        p = rng.random((n, 3))
    return p.astype(np.float32)


@pytest.mark.parametrize("leaf", [1, 3, 64])
@pytest.mark.parametrize("kind", ["uniform", "two", "runs", "line"])
@pytest.mark.parametrize("n", [1, 2, 9, 63, 64, 65, 257, 4095, 4096, 4097, 12289])
def test_topology_equals_the_oracle(sbh, oracle_mod, kind, n, leaf):
    rng = np.random.default_rng(n)
    pts = _points(kind, n, rng)
    w = rng.uniform(0.5, 1.5, n).astype(np.float32)
    t = sbh.sbh_build(dev(pts), dev(w), leaf_size=leaf)
    sbh.sbh_eval_bh(t, dev(pts[:1]), "coulomb", theta=0.5)  # builds the 8-ary tree
    for which, d in ((0, 4), (1, 2)):
        o = oracle_mod.Tree(pts, w, leaf_size=leaf, d=d)
        g, e = sbh.sbh_tree_export(t, which), o.export()
        assert g["info"]["n_nodes"] == e["begin"].shape[0]
        for k in ("perm", "begin", "end", "first_child", "nchild", "level"):
            np.testing.assert_array_equal(g[k], e[k], err_msg=f"{k} of tree {which}")
        par = np.full(e["begin"].shape[0], -1)
        for v in np.nonzero(e["nchild"])[0]:
            par[e["first_child"][v]:e["first_child"][v] + e["nchild"][v]] = v
        np.testing.assert_array_equal(g["parent"], par)
        np.testing.assert_array_equal(g["com_mass"][:, 3], e["mass"].astype(np.float32))
