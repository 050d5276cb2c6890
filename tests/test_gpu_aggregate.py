"""The tree's records where their kernel's split can go wrong: leaves with more children than the eight
lanes of a node, than the 64 prefix sums kept (duplicates), equal masses (quotients on the middle of
two floats), weights and coordinates at FP32's limits, and generations of one node and of thousands.

Each record is defined by FP64 sums in the children's order and quotients rounded to FP32, which numpy
does here from the exported tree, so records are compared bit for bit.
"""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _points(case):
    rng = np.random.default_rng(11)
    if case == "one":
        return rng.random((1, 3)), np.ones(1)
    if case == "duplicates":  # leaves at the deepest level with 9, 64, 65, 200 and 1,000 points
        return np.repeat(rng.random((5, 3)), [9, 64, 65, 200, 1000], axis=0), rng.random(1338) + 0.5
    if case == "equal":
        return rng.integers(0, 1 << 20, (20000, 3)) / float(1 << 20), np.ones(20000)
    if case == "range":  # masses over 2^-140 .. 2^100, coordinates 2^-130 .. 1 with zeros
        p = rng.random((3000, 3)) * 2.0 ** -rng.integers(0, 130, (3000, 3)) * (rng.random((3000, 3)) < 0.8)
        return p, 2.0 ** rng.integers(-140, 100, 3000)
    return rng.normal(size=(30011, 3)), rng.random(30011) + 0.5


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("leaf", [1, 7])
@pytest.mark.parametrize("case", ["one", "duplicates", "equal", "range", "normal"])
def test_records_are_the_rounded_fp64_sums(sbh, case, leaf, which):
    p, w = (np.asarray(x, np.float32) for x in _points(case))
    v = np.random.default_rng(5).normal(size=p.shape).astype(np.float32)
    v[::3, 0] = 0.0
    tree = sbh.sbh_build(dev(p), dev(w), dev(v), leaf_size=leaf)
    sbh.sbh_eval_bh(tree, dev(p[:1]), "coulomb")
    ex = sbh.sbh_tree_export(tree, which)
    fc, nc, parent, perm = ex["first_child"], ex["nchild"], ex["parent"], ex["perm"]
    N = len(fc)
    a = np.zeros((N, 7))
    point = nc == 0
    i = perm[ex["begin"][point]]
    W = w.astype(np.float64)[i]
    a[point] = np.column_stack([W, W[:, None] * p[i].astype(np.float64), W[:, None] * v[i].astype(np.float64)])
    pre = np.zeros(N)
    for u in range(N - 1, -1, -1):  # children have larger ids
        if nc[u]:
            s = np.zeros(7)
            for c in range(fc[u], fc[u] + nc[u]):
                s = s + a[c]
                pre[c] = s[0]
            a[u] = s
    com = np.where(point[:, None], 0, a[:, 1:4] / a[:, :1]).astype(np.float32)
    com[point] = p[i]
    dip = a[:, 4:].astype(np.float32)
    dip[point] = w[i, None] * v[i]
    cdf = np.ones(N, np.float32)
    if N > 1:
        cdf[1:] = (pre[1:] / a[parent[1:], 0]).astype(np.float32)
        cdf[(fc + nc - 1)[~point]] = 1.0
    assert np.array_equal(ex["com_mass"][:, :3], com) and np.array_equal(ex["com_mass"][:, 3], a[:, 0].astype(np.float32))
    assert np.array_equal(ex["dipole"], dip)
    assert np.array_equal(ex["cdf"], cdf)
    for u in range(0, N, max(1, N // 500)):
        if nc[u]:
            f, k = fc[u], int(nc[u])
            uj = -(-(np.arange(k, dtype=np.int64) << 24) // k) * 2.0 ** -24
            want = (cdf[f:f + k - 1][None, :].astype(np.float64) <= uj[:, None]).sum(1)
            assert np.array_equal(ex["guide"][f:f + k], want.astype(np.uint8))
