"""The Barnes-Hut walk's one-comparison test, its node records and its query order.

Every query's sum is the same FP32 terms in the same order whatever order the queries are walked in,
with or without the walk records, so results are compared bit for bit:
- a large call (walked in Morton order) against the same queries in calls too small to be reordered,
  also for queries far outside the sources' cube and on the sources;
- a call without memory for the records against one with them.
The test itself against the quotient it stands for: a walk over the exported 8-ary tree with root and
division rounded to nearest in FP32 opens the same nodes, so its FP64 sum of the Coulomb terms is the
kernel's up to the FP32 rounding of at most 500 terms (3e-6 of their sum: 2^-22 a term and the
additions' 2^-24 each, which average out).
"""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _tree(sbh, n=3000, normals=False, seed=0):
    rng = np.random.default_rng(seed)
    p = rng.random((n, 3), dtype=np.float32)
    w = rng.random(n, dtype=np.float32) + np.float32(0.5)
    v = rng.normal(size=(n, 3)).astype(np.float32) if normals else None
    return sbh.sbh_build(dev(p), dev(w), dev(v), leaf_size=3), p, w, v


@pytest.mark.parametrize("kind", ["coulomb", "winding", "smoothdist"])
@pytest.mark.parametrize("nq", [(1 << 16), (1 << 16) + 1, 100003, 1 << 19, (1 << 19) + 1, 600011])
def test_order_of_queries_changes_nothing(sbh, kind, nq):
    import torch
    tree, p, _, _ = _tree(sbh, normals=kind == "winding")
    rng = np.random.default_rng(nq)
    q = (rng.random((nq, 3)) * 3 - 1).astype(np.float32)
    q[:1000] *= 50
    q[1000:4000] = p
    Q = dev(q)
    for theta in (0.0, 0.5, 1.3):
        m = 4099 if theta == 0.0 else nq
        whole = sbh.sbh_eval_bh(tree, Q, kind, theta, False)[:m]
        parts = torch.cat([sbh.sbh_eval_bh(tree, Q[a:min(a + 5000, m)], kind, theta, False) for a in range(0, m, 5000)])
        assert torch.equal(whole, parts)


@pytest.mark.parametrize("vote", [False, True])
@pytest.mark.parametrize("nq", [70001, 600011])
def test_without_memory_for_the_records(sbh, nq, vote):
    import torch
    tree, p, w, _ = _tree(sbh, n=20000)
    Q = dev(np.random.default_rng(1).random((nq, 3), dtype=np.float32))
    want = sbh.sbh_eval_bh(tree, Q, "coulomb", 0.7, vote)
    other = sbh.sbh_build(dev(p), dev(w), leaf_size=3)
    used = sbh.sbh_memory_in_use()
    sbh.sbh_eval_bh(other, Q[:1], "coulomb", 0.7)
    full = sbh.sbh_memory_in_use() - used
    records = 32 * (2 * 20000 + 1)
    third = sbh.sbh_build(dev(p), dev(w), leaf_size=3)
    now = sbh.sbh_memory_in_use()
    sbh.sbh_set_memory_limit(now + full - 1)
    try:
        got = sbh.sbh_eval_bh(third, Q, "coulomb", 0.7, vote)
        assert sbh.sbh_memory_in_use() - now == full - records
    finally:
        sbh.sbh_set_memory_limit(0)
    assert torch.equal(got, want)


@pytest.mark.parametrize("vote", [False, True])
@pytest.mark.parametrize("nq", [1000, 70001, 600011])
def test_trees_with_normals_walk_alike(sbh, nq, vote):
    """Normals change a tree's walk records, not its nodes or its masses."""
    import torch
    plain, p, _, _ = _tree(sbh)
    other, _, _, v = _tree(sbh, normals=True)
    Q = dev(np.random.default_rng(2).random((nq, 3), dtype=np.float32))
    for kind in ("coulomb", "smoothdist"):
        assert torch.equal(sbh.sbh_eval_bh(plain, Q, kind, 0.7, vote), sbh.sbh_eval_bh(other, Q, kind, 0.7, vote))


@pytest.mark.parametrize("theta", [0.3, 0.5, 0.777, 1.0, 40.0])
def test_opening_rule_is_the_rounded_quotient(sbh, theta):
    tree, p, _, _ = _tree(sbh, n=500, seed=3)
    rng = np.random.default_rng(4)
    q = rng.random((300, 3)).astype(np.float32) * 2 - np.float32(0.5)
    got = sbh.sbh_eval_bh(tree, dev(q), "coulomb", theta, False, softening=1e-3).cpu().numpy()
    ex = sbh.sbh_tree_export(tree, 1)
    f = np.float32
    beta = f(1) / f(theta)
    pm, fc, nc, level = (ex[k] for k in ("com_mass", "first_child", "nchild", "level"))
    diam = f(1.7320508075688772) * f(ex["info"]["side"])
    for i in range(len(q)):
        total, size, stack = 0.0, 0.0, [0]
        while stack:
            v = stack.pop()
            d = pm[v, :3] - q[i]
            s = f(f(f(d[0] * d[0]) + f(d[1] * d[1])) + f(d[2] * d[2]))
            if nc[v] == 0 or f(np.sqrt(s) / f(diam * f(2.0) ** -int(level[v]))) >= beta:
                t = float(pm[v, 3]) / np.sqrt(float((d.astype(np.float64) ** 2).sum()) + 1e-6)
                total += t
                size += abs(t)
            else:
                stack.extend(range(fc[v], fc[v] + nc[v]))
        # a node opened or not opened in error changes the sum by far more than FP32 rounding of its terms
        assert abs(got[i] - total) <= 3e-6 * size
