"""The training kernels at the sizes where their split of the work can go wrong.

- Loss and gradient against the oracle's FP64 ones for sets of every width around the groups of four
  rows and the 32 rows of a warp, and for more sets than one launch has warps (a warp then takes
  several). A sum of K FP32 products is within K 2^-23 of its terms' sizes (K is 32 per unit, and the
  terms of a set's rows and of the sets are added one after the other): 1e-4 of the largest gradient
  covers the cancellation in it, as in the other tests of the gradient.
- Training is the same bit for bit when repeated, also when the losses of more steps than there are
  training queries are asked for, and its last step's loss is that of the weights before it.
"""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [list(range(2, 65)), [64] * 3, [2], [3, 64, 33] * 1700])
def test_loss_grad_for_ragged_sets(sbh, oracle_mod, sizes):
    import torch
    rng = np.random.default_rng(len(sizes))
    w = rng.normal(scale=0.3, size=oracle_mod.MLP_NPARAM).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = rng.normal(size=(off[-1], 6)).astype(np.float32)
    t = rng.random(off[-1]).astype(np.float32)
    net = sbh.sbh_mlp_create(0)
    sbh.sbh_mlp_set_weights(net, w)
    loss, grad = sbh.sbh_mlp_loss_grad(net, dev(x), dev(t), torch.from_numpy(off).cuda())
    ref_loss, ref_g = oracle_mod.mlp_loss_grad(w.astype(np.float64), x.astype(np.float64), t.astype(np.float64), off)
    assert abs(float(loss.item()) - ref_loss) <= 1e-4 * abs(ref_loss)
    g = grad.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(g - ref_g)) <= 1e-4 * np.max(np.abs(ref_g)), np.max(np.abs(g - ref_g)) / np.max(np.abs(ref_g))


@pytest.mark.parametrize("nq,steps", [(1, 5), (3, 7), (40, 12)])
def test_training_repeats(sbh, nq, steps):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nq)
    p = torch.rand(3000, 3, generator=g, device="cuda")
    q = torch.rand(nq, 3, generator=g, device="cuda")
    tree = sbh.sbh_build(p, torch.ones(3000, device="cuda"))
    got = []
    for k in (steps, steps, steps - 1):
        net = sbh.sbh_mlp_create(3)
        losses = np.asarray(sbh.sbh_mlp_train(net, tree, q, "coulomb", 1.0, k))
        got.append((losses, sbh.sbh_mlp_get_weights(net)[0]))
    assert got[0][0].shape == (steps,) and np.all(np.isfinite(got[0][0]))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0][:-1], got[2][0]) and not np.array_equal(got[0][1], got[2][1])


@pytest.mark.parametrize("kind", ["coulomb", "winding"])
def test_single_points_have_no_residual(sbh, kind):
    """A child that is one source is its own centre of mass: its target is zero exactly (with normals along
    an axis, so that the dipole m n is exact), and a set of such children then has uniform targets."""
    import torch
    rng = np.random.default_rng(9)
    n = 5000
    p = rng.random((n, 3)).astype(np.float32)
    w = (rng.random(n) + 0.5).astype(np.float32)
    v = np.zeros((n, 3), np.float32)
    v[np.arange(n), rng.integers(0, 3, n)] = 1.0
    tree = sbh.sbh_build(dev(p), dev(w), dev(v) if kind == "winding" else None)
    ex = sbh.sbh_tree_export(tree, 0)
    nodes = [u for u in range(len(ex["nchild"])) if 2 <= ex["nchild"][u] <= 64
             and np.all(ex["nchild"][ex["first_child"][u]:ex["first_child"][u] + ex["nchild"][u]] == 0)][:300]
    assert len(nodes) > 50
    q = rng.random((len(nodes), 3)).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(ex["nchild"][nodes])]).astype(np.int64)
    _, targets = sbh.sbh_mlp_dataset(tree, dev(q), torch.arange(len(nodes), dtype=torch.int32, device="cuda"),
                                     torch.tensor(nodes, dtype=torch.int32, device="cuda"), torch.from_numpy(off).cuda(), kind)
    assert bool((targets == 0).all())
