"""Brute force where its work is split: source counts around a pair, a warp's share, a tile and a
cluster's tiles, query counts around a group and around the change from two queries a lane to four.
The reference is the FP64 sum of the same terms on the host; the tolerance is relative to the sum of
the terms' magnitudes: each FP32 term is within about ten roundings (2^-24 each) of its value and an
FP32 partial adds up 256 of them at most in two halves, the rest is FP64: 2e-6 leaves room."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu
ALPHA, EPS, G = 30.0, 1e-3, (0.3, -0.2, 0.7)


def _reference(kind, p, w, v, q):
    """(value, gradient, magnitude of the value's terms, magnitude of the gradient's terms), FP64"""
    p, w, q = p.astype(np.float64), w.astype(np.float64), q.astype(np.float64)
    d = p[None] - q[:, None]
    r2 = (d ** 2).sum(2)
    if kind == "coulomb":
        t = w / np.sqrt(r2 + EPS ** 2)
        g = t / (r2 + EPS ** 2)
        return t.sum(1), (g[..., None] * d).sum(1), np.abs(t).sum(1), np.abs(g[..., None] * d).sum(1)
    if kind == "winding":
        nv = v.astype(np.float64) * w[:, None]
        r = np.sqrt(r2)
        dn = (d * nv[None]).sum(2)
        t = dn / r ** 3 / (4 * np.pi)
        g = (3 * (dn / r ** 5)[..., None] * d - nv[None] / r[..., None] ** 3) / (4 * np.pi)
        nn = np.linalg.norm(nv, axis=1)[None]
        return t.sum(1), g.sum(1), (nn / r2 / (4 * np.pi)).sum(1), np.repeat((4 * nn / r ** 3 / (4 * np.pi)).sum(1)[:, None], 3, 1)
    if kind == "smoothdist":
        r = np.sqrt(r2)
        ref = r.min(1, keepdims=True)
        e = w * np.exp(-ALPHA * (r - ref))
        s = e.sum(1)
        g = -(e / s[:, None] / r)[..., None] * d
        # d = ref - log(s) / alpha: a distance's rounding goes straight into it; a term's exponent alpha (r - ref),
        # up to about 20 where it counts, turns an FP32 rounding of it into 20 of the term
        return ref[:, 0] - np.log(s) / ALPHA, g.sum(1), 1 + np.abs(ref[:, 0]), np.full_like(g.sum(1), 20.0)
    h = 1 + (d * np.array(G)).sum(2)
    return (w * h).sum(1), np.broadcast_to(-(w[:, None] * np.array(G)).sum(0), (q.shape[0], 3)), (w * (1 + np.abs(d).sum(2))).sum(1), w.sum()


@pytest.mark.parametrize("n,nq", [(1, 1), (2, 63), (3, 65), (15, 64), (17, 129), (1023, 33), (1024, 1), (1025, 5),
                                  (2047, 40), (2049, 128), (8191, 31), (8193, 65), (33, 152 * 128 - 1),
                                  (1027, 152 * 128 + 1)])
@pytest.mark.parametrize("kind", ["coulomb", "winding", "smoothdist", "affine"])
def test_brute_splits_add_up(sbh, kind, n, nq):
    rng = np.random.default_rng(n + nq)
    p, q = rng.random((n, 3)).astype(np.float32), rng.random((nq, 3)).astype(np.float32)
    w = rng.uniform(0.5, 1.5, n).astype(np.float32)
    v = rng.normal(size=(n, 3)).astype(np.float32)
    kw = dict(kernel=kind, normals=dev(v), softening=EPS, alpha=ALPHA, affine=G)
    at = np.unique(np.concatenate([np.arange(min(nq, 40)), np.arange(max(0, nq - 40), nq)]))
    F, dF, A, dA = _reference(kind, p, w, v, q[at])
    out, grad = sbh.sbh_eval_brute_grad(dev(p), dev(w), dev(q), **kw)
    for f in (sbh.sbh_eval_brute(dev(p), dev(w), dev(q), **kw), out,
              sbh.sbh_eval_brute(dev(p), dev(w), dev(q), fp64_accum=False, **kw)):
        assert np.all(np.abs(f.cpu().numpy()[at] - F) <= 2e-6 * A)
    assert np.all(np.abs(grad.cpu().numpy()[at] - dF) <= 2e-6 * dA)


def test_coincident_and_nan_sources_add_nothing_to_a_winding_sum(sbh):
    """A source on the query, or with a NaN coordinate, leaves the winding sum and its gradient as they
    are, also where it shares a staged pair with another source or is an odd last one."""
    rng = np.random.default_rng(3)
    p, v = rng.random((2051, 3)).astype(np.float32), rng.normal(size=(2051, 3)).astype(np.float32)
    q = rng.random((70, 3)).astype(np.float32)
    w = np.ones(2051, np.float32)
    for bad in (4, 5, 1024, 2050):
        keep = np.arange(2051) != bad
        for value in (q[7], np.full(3, np.nan, np.float32)):
            pb = p.copy()
            pb[bad] = value
            out, grad = sbh.sbh_eval_brute_grad(dev(pb), dev(w), dev(q), "winding", dev(v))
            F, dF, A, dA = _reference("winding", p[keep], w[keep], v[keep], q[7:8])
            assert abs(out[7].item() - F[0]) <= 2e-6 * A[0]
            assert np.all(np.abs(grad[7].cpu().numpy() - dF[0]) <= 2e-6 * dA[0])
            plain = sbh.sbh_eval_brute(dev(pb), dev(w), dev(q), "winding", dev(v))
            assert abs(plain[7].item() - F[0]) <= 2e-6 * A[0]
