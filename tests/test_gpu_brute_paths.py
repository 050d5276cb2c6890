"""Brute force around the lines between its ways of sharing work out: a warp with queries of its own or
eight on the same ones, one, two or four queries a lane, one to eight blocks to a query (whose shares of
the sources are uneven where the number of sources is odd). Reference and tolerance are those of
test_gpu_brute_split, for the first and the last queries of a call.

And what the lines are for, as ratios of times that a call is far from on either side: joining parts of
a query must not outweigh its terms (ten sources, with FP64 sums and without: 117 / 101 us here; 499 / 127
with every query split), and a share's size must not be rounded up to what costs as much as the next
(10 tiles of 1,024 sources against 16, by eight blocks: 0.63 of the work, and the same time if shares are
whole tiles)."""
import numpy as np
import pytest

from gpu_util import dev
from test_gpu_brute_split import ALPHA, EPS, G, _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq", [(1, 300), (127, 257), (128, 257), (255, 65536), (256, 65535), (257, 65536),
                                  (1023, 65536), (1024, 65536), (1023, 65535), (2047, 30001), (2050, 20011),
                                  (8191, 3001), (10001, 100003), (4097, (1 << 18) - 1), (2049, 1 << 18),
                                  (515, (5 << 17) - 1), (1, 5 << 17), (4096, (5 << 17) + 33), (4097, 5 << 17)])
@pytest.mark.parametrize("kind", ["coulomb", "winding", "smoothdist", "affine"])
def test_every_path_adds_up(sbh, kind, n, nq):
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


def _time(f):
    import torch
    f()
    times = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


def test_few_sources_cost_their_terms(sbh):
    import torch
    p, w, q = torch.rand(10, 3, device="cuda"), torch.ones(10, device="cuda"), torch.rand(10 ** 6, 3, device="cuda")
    out = torch.empty(10 ** 6, device="cuda")
    t = [_time(lambda: sbh.sbh_eval_brute(p, w, q, "smoothdist", fp64_accum=f, out=out)) for f in (True, False)]
    assert t[0] < 2 * t[1]


def test_uneven_shares_are_balanced(sbh):
    import torch
    q, out = torch.rand(100000, 3, device="cuda"), torch.empty(100000, device="cuda")
    t = []
    for n in (10 * 1024, 16 * 1024):
        p, w = torch.rand(n, 3, device="cuda"), torch.ones(n, device="cuda")
        t.append(_time(lambda: sbh.sbh_eval_brute(p, w, q, "coulomb", out=out)))
    assert t[0] < 0.85 * t[1]


@pytest.mark.parametrize("nq", [100, 70000])
def test_the_largest_alpha_gives_the_nearest_source(sbh, nq):
    """alpha only has to be finite: the smooth distance is then the smallest distance, a rounded root."""
    rng = np.random.default_rng(nq)
    p, q = rng.random((300, 3)).astype(np.float32), rng.random((nq, 3)).astype(np.float32)
    w = np.ones(300, np.float32)
    want = np.sqrt(((p[None].astype(np.float64) - q[:100, None]) ** 2).sum(2).min(1))
    for alpha in (2.0e38, 3.0e38):
        out, grad = sbh.sbh_eval_brute_grad(dev(p), dev(w), dev(q), "smoothdist", alpha=alpha)
        for f in (out, sbh.sbh_eval_brute(dev(p), dev(w), dev(q), "smoothdist", alpha=alpha),
                  sbh.sbh_eval_brute(dev(p), dev(w), dev(q), "smoothdist", fp64_accum=False, alpha=alpha)):
            assert np.all(np.abs(f.cpu().numpy()[:100] - want) <= 1e-6 * want)
        assert np.all(np.abs(np.linalg.norm(grad.cpu().numpy(), axis=1) - 1) < 1e-6)
