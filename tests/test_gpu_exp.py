"""The exponential of the smooth distance's terms against FP64, over its range down to where it is zero.

Two sources, one on the query with mass 2^-126 and one at distance 1 with mass 1: the raw sum is
2^-126 + exp(-alpha), in the frame of the source on the query. Tolerance, relative: 2^-22 for PTX's
ex2.approx.ftz.f32, doubled for the sum's three roundings; for an exponent of x, |x| 2^-22 for the
roundings of log2 e, of the product with it, and of the distance (a reciprocal root to 2^-22.9)."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("order", [0, 1])  # which source comes first
def test_exponential_of_the_smooth_distance(sbh, order, grad):
    p = np.array([[0, 0, 0], [1, 0, 0]], np.float32)
    tiny = 2.0 ** -126
    w = np.array([tiny, 1.0], np.float32)
    if order:
        p = np.ascontiguousarray(1 - p)  # the source on the query is the last in Morton order
    tree = sbh.sbh_build(dev(p), dev(w))
    q = dev(p[:1])
    opts = sbh.eval_opts(raw_sum=1)
    alphas = np.concatenate([np.geomspace(1e-6, 100, 600), np.linspace(80, 110, 400)]).astype(np.float32)
    for a in alphas:
        f = sbh.sbh_eval_grad if grad else sbh.sbh_eval
        got = f(tree, q, "smoothdist", 1, 0, opts=opts, alpha=float(a))
        got = float((got[0] if grad else got).item())
        x = -float(a)
        if x < -87.35:  # below 2^-126 = exp(-87.3365...)
            assert got == tiny
        elif x > -87.32:
            want = np.exp(x)
            assert abs(got - tiny - want) <= want * (2.0 ** -21 + abs(x) * 2.0 ** -22) + tiny * 2.0 ** -22
