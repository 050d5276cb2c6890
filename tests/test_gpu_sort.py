"""The radix sort of the Morton codes at sizes around a tile (4,096 keys) and with more tiles than run at
once, for spread, repeated and equal keys: sbh_tree_export's `perm` must be the stable order of the codes."""
import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["uniform", "few", "equal"])
@pytest.mark.parametrize("n", [1, 2, 31, 4095, 4096, 4097, 8193, 100003, (1 << 21) + 1])
def test_sort_is_the_stable_order_of_the_codes(sbh, kind, n):
    if kind == "equal" and n > 10000:
        pytest.skip("every point in one cell: the tree has one node with n children")
    rng = np.random.default_rng(n)
    pts = rng.random((n, 3)).astype(np.float32)
    if kind == "few":
        pts = pts[: max(1, n // 8)][rng.integers(0, max(1, n // 8), n)]
    if kind == "equal":
        pts[:] = pts[0]
    t = sbh.sbh_build(dev(pts), dev(np.ones(n, np.float32)))
    e = sbh.sbh_tree_export(t, 0)
    code = np.empty(n, np.uint64)
    code[e["perm"]] = e["code"]
    np.testing.assert_array_equal(e["perm"], np.argsort(code, kind="stable"))
