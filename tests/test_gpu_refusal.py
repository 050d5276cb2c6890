"""Input that sbh_build refuses is refused without building the tree: points that are not numbers, or more
points in one cell than a node has children for, are one leaf of all of them, which a single warp would
work on for seconds. The limit of half a second is a hundred times what a build of as many spread
points takes."""
import time

import pytest

pytestmark = pytest.mark.gpu


def _refused(sbh, p, w):
    import torch
    torch.cuda.synchronize()
    held = sbh.sbh_memory_in_use()
    start = time.perf_counter()
    with pytest.raises(sbh.SBHError) as e:
        sbh.sbh_build(p, w)
    took = time.perf_counter() - start
    torch.cuda.synchronize()
    assert sbh.sbh_memory_in_use() == held
    return e.value.status, took


@pytest.mark.parametrize("bad", ["one", "all", "weights"])
@pytest.mark.parametrize("n", [1000, 1 << 22])
def test_bad_input(sbh, n, bad):
    import torch
    p = torch.rand(n, 3, device="cuda")
    w = torch.ones(n, device="cuda")
    if bad == "weights":  # coincident points, none of them with a mass
        p[:] = 0.5
        w[:] = 0.0
    else:
        p[:1 if bad == "one" else n] = float("nan")
    sbh.sbh_build(torch.rand(n, 3, device="cuda"), torch.ones(n, device="cuda")).free()  # the pool holds the memory
    status, took = _refused(sbh, p, w)
    assert status == 1  # SBH_EINVAL
    assert took < 0.5


@pytest.mark.parametrize("others", [0, 1000])
def test_more_points_in_a_cell_than_children(sbh, others):
    import torch
    n = (1 << 24) + others
    p = torch.rand(n, 3, device="cuda")
    p[others:] = 0.25
    w = torch.ones(n, device="cuda")
    _refused(sbh, p, w)
    status, took = _refused(sbh, p, w)
    assert status == 5  # SBH_EUNSUPPORTED
    assert took < 0.5
