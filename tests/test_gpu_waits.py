"""The bounded waits between the build's blocks: what a caller gets when one gives up.

A copy of the library is built whose waits all give up at once (SBH_SPIN_LIMIT = -1). Its sorts and trees
are incomplete, so what is tested is that this is said and that nothing else follows from it: sbh_build
returns SBH_ETIMEOUT and keeps no memory, sbh_morton_sort_noalloc marks its output by perm[0] = -1. Up
to 4,096 points no block of the sort waits for another.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(sbh, tmp_path_factory):
    from paper_2506_02219_gb300 import _build
    out = tmp_path_factory.mktemp("impatient")
    objs = []
    for src in _build._sources():
        name = os.path.basename(src)
        obj = os.path.join(_build.OBJDIR, name + ".o")
        if name == "sbh_build.cu" or not os.path.exists(obj):
            obj = str(out / (name + ".o"))
            subprocess.run([_build._nvcc(), *_build.NVCC_FLAGS, *_build.ARCH, "-DSBH_SPIN_LIMIT=-1", "-c", src, "-o", obj],
                           check=True)
        objs.append(obj)
    lib = str(out / "libsbh_impatient.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-shared", "-o", lib, *objs], check=True)
    lib = ctypes.CDLL(lib)
    P, I64 = ctypes.c_void_p, ctypes.c_int64
    lib.sbh_build.argtypes = [P, P, P, I64, ctypes.c_int32, P, ctypes.POINTER(P)]
    lib.sbh_morton_sort_noalloc.argtypes = [P, I64, P, P, P]
    lib.sbh_memory_in_use.restype = ctypes.c_uint64
    return lib


@pytest.mark.parametrize("normals", [False, True])
@pytest.mark.parametrize("n", [3000, 5000, 100003, 1 << 21])
def test_build_says_that_a_wait_gave_up(impatient, n, normals):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    p = torch.rand(n, 3, generator=g, device="cuda")
    w = torch.ones(n, device="cuda")
    for _ in range(3):
        tree = ctypes.c_void_p()
        status = impatient.sbh_build(p.data_ptr(), w.data_ptr(), p.data_ptr() if normals else None, n, 1, None,
                                     ctypes.byref(tree))
        torch.cuda.synchronize()
        assert status == 4 and not tree  # SBH_ETIMEOUT
        assert impatient.sbh_memory_in_use() == 0


@pytest.mark.parametrize("n", [4096, 4097, 30011, 65536])
def test_sort_marks_a_damaged_order(impatient, sbh, n):
    import torch
    p = dev(np.random.default_rng(n).random((n, 3)))
    want = sbh.sbh_tree_export(sbh.sbh_build(p, torch.ones(n, device="cuda")), 0)
    code = torch.empty(n, dtype=torch.int64, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    for _ in range(3):
        perm.fill_(-7)
        assert impatient.sbh_morton_sort_noalloc(p.data_ptr(), n, code.data_ptr(), perm.data_ptr(), None) == 0
        assert (perm[0].item() == -1) == (n > 4096)
    if n <= 4096:
        np.testing.assert_array_equal(perm.cpu().numpy(), want["perm"])
        np.testing.assert_array_equal(code.cpu().numpy().astype(np.uint64), want["code"])
