"""Single kernels of the library on hand-made blocks (tests/device_harness.cu, built
here): what a kernel does in states that no sequence of public calls reaches."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ERR_GRADED = 2


def build(path, *defines):
    from paper_1902_00088_gb300 import build as b
    so = str(path / "libdevice_harness.so")
    subprocess.check_call([b._nvcc()] + b.ARCH + b.FLAGS + list(defines) +
                          ["-I", b.SRC, "-shared", "-o", so, os.path.join(HERE, "device_harness.cu")])
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return build(tmp_path_factory.mktemp("harness"))


def block(dim, form, seed):
    n = (17 ** dim + 3) // 4 * 4
    return np.random.default_rng(seed).standard_normal(n).astype(np.float32 if form == 1 else np.float64)


# forms: 0 FP64, 1 FP32, 2 FP64 state with FP32 stages
@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("dim,warp", [(2, 0), (2, 1), (3, 0)])
def test_stage_leaves_edge_nodes_without_an_owner(lib, dim, warp, form):
    # a block in a tree that is not graded: the error is set, and the state's edge
    # nodes, which no leaf holds, are not overwritten
    y = block(dim, form, 3)
    want = y.copy()
    err = ctypes.c_int(0)
    assert lib.ownerless_stage(dim, form, warp, y.ctypes.data_as(ctypes.c_void_p), ctypes.byref(err))
    assert err.value == ERR_GRADED
    np.testing.assert_array_equal(y, want)


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("Bs", [17, 33])
def test_refinement_keeps_a_thousand_threads_per_sm(lib, Bs, fp64):
    # its launch shape is its own: with the stage's 160 threads an SM held 640 of them
    assert lib.refine_threads_per_sm(Bs, fp64) >= 1024
