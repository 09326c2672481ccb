"""Single kernels of the library on hand-made blocks (tests/device_harness.cu, built
here): what a kernel does in states that no sequence of public calls reaches, and what
the kernels' roundings on the integer pipes give at the ends of their formats."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ERR_GRADED, ERR_TIMEOUT = 2, 16


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


@pytest.fixture(scope="module")
def lib_impatient(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return build(tmp_path_factory.mktemp("harness0"), "-DMR_WAIT_POLLS=0")


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


# kernel: dimension, block size, type; 4 and 5 are the details, the others stages
PERIODIC = {0: (2, 17, np.float32), 1: (2, 17, np.float32), 2: (2, 33, np.float64), 3: (3, 17, np.float32),
            4: (2, 17, np.float32), 5: (2, 33, np.float64)}


def run_periodic(lib, kernel):
    dim, B, dt = PERIODIC[kernel]
    f = np.random.default_rng(4).standard_normal((4, (B ** dim + 3) // 4 * 4)).astype(dt)
    before = f.copy()
    md, err = ctypes.c_double(-1.0), ctypes.c_int(0)
    assert lib.periodic_block(kernel, f.ctypes.data_as(ctypes.c_void_p), ctypes.byref(md), ctypes.byref(err))
    return before, f, md.value, err.value


@pytest.mark.parametrize("kernel", sorted(PERIODIC))
def test_wait_that_runs_out(lib, lib_impatient, kernel):
    # built to give up at once, the first wait for a block's bulk copies runs out (the
    # copies land in the second one): the kernel reports it and leaves, and it stores
    # nothing of the block whose values it does not have
    before, after, md, err = run_periodic(lib_impatient, kernel)
    assert err == ERR_TIMEOUT and md == -1.0
    np.testing.assert_array_equal(before, after)
    # the same launch with the library's limit
    before, after, md, err = run_periodic(lib, kernel)
    assert err == 0
    if kernel >= 4:
        assert md > 0.0
    else:
        assert not np.array_equal(before, after)


def same(a, b):
    # equal bits, or both NaN
    u = np.uint32 if a.dtype == np.float32 else np.uint64
    return (a.view(u) == b.view(u)) | (np.isnan(a) & np.isnan(b))


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def fp64_patterns():
    # every exponent with the mantissas next to every rounding boundary of FP32 results,
    # normal (the low 29 bits) and subnormal (up to the whole mantissa), and random ones
    m = {0, 1, (1 << 52) - 1}
    for s in range(29, 53):
        for k in (0, 1, 2, 3):
            for d in (-1, 0, 1):
                m.add(((k << s) + (1 << (s - 1)) + d) & ((1 << 52) - 1))
    m = np.array(sorted(m) + list(np.random.default_rng(1).integers(0, 1 << 52, 64)), np.uint64)
    e = np.arange(2048, dtype=np.uint64) << np.uint64(52)
    u = (e[:, None] | m[None, :]).ravel()
    return np.concatenate([u, u | np.uint64(1 << 63)]).view(np.float64)


def test_roundings_are_the_conversions(lib):
    d = fp64_patterns()
    f, w, q = np.empty(len(d), np.float32), np.empty(len(d)), np.empty(len(d))
    assert lib.round_values(len(d), ptr(d), ptr(f), ptr(w), ptr(q))
    with np.errstate(all="ignore"):
        assert same(f, d.astype(np.float32)).all()
        assert same(w, f.astype(np.float64)).all()
        assert same(q, d / 16.0).all()
    m = np.concatenate([[0, 1, 2, 3, (1 << 23) - 1], 1 << np.arange(23), np.random.default_rng(2).integers(0, 1 << 23, 200)])
    u = ((np.arange(512) << 23)[:, None] | m[None, :]).ravel().astype(np.uint32)
    f = u.view(np.float32)
    d = np.empty(len(f))
    assert lib.widen_values(len(f), ptr(f), ptr(d))
    with np.errstate(all="ignore"):
        assert same(d, f.astype(np.float64)).all()
