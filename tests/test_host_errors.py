"""Errors of CUDA runtime calls on the host path, made by a stand-in for the runtime
(tests/fake_cudart.cpp): no GPU is needed."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
MR_ECUDA = 4


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_1902_00088_gb300 import build as b
    d = tmp_path_factory.mktemp("fake_cudart")
    objs = []
    for src in (os.path.join(b.SRC, "mr_api.cu"), os.path.join(HERE, "fake_cudart.cpp")):
        objs.append(str(d / os.path.basename(src)) + ".o")
        subprocess.check_call([b._nvcc()] + b.ARCH + ["-O1", "-std=c++17", "-fmad=false", "-I", b.SRC,
                                                      "-c", src, "-o", objs[-1]])
    out = str(d / "host_errors")
    # the launchers that this path does not reach stay undefined
    subprocess.check_call(["g++", "-static", "-no-pie", "-o", out] + objs +
                          ["-Wl,--unresolved-symbols=ignore-all", "-lpthread"])
    return out


def test_cnn_eval_leaves_no_copy_behind_an_error(exe):
    # the caller's arrays may be freed as soon as the call returns, whichever runtime call failed
    rows = [line.split() for line in subprocess.check_output([exe], text=True).splitlines()]
    assert {"cudaMallocAsync", "cudaMemcpyAsync", "cudaMemsetAsync", "cudaGetLastError",
            "cudaStreamSynchronize"} == {r[0] for r in rows}
    assert [r[0] for r in rows].count("cudaMemcpyAsync") == 6
    for name, status, queued in rows:
        assert int(status) == MR_ECUDA, name
        assert int(queued) == 0, name
