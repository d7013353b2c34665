"""The host side of the multi-domain batch over a faked CUDA runtime (tests/c/batch_host.cpp): no GPU, and none
needed to make an allocation fail or to see what a call launches."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    from paper_2306_16274_gb300 import build
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    tmp = tmp_path_factory.mktemp("batch_host")
    obj, exe = tmp / "batch.o", tmp / "batch_host"
    inc = ["-I", build.INCLUDE, "-I", build.CSRC, "-I", os.path.join(os.path.dirname(os.path.dirname(cc)), "include")]
    for cmd in ([cc, *build.ARCH, *build.FLAGS, *inc[:2], "-c", os.path.join(build.CSRC, "batch.cu"), "-o", str(obj)],
                [cxx, "-std=c++17", "-O1", "-Wno-deprecated-declarations", *inc,
                 os.path.join(ROOT, "tests", "c", "batch_host.cpp"), str(obj), "-o", str(exe)]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("scenario", ["failed_rebuild", "tune_after_change", "set_group_after_change", "odd_calls",
                                      "near_planes", "sm_count"])
def test_batch_host(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr)
