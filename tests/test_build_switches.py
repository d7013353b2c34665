"""The compile-time switches of the step kernels: the sources go through the device front end (every template
instantiated, no code generated) with each switch away from its default."""
import os
import subprocess

import pytest


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("switch", ["LBM_ZM_PREFETCH=0", "LBM_BOUNDS_CHECK=1", "LBM_LDPOP_HINT=0", "LBM_LDPOP_HINT=1",
                                    "LBM_LDPOP_HINT=3", "LBM_LDPOP_HINT=4", "LBM_STPOP_CS=0", "LBM_LDWORD_HINT=0",
                                    "LBM_ZM_CARVEOUT=50"])
def test_switch_compiles(lattice, switch, tmp_path):
    from paper_2306_16274_gb300 import build
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    r = subprocess.run([cc, *build.ARCH, "-std=c++17", "-fdevice-syntax-only", "-D" + switch, "-I", build.INCLUDE, "-c",
                        os.path.join(build.CSRC, f"kernels_q{lattice}.cu"), "-o", str(tmp_path / "x.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
