"""Accuracy of the FP64 form's fixed-point sine transform: its own functions,
compiled for the host (fixed_point_host.cu), against FP64 butterflies on the
same lines.  The form replaced those, so on no kind of line may its root mean
square error over the drawn lines be larger; and no value or shift may leave the
limits that the scale plan promises.  The lines that tell are those whose norm is
little more than their largest entry: a point source over a small background."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("fixed_point") / "host"
    subprocess.run([NVCC, "-arch=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-w",
                    "-I", os.path.join(ROOT, "paper_2408_00488_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(HERE, "fixed_point_host.cu"), "-o", str(out)], check=True)
    return out


@pytest.mark.parametrize("N", [64, 128, 256, 512, 1024, 2048, 4096, 8192])
def test_error_not_above_fp64(program, N):
    lines = subprocess.run([str(program), str(N)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(lines) >= 15
    for line in lines:
        n, lanes, kind, fixed, fp64, bad = line.split()
        assert int(bad) == 0, line
        assert 0 < float(fixed) <= float(fp64), line
