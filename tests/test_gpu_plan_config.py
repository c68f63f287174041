"""Plan.config names the kernels that run: the FP64 form's fixed-point lines with
their lanes per line, the FP32 forms' variants."""
import re

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def csl():
    import __graft_entry__ as g
    g.build()
    import paper_2408_00488_gb300 as csl
    return csl


@pytest.mark.parametrize("ns", [(7, 15), (31, 63), (127, 255), (511, 1023), (4095, 7)])
def test_lanes_of_the_fixed_point_lines(csl, ns):
    import torch
    faces = [torch.from_numpy(np.ascontiguousarray(f)).to("cuda:0") for f in W.sample_faces(2, ns, W.coef_const(1.0))]
    for autotune in (False, True):
        with csl.Plan(faces, 1 + 1j, autotune=autotune) as p:
            passes = re.findall(r"\[N=(\d+) (long-line )?fixed-point(\d+) lines=(\d+) threads=(\d+) ", p.config)
            assert [int(q[0]) for q in passes] == [n + 1 for n in ns], p.config
            for N, long_line, lanes, lines, threads in passes:
                assert int(lanes) * int(lines) == int(threads) and bool(long_line) == (int(N) > 1024), p.config
    with csl.Plan(faces, 1 + 1j, precision="fp32", autotune=False) as p:
        assert "fixed-point" not in p.config and len(re.findall(r"\[N=\d+ (warp|stockham|long-line)", p.config)) == 2
