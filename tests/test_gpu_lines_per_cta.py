"""The option lines_per_cta: any positive number gives a plan that runs, with the
results of the default tile (the lines of a tile do not mix)."""
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


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ns", [(63, 7), (127, 15), (127, 31), (63, 63), (31, 127), (127, 255), (63, 511), (63, 1023),
                                (15, 31, 63), (127, 15, 127)])
def test_every_request_runs(csl, precision, ns):
    import torch
    faces = [dev(f) for f in W.sample_faces(len(ns), ns, W.coef_const(1.0))]
    v = dev(W.rhs_uniform(tuple(reversed(ns)), 3))
    with csl.Plan(faces, 1 + 50j, precision=precision, autotune=False) as p:
        ref = p.precondition(v)
    for lines in (1, 2, 3, 8, 16, 64, 100, 1024, 2**31 - 1):
        with csl.Plan(faces, 1 + 50j, precision=precision, lines_per_cta=lines) as p:
            assert max(int(t) for t in re.findall(r"threads=(\d+)", p.config)) <= 256
            assert torch.equal(p.precondition(v), ref), lines
            if lines in (8, 64):
                assert p.solve(v, tol=1e-6)[1].converged
