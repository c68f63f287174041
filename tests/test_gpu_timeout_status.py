"""How a solve ends when a bounded device wait gave up (a tensor-core transform
whose commit never arrives).  No wait is forced: the hooks record the time-out
as such a wait records it and run the scalar steps that have to report it."""
import ctypes

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


@pytest.mark.parametrize("blocks", [1, 2, 64, 1024])
def test_recorded_while_the_kernel_runs(csl, blocks):
    """After the kernel copied the state: the copy must not be stored over it."""
    out = (ctypes.c_int * 2)()
    for late in (0, blocks // 2, blocks - 1):
        assert csl.lib.csl_test_timeout_raised(blocks, late, out) == csl.OK
        assert list(out) == [1, csl.TIMEOUT]
    assert csl.lib.csl_test_timeout_raised(blocks, -1, out) == csl.OK
    assert list(out) == [0, csl.OK]
    assert csl.lib.csl_test_timeout_raised(blocks, blocks, out) == csl.INVALID_ARG


@pytest.mark.parametrize("precision,ns", [("bf16x3", (31, 31, 31)), ("bf16x6", (31, 63)), ("fp32", (31, 15)),
                                          ("fp64", (15, 31)), ("fp64", (7, 7, 15))])
def test_recorded_by_an_earlier_kernel(csl, precision, ns):
    """Stencil and MID pass end the solve; the plan solves as before afterwards."""
    import torch
    dim = len(ns)
    faces = [torch.from_numpy(np.ascontiguousarray(f)).to("cuda:0")
             for f in W.sample_faces(dim, ns, W.coef_const(1.0))]
    f = torch.from_numpy(W.rhs_uniform(tuple(reversed(ns)), 5)).to("cuda:0")
    out = (ctypes.c_int * 2)()
    with csl.Plan(faces, 1 + 10j, precision=precision, autotune=False) as p:
        z, info = p.solve(f, tol=1e-8)
        assert info.converged
        for kernel in (0, 2 if dim == 2 else 3):
            assert csl.lib.csl_test_timeout_seen(p._h, kernel, out) == csl.OK
            assert list(out) == [1, csl.TIMEOUT]
        again, info = p.solve(f, tol=1e-8)
        assert info.converged and torch.equal(z, again)
