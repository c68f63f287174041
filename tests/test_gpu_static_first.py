"""csl_precondition_static as the first call of a process, before any plan exists:
every line length and precision, in a process of its own, against the oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import oracle as O, workloads as W
import paper_2408_00488_gb300 as csl
for ns in {grids!r}:
    v = W.rhs_normal(tuple(reversed(ns)), 1)
    r1, r2 = O.precond_apply(v.real, v.imag, 1.3, 2.0, 5.0)
    ref = r1 + 1j * r2
    out = csl.precondition_static(torch.from_numpy(v).to("cuda:0"), 1.3, 2 + 5j, {precision!r}).cpu().numpy()
    err = np.abs(out - ref).max() / np.abs(ref).max()
    assert err < {tol!r}, (ns, err)
"""


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
@pytest.mark.parametrize("grids", [[(15, 15), (3, 7), (511, 255)], [(1023, 255), (31, 31, 31)], [(127, 1023), (63, 63, 63)]])
def test_before_any_plan(grids, precision, tol):
    code = PROGRAM.format(root=ROOT, grids=grids, precision=precision, tol=tol)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
