"""Rows whose staged copy is just below 48 KB of dynamic shared memory (csrc/hubrows.cuh): 3,003
down-spin states in FP64, with 14 sites and 8 down electrons.  The seed product has 4 KB of
static shared memory besides, so such a launch needs the opt-in to more than 48 KB.  The limit of
a kernel stays raised for the whole process, so each solve runs in a process of its own.

Bound: the recursive residual is at most 1e-10 ||b||; its distance from the true one is about
(iterations) 2^-53 ||A|| max ||x|| <= 500 x 1.1e-16 x 60 x 1e3: 1e-8."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import numpy as np, torch, workloads
from paper_2506_09551_gb300 import api
ops = [api.Operator.hubbard(api.model(14, nu - 1, nd, core_site=2), True) for nu, nd in {sectors}]
op = ops[0] if len(ops) == 1 else api.Operator.direct_sum(ops, [0.25 * i for i in range(len(ops))])
b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), device="cuda")
shifts = np.linspace(-2.0, 2.0, 3) + 0j
x, per, info, st = op.multishift_solve(b, shifts, 3.0 - 0.5j, tol=1e-10, maxit=2000)
assert st == 0 and per["converged"].all()
for k, s in enumerate(shifts):
    r = op.apply(x[k][None], 3.0 - 0.5j - s)[0] - b
    assert float(torch.linalg.vector_norm(r)) <= 1e-8 * float(torch.linalg.vector_norm(b))
"""


@pytest.mark.parametrize("sectors", [[(2, 8)], [(1, 8), (2, 6)]], ids=["one", "sum"])
def test_rows_just_below_the_default_limit(cuda, sectors):
    r = subprocess.run([sys.executable, "-c", CODE.format(sectors=sectors)], cwd=ROOT, capture_output=True, text=True,
                       timeout=200)
    assert r.returncode == 0, r.stderr[-2000:]
