"""Solves in the forms that they fall back to, against the form they take first.

A cooperative launch that the runtime refuses (its CTAs do not all fit, as in a context limited to
part of the SMs) must leave the solve to the launch-per-product form.  The refusal is faked on
the host.  Bounds: the recursive residual is at most 1e-10 ||b|| (1e-6 in FP32), and its distance
from the true one about (iterations) 2^-53 ||A|| max ||x|| ~ 5e-10 (FP32, 2^-24 and the square
root of the iterations for independent roundings: 5e-5): 1e-9 and 1e-4."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

C0 = -0.3 - 0.3j


@pytest.fixture
def limits(cuda, lib):
    yield lib.msb_test_solver_limits
    lib.msb_test_solver_limits(0)


def _operator(kind):
    from paper_2506_09551_gb300 import api
    if kind == "ring":
        return api.Operator.hubbard(api.model(8, 4, 4, core_site=1), True)
    if kind == "cluster":                   # 3 x 3 with diagonal hopping: the second pair of tables
        return api.Operator.hubbard(api.model(9, 3, 3, core_site=1, lx=3, tp=-0.3), True)
    return api.Operator.csr(*workloads.random_symmetric_csr(4003, 3, seed=4))


def _check(op, prec, ns, **kw):
    from paper_2506_09551_gb300 import api
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), dtype=api.cdtype(prec), device="cuda")
    shifts = np.linspace(-4.0, 5.0, ns) + 0j
    x, per, info, st = op.multishift_solve(b, shifts, C0, tol=1e-6 if prec else 1e-10, maxit=3000, prec=prec, **kw)
    assert st == 0 and per["converged"].all()
    b, x = b.to(torch.complex128), x.to(torch.complex128)
    for k, s in enumerate(shifts):
        r = op.apply(x[k][None], C0 - s)[0] - b
        assert float(torch.linalg.vector_norm(r)) <= (1e-4 if prec else 1e-9) * float(torch.linalg.vector_norm(b))
    return x, info


@pytest.mark.parametrize("kind", ["ring", "cluster", "csr"])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ns", [3, 12])
def test_refused_cooperative_launch(limits, kind, prec, ns):
    op = _operator(kind)
    _, a = _check(op, prec, ns)
    limits(1)
    _, b = _check(op, prec, ns)
    # the fallback did run: three launches per iteration instead of one per window
    assert b["kernel_launches"] > 2 * b["iterations"] > 4 * a["kernel_launches"]
