"""The windowed per-shift update (csrc/flush_tc.cuh) against the recurrence (k_flush).

The seed recurrence does not depend on the number of shifts, and a solve of fewer than eight
shifts keeps the recurrence form of the per-shift update, so a solve of many shifts (one
contraction per window of 64 iterations) must give, shift by shift, what solves of up to seven
shifts give.  Covered: windows of 1 to 64 iterations and several windows, ragged tiles of
shifts and of elements (64 per tile), shifts that freeze at different iterations, and
right-hand sides of extreme scale (rho = (b, b) has to stay a normal number).

Bound: per window each of x and P takes one sum of up to 128 products whose operands are
rounded at 2^-54 of the largest of their scale (window and 64 elements), which lies within a
factor ~2^6 of the typical element here, against 64 FMAs rounded at 2^-53 each: 2^6 sqrt(128)
2^-54 ~ 4e-14 of the norm per window, over at most ~20 windows: 1e-12."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

BAR = 1e-12


def _system(n, seed=3):
    from paper_2506_09551_gb300 import api
    rowptr, col, val = workloads.random_symmetric_csr(n, 3, seed=seed)
    return api.Operator.csr(rowptr, col, val)


def _solve(op, b, shifts, **kw):
    x, per, info, st = op.multishift_solve(b, shifts, -0.3 - 0.3j, allow_status=(5,), **kw)
    return x.cpu().numpy(), per, info


def _compare(op, b, shifts, scale=1.0, **kw):
    x, per, info = _solve(op, b, shifts, **kw)
    for i in range(0, len(shifts), 7):
        xs, ps, _ = _solve(op, b, shifts[i:i + 7], **kw)
        for k in range(len(xs)):
            err = np.linalg.norm((x[i + k] - xs[k]) / scale) / np.linalg.norm(xs[k] / scale)
            assert np.isfinite(err) and err <= BAR, (i + k, err)
            assert per["iters"][i + k] == ps["iters"][k]


@pytest.mark.parametrize("n", [9, 64, 65, 300, 1001])
@pytest.mark.parametrize("ns", [8, 9, 41])
@pytest.mark.parametrize("maxit", [1, 7, 64, 65, 130])
def test_capped(cuda, n, ns, maxit):
    op = _system(n)
    b = torch.tensor(workloads.random_complex_rhs(n, 5), device="cuda")
    _compare(op, b, np.linspace(-4.0, 5.0, ns), tol=0.0, maxit=min(maxit, n // 2))


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -450, 2.0 ** 450])
def test_converged(cuda, scale):
    op = _system(4003)
    b = torch.tensor(workloads.random_complex_rhs(4003, 6) * scale, device="cuda")
    _compare(op, b, np.linspace(-6.0, 6.0, 21), scale, tol=1e-11, maxit=3000)
