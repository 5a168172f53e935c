"""Solves of short vectors (k_window in csrc/msbicg.cu: a window of iterations in one cooperative
launch) at the sizes where it can go wrong: a few elements, ragged last CTAs, the edges of one and
two elements per thread and of the rule, windows cut by the iteration cap, more shifts than threads, and
endings other than convergence.  A direct sum of one operator takes the launch-per-product form of
the same recurrence.

Bounds.  Capped runs: the two forms round the sums behind alpha and beta and the product
differently, a relative perturbation of about 2^-52 in every iteration, which the recurrence can
amplify (it loses orthogonality as Ritz values converge).  The amplification is measured: the
change of the reference form's result when b is perturbed by 2^-52 relative; the forms may differ
by 4 (iterations) times that, and 1e-13.  Converged runs: the recursive residual is at most 1e-10 ||b||, and its distance from
the true one is about (iterations) 2^-53 ||A|| max ||x_m|| ~ 300 x 1e-16 x 15 x 1e3 ~ 5e-10: 1e-9."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

C0 = -0.3 - 0.3j


def _solve(op, b, shifts, **kw):
    x, per, info, st = op.multishift_solve(b, shifts, C0, allow_status=(4, 5), **kw)
    return x.cpu().numpy(), per, st


def _hub(L, nu, nd):
    from paper_2506_09551_gb300 import api
    op = api.Operator.hubbard(api.model(L, nu - 1, nd, core_site=1), True)
    return op, api.Operator.direct_sum([op], [0.0])


@pytest.mark.parametrize("case", [(4, 4, 3), (4, 2, 1), (5, 3, 2), (8, 5, 4), (9, 5, 3), (10, 5, 4)])
@pytest.mark.parametrize("ns", [1, 7, 41, 300])
@pytest.mark.parametrize("maxit", [1, 63, 64, 65, 130])
def test_capped(cuda, case, ns, maxit):
    op, ref = _hub(*case)
    maxit = min(maxit, max(1, op.dim // 4))
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), device="cuda")
    shifts = np.linspace(-4.0, 5.0, ns) + 0j
    x, per, st = _solve(op, b, shifts, tol=0.0, maxit=maxit)
    xr, pr, sr = _solve(ref, b, shifts, tol=0.0, maxit=maxit)
    assert st == sr and np.array_equal(per["iters"], pr["iters"])
    noise = np.random.default_rng(8).standard_normal((2, op.dim)) * 2.0 ** -52
    bp = b + torch.tensor((noise[0] + 1j * noise[1]), device="cuda") * torch.abs(b)
    xp, _, _ = _solve(ref, bp, shifts, tol=0.0, maxit=maxit)
    for k in range(ns):
        amp = np.linalg.norm(xp[k] - xr[k])
        assert np.linalg.norm(x[k] - xr[k]) <= 4 * maxit * amp + 1e-13 * np.linalg.norm(xr[k])


@pytest.mark.parametrize("n", [9, 63, 65, 9664, 9665, 38656, 38657, 57984, 57985])
@pytest.mark.parametrize("ns", [1, 9])
def test_converged(cuda, n, ns):
    from paper_2506_09551_gb300 import api
    rowptr, col, val = workloads.random_symmetric_csr(n, 3, seed=4)
    op = api.Operator.csr(rowptr, col, val)
    b = torch.tensor(workloads.random_complex_rhs(n, 6), device="cuda")
    shifts = np.linspace(-5.0, 5.0, ns) + 0j
    x, per, _ = _solve(op, b, shifts, tol=1e-10, maxit=3000)
    assert np.all(per["converged"])
    for k, s in enumerate(shifts):
        xk = torch.tensor(x[k], device="cuda")
        r = op.apply(xk[None], C0 - s)[0] - b
        assert float(torch.linalg.vector_norm(r)) <= 1e-9 * float(torch.linalg.vector_norm(b))


@pytest.mark.parametrize("ns", [1, 12])
def test_fp32(cuda, ns):
    op, ref = _hub(8, 5, 4)
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), device="cuda").to(torch.complex64)
    shifts = np.linspace(-4.0, 5.0, ns) + 0j
    x, per, _ = _solve(op, b, shifts, tol=0.0, maxit=20, prec=1)
    xr, pr, _ = _solve(ref, b, shifts, tol=0.0, maxit=20, prec=1)
    # 20 iterations: sqrt(n) 2^-24 ~ 4e-6 in the sums, growth below 1e2
    assert np.array_equal(per["iters"], pr["iters"]) and np.linalg.norm(x - xr) <= 4e-4 * np.linalg.norm(xr)


@pytest.mark.parametrize("kind", ["zero", "isotropic", "nan"])
def test_endings(cuda, kind):
    """The same status as the other form for b = 0, (b, b) = 0 with b != 0, and a NaN."""
    op, ref = _hub(8, 5, 4)
    b = workloads.random_complex_rhs(op.dim, 5)
    if kind == "nan":
        b[3] = np.nan
    else:
        b[:] = 0
        if kind == "isotropic":
            b[0], b[1] = 1.0, 1.0j
    b = torch.tensor(b, device="cuda")
    shifts = np.linspace(-4.0, 5.0, 9) + 0j
    out = []
    for o in (op, ref):
        x, per, info, st = o.multishift_solve(b, shifts, C0, tol=1e-10, maxit=2000, allow_status=(4, 5, 6))
        out.append((st, list(per["converged"]), list(per["iters"])))
        if kind == "zero":
            assert not torch.any(x != 0)
    assert out[0] == out[1]


@pytest.mark.parametrize("e", [-450, 450])
def test_scale(cuda, e):
    """The exponent management scales by powers of two only: 2^e b gives 2^e x, bit for bit."""
    op, _ = _hub(8, 5, 4)
    b = workloads.random_complex_rhs(op.dim, 5)
    shifts = np.linspace(-4.0, 5.0, 9) + 0j
    x, per, _ = _solve(op, torch.tensor(b, device="cuda"), shifts, tol=1e-10, maxit=2000)
    xs, ps, _ = _solve(op, torch.tensor(b * 2.0 ** e, device="cuda"), shifts, tol=1e-10, maxit=2000)
    assert np.all(per["converged"]) and np.array_equal(per["iters"], ps["iters"])
    assert np.array_equal(xs, x * 2.0 ** e)
