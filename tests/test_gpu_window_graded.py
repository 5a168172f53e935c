"""The windowed per-shift update (csrc/flush_tc.cuh) element by element, on systems whose
solutions span many decades: a solve of many shifts must agree, in every element, with solves of
up to seven shifts, which keep the recurrence (the seed recurrence is the same for both).

Bound: an element is a sum of up to ~130 terms, each rounded at 2^-53, and lies below its largest
partial sum by at most the deepest cancellation among the 41 x 1001 elements compared, a factor of
about 200 for complex values: 130 x 2^-53 x 200 = 3e-12, times 30 for the growth of the terms:
1e-10.  The median has neither cancellation nor extremes: sqrt(130) 2^-53 = 1.3e-15, times 8."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

N = 1001
C0 = -0.3 - 0.3j


def _system(kind):
    """CSR arrays, right-hand side, iterations."""
    rng = np.random.default_rng(7)
    g = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    ptr, idx = np.arange(N + 1, dtype=np.int64), np.arange(N, dtype=np.int32)
    if kind == "interleaved":        # neighbours 18 decades apart
        return (ptr, idx, rng.choice(np.linspace(1.0, 5.0, 20), N)), g * np.where(np.arange(N) % 2, 1.0, 1e-18), 20
    if kind == "decades":            # every size from 1 to 1e-30, several windows
        return (ptr, idx, rng.uniform(1.0, 5.0, N)), g * 10.0 ** rng.uniform(-30.0, 0.0, N), 130
    if kind == "subnormal":          # some elements at the end of the exponent range
        return (ptr, idx, rng.choice(np.linspace(1.0, 5.0, 20), N)), g * np.where(np.arange(N) % 3, 1.0, 2.0 ** -1050), 20
    if kind == "chain":              # reached one element per iteration, decaying by 20 each
        d = rng.uniform(6.0, 8.0, N)
        rows = [[j for j in (i - 1, i, i + 1) if 0 <= j < N] for i in range(N)]
        col = np.array([j for r in rows for j in r], dtype=np.int32)
        val = np.array([d[i] if i == j else 0.3 for i, r in enumerate(rows) for j in r])
        b = np.zeros(N, complex)
        b[0] = 1.0 + 0.5j
        return (np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64), col, val), b, 80
    return workloads.random_symmetric_csr(N, 3, seed=3), g, 130


@pytest.mark.parametrize("kind", ["interleaved", "decades", "subnormal", "chain", "random"])
@pytest.mark.parametrize("ns", [8, 41])
def test_elementwise(cuda, kind, ns):
    from paper_2506_09551_gb300 import api
    csr, b, maxit = _system(kind)
    op = api.Operator.csr(*csr)
    b = torch.tensor(b, device="cuda")
    shifts = np.linspace(-4.0, 0.5, ns) + 0j

    def solve(s):
        x, per, _, _ = op.multishift_solve(b, s, C0, tol=0.0, maxit=maxit, allow_status=(5,))
        return x.cpu().numpy(), per["iters"]

    x, it = solve(shifts)
    ref = [solve(shifts[i:i + 7]) for i in range(0, ns, 7)]
    xr, itr = np.concatenate([r[0] for r in ref]), np.concatenate([r[1] for r in ref])
    assert np.array_equal(it, itr)
    assert np.array_equal(x == 0, xr == 0)
    on = np.abs(xr) > (1e-290 if kind != "subnormal" else 2.0 ** -1056)
    err = np.abs(x - xr)[on] / np.abs(xr)[on]
    # below 2^-1022 a value is a multiple of 2^-1074 whatever the method
    quantum = 2.0 ** -1074 * maxit / np.abs(xr)[on] if kind == "subnormal" else 0.0
    assert np.all(err <= 1e-10 + quantum), err.max()
    assert np.median(err) <= 1e-14
