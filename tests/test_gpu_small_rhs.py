"""Right-hand sides whose rho = (r, r) passes through the subnormal numbers: (b, b) is normal, but the
residual falls by 2^-20 before it is rescaled.  1 / rho is not representable there, the quotient
beta of two such numbers is; rho keeps at least 46 bits.
Bound: the recursive residual is at most 1e-10 ||b||, its distance from the true one about
(iterations) 2^-53 ||A|| max ||x|| ~ 5e-10 as for other right-hand sides of this system: 2e-9."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

C0 = -0.3 - 0.3j


@pytest.mark.parametrize("form", ["one", "sum"])
@pytest.mark.parametrize("e", [-498, -500, -502])
def test_converges(cuda, form, e):
    from paper_2506_09551_gb300 import api
    op = api.Operator.hubbard(api.model(8, 4, 4, core_site=1), True)
    if form == "sum":
        op = api.Operator.direct_sum([op], [0.0])
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), device="cuda")
    shifts = np.linspace(-4.0, 5.0, 9) + 0j
    x, per, info, st = op.multishift_solve(b * 2.0 ** e, shifts, C0, tol=1e-10, maxit=4000)
    assert st == 0 and per["converged"].all()
    for k, s in enumerate(shifts):
        r = op.apply((x[k] * 2.0 ** -e)[None], C0 - s)[0] - b
        assert float(torch.linalg.vector_norm(r)) <= 2e-9 * float(torch.linalg.vector_norm(b))
