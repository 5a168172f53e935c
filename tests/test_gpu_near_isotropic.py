"""rho = (r, r) of a residual that is close to isotropic, |rho| << ||r||^2, in one thread of the
vector kernels.  The elements b = (1, 2i, 2, i) on diagonal entries (0, 3, 5, 8) are the third
difference: sum b^2, sum d b^2 and sum d^2 b^2 vanish, so with one more element b = 1 on 16 the
first step is alpha_0 = 1/16, r_1 = (1 - d / 16) b, and the squares of r_1 cancel exactly.  A last
element b = 1e-9 on 0 leaves rho_1 = 1e-18: the recurrence goes on.  All numbers but that one are
dyadic, so every sum here is exact; only a rho formed from sums of the size of ||r||^2 loses it
and ends as a breakdown after one iteration."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ns", [1, 8])
def test_rho_keeps_the_small_term(cuda, prec, ns):
    from paper_2506_09551_gb300 import api, native
    # threads of the vector kernels: three CTAs of 256 per SM, one CTA left out; two adjacent
    # elements per thread in FP32
    step = (3 * torch.cuda.get_device_properties(0).multi_processor_count - 1) * 256 * (1 + prec)
    n = 4 * step + 2
    idx = step * np.arange(5)
    d, b = np.ones(n), np.zeros(n, complex)
    d[idx], b[idx] = [0.0, 3.0, 5.0, 8.0, 0.0], [1.0, 2.0j, 2.0, 1.0j, 1e-9]
    d[2], b[2] = 16.0, 1.0
    op = api.Operator.csr(np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), d)
    _, _, info, st = op.multishift_solve(torch.tensor(b, device="cuda"), np.arange(ns) * 0.0625j, tol=0.0, maxit=2,
                                         prec=prec, allow_status=(4, 5))
    assert info["iterations"] == 2 and st == native.MSB_EMAXITER
