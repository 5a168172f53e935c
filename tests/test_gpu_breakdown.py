"""A breakdown of the recurrence after it has started, (r, r) = 0 with r != 0, exact in dyadic
numbers: two elements b = (1, i) on equal diagonal entries cancel in every product, so the
recurrence is that of the remaining block, and ends with rho = 0 once that block is solved.
The last residual r_m / zeta_m must then belong to x_m like any other: its distance dr from the
true residual is rounding, a few times 2^-53 ||b||."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

pytestmark = pytest.mark.gpu

# first iteration: block (2), b = 1; second: block ((1, 1), (1, 3)), b = (1, 0)
CASES = {1: (np.diag([1.0, 1.0, 2.0]), [1.0, 1.0j, 1.0]),
         2: (np.array([[4.0, 0, 0, 0], [0, 4.0, 0, 0], [0, 0, 1.0, 1.0], [0, 0, 1.0, 3.0]]), [1.0, 1.0j, 1.0, 0.0])}


@pytest.mark.parametrize("at", [1, 2])
@pytest.mark.parametrize("ns", [1, 5, 11])
def test_last_residual(cuda, at, ns):
    from paper_2506_09551_gb300 import api
    A, b = CASES[at]
    m = sp.csr_matrix(A)
    op = api.Operator.csr(m.indptr.astype(np.int64), m.indices.astype(np.int32), m.data)
    # device memory that a new allocation may get again, so that nothing unwritten reads as zero
    junk = torch.full((1 << 20,), float("nan"), dtype=torch.float64, device="cuda")
    del junk
    torch.cuda.empty_cache()
    shifts = np.concatenate([[0.0], 0.25 + np.arange(ns - 1) / 8.0]) + 0.0j
    shifts[1:] += 0.5j
    x, per, seeds, info, st = op.multishift_reseeded(torch.tensor(b, device="cuda"), shifts, maxit=100, max_seeds=1)
    assert info["iterations"] == at
    assert np.all(per["dr"] <= 32 * 2.0 ** -53 * np.linalg.norm(b)), per["dr"]
    r = np.array(b) - A @ x[0].cpu().numpy()
    assert np.linalg.norm(r) > 0.5 and r @ r == 0
