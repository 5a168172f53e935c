"""What the autotuner may choose for the solve, and what a solve reports of its per-shift update.

Iterations per graph have no effect where a window of iterations is one cooperative launch: the
trials time the same launches there, so the default has to stay."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
def test_default_block_stays_where_it_has_no_effect(cuda, prec):
    from paper_2506_09551_gb300 import api
    m = api.model(6, 3, 3)
    try:
        assert [api.autotune(m, prec, n_in)["block"] for n_in in (3, 5, 9, 11)] == [8 if prec else 4] * 4
    finally:
        api.autotune_forget()


@pytest.mark.parametrize("form", ["one", "sum"])
@pytest.mark.parametrize("prec,window", [(0, 56), (1, 32)])
@pytest.mark.parametrize("block", [1, 4, 16])
def test_flushes_are_the_launched_updates(cuda, form, prec, window, block):
    """One per window of iterations, and those of a block or window already in flight at the end."""
    from paper_2506_09551_gb300 import api
    op = api.Operator.hubbard(api.model(8, 4, 4, core_site=1), True)
    if form == "sum":
        op = api.Operator.direct_sum([op], [0.0])
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), dtype=api.cdtype(prec), device="cuda")
    _, _, info, _ = op.multishift_solve(b, np.linspace(-4.0, 5.0, 9), -0.3 - 0.3j, tol=0.0, maxit=100, block=block,
                                        prec=prec, allow_status=(5,))
    windows = -(-info["iterations"] // window)
    assert info["iterations"] == 100 and windows <= info["flushes"] <= windows + 3
