"""The two forms of a plain apply, row-tiled and element by element, each forced at every size of
test_gpu_hub_rows.py with its references and bounds, and left to their rule on both sides of its
lines, where the two have to agree within those bounds."""
import ctypes as C

import numpy as np
import pytest
import torch

import test_gpu_hub_rows as rows
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture
def form(cuda, lib):
    lib.msb_test_apply_form.argtypes = [C.c_int]
    yield lib.msb_test_apply_form
    lib.msb_test_apply_form(0)


@pytest.mark.parametrize("case", rows.CASES)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("which", [1, 2])
def test_forced(form, cuda, case, prec, which):
    form(which)
    rows.test_apply(cuda, case, prec, 0)


@pytest.mark.parametrize("cases", [(2, 3, 8), (1, 6), (5, 4)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("which", [1, 2])
def test_forced_sum(form, cuda, cases, prec, which):
    form(which)
    rows.test_direct_sum(cuda, cases, prec)


LINES = [  # (L, n_up, n_dn, vectors): few long rows, odd rows, short rows, each side of a line
    (13, 1, 7, 1), (13, 1, 7, 6), (12, 2, 7, 1), (12, 2, 7, 6), (14, 2, 6, 1), (13, 4, 5, 1), (13, 4, 5, 2),
    (14, 6, 2, 1), (14, 12, 1, 1), (15, 1, 8, 1), (15, 1, 8, 4), (13, 3, 9, 1), (13, 3, 9, 5)]


@pytest.mark.parametrize("case", LINES)
@pytest.mark.parametrize("prec", [0, 1])
def test_rule(form, case, prec):
    from paper_2506_09551_gb300 import api
    L, nu, nd, nvec = case
    op = api.Operator.hubbard(api.model(L, nu, nd))
    x = torch.tensor(workloads.random_complex_vectors(op.dim, nvec, seed=L), dtype=api.cdtype(prec), device="cuda")
    out = []
    for which in (0, 1, 2):
        form(which)
        out.append(op.apply(x, 0.75 - 0.3j, prec).to(torch.complex128))
    norm = float(torch.linalg.vector_norm(out[2]))
    assert torch.equal(out[0], out[1]) or torch.equal(out[0], out[2])
    assert float(torch.linalg.vector_norm(out[1] - out[2])) <= 2 * rows._bar(L, prec) * norm
