"""The row-tiled Hubbard product (csrc/hubrows.cuh) at the sizes where its tiles can go wrong:
several short rows per CTA with a ragged last tile, rows of odd length, rows split over CTAs,
a single state per species, direct sums of uneven parts, many columns, and FP32 vectors that do
not start on a 16-byte boundary.  Bounds: a sum of at most 2 L + 1 terms, each rounded once or
twice, so (2 L + 4) half-ulps of the working precision in the 2-norm."""
import numpy as np
import pytest
import torch

from oracle import hubbard
import workloads

pytestmark = pytest.mark.gpu

CASES = [  # (L, n_up, n_dn, periodic, core or None, columns)
    (4, 0, 4, True, None, 1),      # one state per species
    (5, 2, 1, False, 4, 3),        # rows of 5: 25 rows per tile, one tile
    (6, 3, 2, True, None, 2),      # rows of 15: 8 rows per tile, ragged
    (8, 5, 4, True, 2, 1),
    (9, 4, 2, True, None, 5),      # rows of 36
    (9, 5, 4, False, 0, 2),
    (10, 5, 5, True, None, 1),     # rows of 252
    (12, 3, 6, True, 7, 1),        # rows of 924, split over several CTAs
    (13, 1, 6, True, None, 2),     # rows of 1716
]


def _bar(L, prec):
    return (2 * L + 4) * (2.0 ** -53 if prec == 0 else 2.0 ** -24)


def _op(case):
    L, nu, nd, per, core, _ = case
    return hubbard.hamiltonian(hubbard.Sector(L, nu, nd), 1.0, 8.0, 4.0, core, per)


def _api_op(api, case):
    L, nu, nd, per, core, _ = case
    m = api.model(L, nu - (core is not None), nd, core_site=core or 0, periodic=per)
    return api.Operator.hubbard(m, core is not None)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_apply(cuda, case, prec, shift):
    from paper_2506_09551_gb300 import api
    L, nvec = case[0], case[5]
    op, H = _api_op(api, case), _op(case)
    X = workloads.random_complex_vectors(op.dim, nvec, seed=L)
    if prec:
        X = X.astype(np.complex64).astype(np.complex128)
    c0 = 0.75 - 0.3j
    ref = (H @ X.T).T + c0 * X
    buf = torch.empty(shift + X.size, dtype=api.cdtype(prec), device="cuda")
    x = buf[shift:].view(nvec, op.dim)          # shift = 1: FP32 vectors start off a 16-byte boundary
    x.copy_(torch.tensor(X))
    y = op.apply(x, c0, prec).cpu().numpy()
    assert np.linalg.norm(y - ref) <= _bar(L, prec) * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("cases", [(2, 3, 8), (1, 6), (5, 4)])
def test_direct_sum(cuda, cases, prec):
    from paper_2506_09551_gb300 import api
    cs = [CASES[i] for i in cases]
    shifts = [0.5 * i - 0.25 for i in range(len(cs))]
    parts = [_api_op(api, c) for c in cs]
    op = api.Operator.direct_sum(parts, shifts)
    X = workloads.random_complex_vectors(op.dim, 2, seed=11)
    if prec:
        X = X.astype(np.complex64).astype(np.complex128)
    c0 = -1.5 + 0.3j
    ref, off = np.empty_like(X), 0
    for c, s, p in zip(cs, shifts, parts):
        ref[:, off:off + p.dim] = (_op(c) @ X[:, off:off + p.dim].T).T + (s + c0) * X[:, off:off + p.dim]
        off += p.dim
    y = op.apply(torch.tensor(X, dtype=api.cdtype(prec), device="cuda"), c0, prec).cpu().numpy()
    assert np.linalg.norm(y - ref) <= _bar(13, prec) * np.linalg.norm(ref)
