"""Solves in the forms that they fall back to, against the form they take first.

A ring of seed residuals that would take too much memory makes the window of the per-shift update
shorter.  FP32, and FP64 with fewer than eight shifts, keep the operations and their order:
bitwise equal.  FP64 with more shifts: one contraction per window, whose error is below that of
64 FMAs per window, over at most 60 windows of at least 16 iterations: 60 x 64 x 2^-53 = 4e-13,
times 2.5 for the growth of the terms: 1e-12 of the norm.

A cooperative launch that the runtime refuses (its CTAs do not all fit, as in a context limited to
part of the SMs) must leave the solve to the launch-per-product form.  The refusal is faked on
the host.  Bounds: the recursive residual is at most 1e-10 ||b|| (1e-6 in FP32), and its distance
from the true one about (iterations) 2^-53 ||A|| max ||x|| ~ 5e-10 (FP32, 2^-24 and the square
root of the iterations for independent roundings: 5e-5): 1e-9 and 1e-4."""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

C0 = -0.3 - 0.3j


@pytest.fixture
def limits(cuda, lib):
    lib.msb_test_solver_limits.argtypes = [C.c_int64, C.c_int]
    yield lib.msb_test_solver_limits
    lib.msb_test_solver_limits(0, 0)


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
    limits(0, 1)
    _, b = _check(op, prec, ns)
    # the fallback did run: three launches per iteration instead of one per window
    assert b["kernel_launches"] > 2 * b["iterations"] > 4 * a["kernel_launches"]


def _ring(op, window, prec):
    """Bytes of the ring of a window of iterations (slots of an even number of elements)."""
    return (window + 1) * ((op.dim + 1) // 2 * 2) * (8 if prec else 16)


@pytest.mark.parametrize("form", ["window", "launches"])
@pytest.mark.parametrize("kind", ["ring", "csr"])
@pytest.mark.parametrize("prec,ns", [(0, 5), (0, 21), (1, 5), (1, 21)])
def test_short_ring(limits, form, kind, prec, ns):
    op = _operator(kind)
    x, a = _check(op, prec, ns)
    for window in (32, 16, 4):
        limits(_ring(op, max(window, 16), prec) if window > 4 else 1, form == "launches")
        y, b = _check(op, prec, ns, block=4)
        assert b["device_bytes"] < a["device_bytes"] or (prec and window == 32)
        assert b["iterations"] == a["iterations"] or form == "launches"
        if form == "launches":              # another order of the sums: another recurrence in the last bits
            continue
        if prec or ns < 8:
            assert torch.equal(x, y)
        else:
            for k in range(ns):
                err = float(torch.linalg.vector_norm(x[k] - y[k]) / torch.linalg.vector_norm(x[k]))
                assert err <= 1e-12, (window, k, err)


@pytest.mark.parametrize("prec", [0, 1])
def test_short_ring_of_a_map(limits, prec):
    """The rows that a map keeps per shift, through every window."""
    from paper_2506_09551_gb300 import api
    m = api.model(6, 3, 3)
    w_in, w = np.linspace(-4.0, 12.0, 11), np.linspace(-1.0, 10.0, 30)
    p = api.map_params(precision=prec, **(dict(solve_tol=1e-6, cf_tol=1e-5) if prec else {}))
    I0 = api.rixs_map(m, p, w_in, w)[0]
    for ring in (33 * 300 * 16, 17 * 300 * 16, 1):
        limits(ring, 0)
        I = api.rixs_map(m, p, w_in, w)[0]
        assert np.array_equal(I, I0) if prec else np.linalg.norm(I - I0) <= 1e-10 * np.linalg.norm(I0)


@pytest.mark.parametrize("block", [1, 2])
def test_breakdown_in_a_later_window(limits, block):
    """The system of test_gpu_breakdown.py that ends at its second iteration, with windows of one and two."""
    from paper_2506_09551_gb300 import api
    op = api.Operator.csr(np.array([0, 1, 2, 4, 6]), np.array([0, 1, 2, 3, 2, 3], dtype=np.int32),
                          np.array([4.0, 4.0, 1.0, 1.0, 1.0, 3.0]))
    b = torch.tensor([1.0, 1.0j, 1.0, 0.0], dtype=torch.complex128, device="cuda")
    limits(1, 0)
    shifts = np.array([0.0, 0.25 + 0.5j, 0.375 + 0.5j])
    x, per, seeds, info, st = op.multishift_reseeded(b, shifts, maxit=100, max_seeds=1, block=block)
    assert info["iterations"] == 2 and np.all(per["dr"] <= 32 * 2.0 ** -53 * 3.0 ** 0.5), per["dr"]


@pytest.mark.parametrize("prec", [0, 1])
def test_capped_solves_take_no_longer_ring(cuda, prec):
    """Workspace of a solve of a few iterations: no more residuals than it can have."""
    from paper_2506_09551_gb300 import api
    op = _operator("ring")
    b = torch.tensor(workloads.random_complex_rhs(op.dim, 5), dtype=api.cdtype(prec), device="cuda")
    size = [op.multishift_solve(b, [0.0], C0, tol=0.0, maxit=m, block=4, prec=prec, allow_status=(5,))[2]["device_bytes"]
            for m in (3, 8, 9, 16, 17, 100)]
    slot = op.dim * (8 if prec else 16)
    assert size[1] - size[0] == 0 and size[2] - size[1] == 12 * slot and size[3] == size[2]
    assert size[4] - size[3] == 16 * slot and size[5] - size[4] == (0 if prec else 24 * slot)
