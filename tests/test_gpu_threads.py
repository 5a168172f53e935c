"""Two host threads with rows of different length: the limit of a kernel's dynamic shared memory is
process-wide, so a thread with short rows must not lower it under the launches of the other.
Every call has to succeed and to give what it gives alone (the products bit for bit; the
continued fraction at a fixed depth too: its sums are taken in a fixed order)."""
import threading

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

SECTORS = [(14, 1, 7), (15, 1, 7)]         # rows of 3,432 and 6,435 down-spin states


def _together(work, reps):
    alone = [w() for w in work]
    errors, start = [], threading.Barrier(len(work))

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(reps):
                    got = work[i]()
                assert np.array_equal(got, alone[i])
        except Exception as e:              # reported by the main thread
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def _ops():
    from paper_2506_09551_gb300 import api
    return [api.Operator.hubbard(api.model(L, nu, nd)) for L, nu, nd in SECTORS]


def test_applies(cuda):
    ops = _ops()
    xs = [torch.tensor(workloads.random_complex_rhs(op.dim, 3), device="cuda")[None] for op in ops]

    def work(i):
        def once():
            for _ in range(50):
                y = ops[i].apply(xs[i], 0.5 - 0.1j)
            return y.cpu().numpy()
        return once

    _together([work(0), work(1)], 40)


def test_continued_fractions(cuda):
    ops = _ops()
    w = np.linspace(0.0, 5.0, 7)
    xs = [torch.tensor(workloads.random_complex_rhs(op.dim, 3), device="cuda")[None] for op in ops]

    def work(i):
        return lambda: np.asarray(ops[i].continued_fraction(xs[i], -3.0, w, 0.1, cf_tol=0.0, cf_check=40, cf_maxdepth=40)[0])

    _together([work(0), work(1)], 30)
