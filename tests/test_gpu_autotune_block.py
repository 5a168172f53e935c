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
