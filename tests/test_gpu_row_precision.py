"""The row sums of single table steps round no further than short chains of additions do: rows of equal values (all
donors match), whose roundings are the same in every thread and do not cancel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def test_sums_of_even_rows(ls):
    import torch
    mu = 2.0 ** -10  # exact in FP32, as 1 - mu is
    errors = []
    for N in (3000, 4500, 5000, 7000, 8500, 9000, 10000, 11000, 12000, 14000, 15000, 17000, 18000, 20000):
        ctx = ls.ls_create(np.zeros((2, N), dtype=np.uint8))
        t = None
        try:
            ls.ls_set_params(ctx, np.full(1, 1e-3), mu)
            t = ls.ls_table_create(ctx, ls.LS_FWD, 0, 4)
            ls.ls_forward(ctx, t, 0)
            log = torch.empty(4, dtype=torch.float64, device="cuda")
            ls.ls_table_read(t, torch.empty(4, N, device="cuda"), log)
            errors.append(float(log[0]) - np.log1p(-mu))  # N - 1 equal entries (1 - mu) / (N - 1)
        finally:
            if t is not None:
                ls.ls_table_destroy(t)
            ls.ls_destroy(ctx)
    # the prior and the product each round by 2^-24 / sqrt(3) (root mean square), a chain of ten additions by
    # sqrt(10 / 9) 2^-24: 8e-8 in all, and twice that allowed
    assert np.sqrt(np.mean(np.square(errors))) <= 1.6e-7, errors
