"""Memory that the library keeps between calls does not keep its own allocations from succeeding."""
import numpy as np
import pytest

import oracle
from paper_2212_11403_gb300 import synth
from tests.test_gpu_grad import check_grad

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def test_table_fits_beside_kept_scratch(ls):
    import torch
    w = synth.make_workload("ls_n10000_l10000", N=1000, L=200, seed=3)
    K, N = 160, 16000
    ctx, big = ls.ls_create(w["h"]), ls.ls_create(np.zeros((2, N), dtype=np.uint8))
    table, full = None, None
    try:
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        ls.ls_set_params(big, np.full(1, 1e-3), 1e-3)
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ls.ls_pac_grad(ctx, synth.rho_intervals(200, K), K)  # 1.9 GB of scratch
        free = torch.cuda.mem_get_info()[0]
        assert before - free > 1.5e9  # kept for the next call
        full = torch.empty(free - (600 << 20), dtype=torch.uint8, device="cuda")
        table = ls.ls_table_create(big, ls.LS_FWD, 0, N)  # 1.0 GB
        ls.ls_forward(big, table, 1)
        torch.cuda.synchronize()
    finally:
        del full
        torch.cuda.empty_cache()
        if table is not None:
            ls.ls_table_destroy(table)
        ls.ls_destroy(big)
        ls.ls_destroy(ctx)


def test_scratch_beyond_what_is_kept(ls):
    """4.8 GB of scratch: the oracle's gradient, and no more than 4 GB held afterwards."""
    import torch
    N, L, K = 1000, 420, 400
    w = synth.make_workload("ls_n10000_l10000", N=N, L=L, seed=4)
    iv = synth.rho_intervals(L, K)
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        rc, pac, gm, gr = ls.ls_pac_grad(ctx, iv, K)
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] <= 4 << 30
    finally:
        ls.ls_destroy(ctx)
    assert rc == 0
    check_grad(pac, gm, gr, oracle.pac_grad(w["h"], w["rho"], w["mu"], iv, K), w["rho"], w["mu"], L, iv, K, N, N)
