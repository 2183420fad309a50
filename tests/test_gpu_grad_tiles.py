"""The gradient against the FP64 oracle in every statistic-pass tile (targets per CTA x quads per lane) at the
edges of its range, with a ragged last CTA, a target range off the tile and blocks smaller than a tile."""
import os

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


@pytest.mark.parametrize("N,t0,t1,budget", [(129, 0, 129, None), (256, 3, 250, None), (257, 0, 257, None), (513, 500, 513, None),
                                            (512, 0, 20, "1"), (1025, 1000, 1025, None), (2048, 2030, 2048, None),
                                            (2049, 0, 17, None), (2561, 2550, 2561, None), (4096, 4090, 4096, None), (4097, 0, 9, None), (5121, 0, 9, None), (8193, 0, 5, None)])
def test_every_tile(ls, N, t0, t1, budget):
    L, K = 60, 7
    w = synth.make_workload("ls_n10000_l10000", N=N, L=L, seed=N)
    iv = synth.rho_intervals(L, K)
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        if budget:
            os.environ["LS_GRAD_BUDGET_MB"] = budget
        try:
            rc, pac, gm, gr = ls.ls_pac_grad(ctx, iv, K, t0, t1)
        finally:
            os.environ.pop("LS_GRAD_BUDGET_MB", None)
    finally:
        ls.ls_destroy(ctx)
    assert rc == 0
    ref = oracle.pac_grad(w["h"], w["rho"], w["mu"], iv, K, targets=np.arange(t0, t1, dtype=np.int32))
    check_grad(pac, gm, gr, ref, w["rho"], w["mu"], L, iv, K, N, t1 - t0)
