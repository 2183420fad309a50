"""The gradient against the FP64 oracle where the scratch ceiling leaves blocks of fewer targets than the
several-target tiles hold, and in every tile with enough targets to be chosen for them."""
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


def run(ls, N, L, K, t0, t1, budget=None):
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
    check_grad(pac, gm, gr, ref, w["rho"], w["mu"], L, iv, K, t1 - t0, N)


# K groups of intervals take (3 K + 2) N floats a target; the ceiling of 1 MiB leaves `block` targets
@pytest.mark.parametrize("N,K,block", [(517, 11, 14), (517, 22, 7), (517, 170, 1), (1000, 11, 7), (1000, 86, 1), (1500, 15, 3),
                                       (1500, 58, 1), (2048, 13, 3), (3000, 29, 1)])
def test_blocks_below_a_tile(ls, N, K, block):
    assert max(1, (1 << 20) // ((3 * K + 2) * N * 4)) == block
    run(ls, N, max(60, K + 2), K, N - 17, N, "1")


# all targets, so that the several-target tiles are chosen (targets per CTA x quads: 8 x 4, 8 x 8, 8 x 16, 4 x 16,
# 4 x 20, 2 x 16, 2 x 20), at the edges of the ranges they serve
@pytest.mark.parametrize("N", [256, 257, 512, 513, 1024, 1025, 2048, 2049, 2560, 2561, 4097])
def test_all_targets(ls, N):
    run(ls, N, 40, 5, 0, N)
