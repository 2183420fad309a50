"""Selection of the K best candidates (one warp per target, C/32 keys a lane): every key count of the
dispatch, C off a multiple of 32, C beyond the donors (padding), K = C, and tied scores."""
import numpy as np
import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N,C,K,ties", [
    (90, 1, 1, False), (150, 31, 7, False), (150, 128, 128, False), (150, 129, 40, True), (300, 256, 100, False),
    (300, 500, 330, False), (700, 513, 512, True), (1100, 1025, 512, False), (2100, 2048, 512, False)])
def test_topk_is_the_sorted_selection(ls, N, C, K, ties):
    import torch
    w = synth.make_workload("ls_n50000_l20000", N=N, L=300, seed=N + C, founders=max(8, N // 25))
    p = (np.random.default_rng(C).normal(0, 1, ls.LS_MLP_PARAMS) * 0.15).astype(np.float32)
    if ties:
        p[:-1] = 0.0  # every score is the output bias
    ctx = ls.ls_create(w["h"])
    m = ls.ls_mlp_create(p)
    try:
        idx = torch.empty((N, 2, K), dtype=torch.int32, device="cuda")
        ls.ls_propose(ctx, C, K, m, idx)
        cand = torch.empty((N, C), dtype=torch.int32, device="cuda")
        feat = torch.empty((N, C, 8), dtype=torch.float32, device="cuda")
        ls.ls_propose_window(ctx, C, 1, cand, feat)
        sc = torch.empty(N * C, dtype=torch.float32, device="cuda")
        ls.ls_mlp_forward(m, feat.reshape(N * C, 8), sc)
        sc, cand, idx = sc.reshape(N, C).cpu().numpy(), cand.cpu().numpy(), idx[:, 1].cpu().numpy()
    finally:
        ls.ls_mlp_destroy(m)
        ls.ls_destroy(ctx)
    for i in range(N):
        n = int((cand[i] >= 0).sum())
        order = np.lexsort((cand[i, :n], -sc[i, :n]))[:K]
        best = np.full(K, -1)
        best[:len(order)] = np.sort(cand[i, :n][order])
        np.testing.assert_array_equal(idx[i], best)
