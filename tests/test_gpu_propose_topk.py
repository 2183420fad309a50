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


# one row, around one tile, more tiles than SMs by one row; rows on and off a 16-byte boundary
@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 1, 152 * 128 * 2 + 5])
@pytest.mark.parametrize("offset", [0, 1])
def test_scorer_row_counts_and_alignment(ls, n, offset):
    import torch

    import oracle.proposal as op
    rng = np.random.default_rng(n)
    p = (rng.normal(0, 1, op.N_PARAMS) * 0.15).astype(np.float32)
    X = rng.random((n, 8)).astype(np.float32)
    m = ls.ls_mlp_create(p)
    try:
        flat = torch.zeros(8 * n + offset, device="cuda")
        Xd = flat[offset:].view(n, 8)
        Xd.copy_(torch.from_numpy(X))
        s = torch.full((n + 1,), 7.0, device="cuda")
        ls.ls_mlp_forward(m, Xd, s[:n])
        s = s.cpu().numpy().astype(np.float64)
    finally:
        ls.ls_mlp_destroy(m)
    assert s[n] == 7.0
    ref = op.mlp_forward_bf16(p.astype(np.float64), X.astype(np.float64))
    # FP32 accumulation against exact sums, and a hidden unit on a BF16 rounding boundary
    assert float(np.max(np.abs(s[:n] - ref))) <= 2e-3 * float(np.max(np.abs(ref)))
