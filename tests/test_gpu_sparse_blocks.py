"""The restricted chain against its float64 oracle where its blocks of 64 loci, its slot counts and its
emission sense can go wrong: ragged L, windows shorter than, equal to and across blocks, every slots-per-lane
variant, mu beyond 1/2 and per locus, with and without the pool."""
import numpy as np
import pytest

import oracle.proposal as op
from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N,L,WS,K,lookahead,mu,pool", [
    (12, 1, 4, 3, 0, 1e-3, True), (20, 63, 64, 5, 2, 1e-3, True), (20, 64, 10, 19, 0, 0.7, True),
    (20, 65, 65, 6, 1, 0.7, False), (24, 130, 100, 9, 2, "locus", True), (80, 129, 64, 70, 0, 1e-2, True),
    (150, 40, 33, 130, 0, 1e-2, False), (280, 20, 16, 257, 0, 1e-2, True), (540, 4, 2, 520, 0, 1e-2, True)])
def test_blocks_and_slots(ls, N, L, WS, K, lookahead, mu, pool):
    import torch
    rng = np.random.default_rng(N + L)
    w = synth.random_tiny(rng, N, L)
    h, rho = w["h"], rng.uniform(0.01, 0.3, L - 1)
    mu = rng.choice([1e-3, 0.02, 0.6], size=L) if mu == "locus" else mu
    Wn = (L + WS - 1) // WS
    S = -np.ones((N, Wn, K), dtype=np.int32)
    for i in range(N):
        for q in range(Wn):
            n = min(N - 1, max(1, K - (i + q) % 3))
            S[i, q, :n] = np.sort(rng.choice(np.delete(np.arange(N), i), size=n, replace=False))
    loci = np.unique([0, L // 2, L - 1]).astype(np.int32)
    ctx = ls.ls_create(h)
    try:
        ls.ls_set_params(ctx, rho, mu)
        d = torch.empty((len(loci), N, N), device="cuda")
        _, pac, _ = ls.ls_sparse_run_all(ctx, torch.from_numpy(S).cuda(), K, WS, loci, d, lookahead=lookahead, pool=pool)
        d = d.cpu().numpy().astype(np.float64)
    finally:
        ls.ls_destroy(ctx)
    U = op.lookahead_sets(S, lookahead) if lookahead else S
    P = op.sparse_posteriors(h, rho, mu, U, WS, loci, pool)
    for k, l in enumerate(loci):
        hd = -0.5 * np.log(np.maximum(P[:, k, :], 2.0 ** -52))
        ref = hd + hd.T
        inset = np.zeros((N, N), dtype=bool)
        for i in range(N):
            v = U[i, l // WS]
            inset[i, v[v >= 0]] = True
        both = inset & inset.T
        np.fill_diagonal(both, False)
        if pool:
            both = ~np.eye(N, dtype=bool)
        got, want = d[k][both], ref[both]
        # FP32 recursions over at most 130 loci: the distance bound of the dense parity tests
        assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(np.abs(want), 1.0)), float(np.max(np.abs(got - want)))
