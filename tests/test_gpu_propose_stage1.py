"""Stage 1 (threshold by bisection, block compaction) against the numpy oracle at the edges of its
layout: 16-donor chunks, 2048 donors a warp, several warps, ties at the threshold, C beyond the donors,
one and two windows."""
import numpy as np
import pytest

import oracle.proposal as op
from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N,L,C,w", [
    (2, 5, 1, 0), (17, 40, 16, 0), (17, 300, 40, 1), (2047, 600, 100, 1), (2049, 600, 1, 2), (2049, 256, 2048, 0),
    (4100, 1030, 333, 4)])
def test_stage1_matches_the_oracle(ls, N, L, C, w):
    import torch
    wl = synth.make_workload("ls_n50000_l20000", N=N, L=L, seed=N + L, founders=max(2, N // 100))
    ctx = ls.ls_create(wl["h"])
    try:
        cand = torch.empty((N, C), dtype=torch.int32, device="cuda")
        feat = torch.empty((N, C, 8), dtype=torch.float32, device="cuda")
        ls.ls_propose_window(ctx, C, w, cand, feat)
        cand, feat = cand.cpu().numpy(), feat.cpu().numpy()
        K = min(C, 512)
        idx = torch.empty((N, op.windows(L), K), dtype=torch.int32, device="cuda")
        ls.ls_propose(ctx, 0, K, None, idx)
        idx = idx.cpu().numpy()
    finally:
        ls.ls_destroy(ctx)
    M = {v: op.mismatch_counts(wl["h"], v) for v in range(max(0, w - 3), min(op.windows(L), w + 4))}
    score = sum(M[v] for v in (w - 1, w, w + 1) if v in M)
    rows = np.unique(np.r_[0, N - 1, np.random.default_rng(0).integers(0, N, 60)])
    for i in rows:
        js = np.delete(np.arange(N), i)
        order = js[np.lexsort((js, score[i, js]))]
        for got, n in ((cand[i], C), (idx[i, w], K)):
            want = np.full(n, -1)
            keep = np.sort(order[:n])
            want[:len(keep)] = keep
            np.testing.assert_array_equal(got, want)
        for d in range(7):
            v = min(max(w + d - 3, 0), op.windows(L) - 1)
            nv = np.float32(1.0) / np.float32(min(256, L - 256 * v))
            j = cand[i][cand[i] >= 0]
            f = np.float64(1.0) - M[v][i, j].astype(np.float64) * np.float64(nv)
            np.testing.assert_allclose(feat[i, :len(j), d], f, rtol=0, atol=2.0 ** -24)
