"""Stage 1 beyond 16384 donors (blocks of 9 to 32 warps) and beyond 65536 (the histogram kernel): candidates and
features of sampled targets against the order of the mismatch sums."""
import numpy as np
import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N,C", [(16384, 300), (16385, 300), (18433, 2048), (40000, 1), (65536, 65), (65537, 65), (65600, 700)])
@pytest.mark.parametrize("L,w", [(200, 0), (520, 1)])
def test_sets_and_features(ls, N, C, L, w):
    import torch
    wl = synth.make_workload("ls_n50000_l20000", N=N, L=L, seed=N + L, founders=400)
    h, Wn = wl["h"], (L + 255) // 256
    ctx = ls.ls_create(h)
    try:
        cand = torch.empty((N, C), dtype=torch.int32, device="cuda")
        feat = torch.empty((N, C, 8), dtype=torch.float32, device="cuda")
        ls.ls_propose_window(ctx, C, w, cand, feat)
        rows = np.unique(np.r_[0, N - 1, 2047, 2048, np.random.default_rng(0).integers(0, N, 12)])
        at = torch.from_numpy(rows).cuda()
        cand, feat = cand[at].cpu().numpy(), feat[at].cpu().numpy()
    finally:
        ls.ls_destroy(ctx)
    for k, i in enumerate(rows):
        M = {}
        for v in range(max(0, w - 3), min(Wn, w + 4)):
            block = h[256 * v:256 * (v + 1)]
            M[v] = np.minimum((block != block[:, i:i + 1]).sum(0), 255)
        score = sum(M[v] for v in (w - 1, w, w + 1) if v in M)
        score[i] = 1 << 20  # never its own donor
        want = np.sort(np.lexsort((np.arange(N), score))[:C])
        np.testing.assert_array_equal(cand[k], want)
        for d in range(7):
            v = min(max(w + d - 3, 0), Wn - 1)
            inv = np.float32(1.0) / np.float32(min(256, L - 256 * v))
            f = 1.0 - M[v][want].astype(np.float64) * np.float64(inv)
            np.testing.assert_allclose(feat[k, :, d], f, rtol=0, atol=2.0 ** -24)  # one rounding of a value up to 1
        assert not feat[k, :, 7].any()
