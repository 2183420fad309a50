"""Short table moves (row kernel: one target per CTA, the row in registers) against the FP64 oracle, over
quads and rows off the 16-byte grid, every elements-per-thread variant and its limits, stores, resumes,
per-locus mu, target ranges, and rows handed in off a 16-byte boundary."""
import numpy as np
import pytest

import oracle
from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def close(got, ref, own):
    """FP32 recursion of a few loci: each entry within 2e-6 relative (a dozen roundings)"""
    ref = np.array(ref)
    at = np.arange(len(own)), own  # the target's own entry is stored as 0
    assert np.all(got[at] == 0.0)
    ref[at] = 0.0
    assert np.all(np.abs(got - ref) <= 2e-6 * np.abs(ref) + 1e-35), float(np.max(np.abs(got - ref) / (np.abs(ref) + 1e-35)))


@pytest.mark.parametrize("N", [2, 3, 31, 33, 128, 1023, 2048, 2052, 2049, 5120, 5124, 10240, 10244, 20477, 20480])
@pytest.mark.parametrize("mu_kind,offset", [("scalar", 0), ("locus", 1)])
def test_short_moves_match_the_oracle(ls, N, mu_kind, offset):
    import torch
    L = 12
    w = synth.make_workload("ls_n200_l1000", N=N, L=L, seed=N, founders=min(N, 20))
    mu = 1e-3 if mu_kind == "scalar" else np.random.default_rng(N).uniform(1e-4, 1e-2, L)
    T = np.unique(np.r_[0, N // 2, N - 1, np.random.default_rng(1).integers(0, N, 5)])
    t0, t1 = (0, N) if N <= 2100 else (N - 300, N)
    T = T[(T >= t0) & (T < t1)]
    if len(T) == 0:
        T = np.array([t0, t1 - 1])
    ref = oracle.run(w["h"], w["rho"], mu, np.arange(L), targets=T.astype(np.int32), want=("alpha", "beta", "logF", "logG"))
    ctx = ls.ls_create(w["h"])
    tabs = []
    try:
        ls.ls_set_params(ctx, w["rho"], mu)
        n = t1 - t0
        fw, bw = ls.ls_table_create(ctx, ls.LS_FWD, t0, t1), ls.ls_table_create(ctx, ls.LS_BWD, t0, t1)
        tabs = [fw, bw]
        flat = torch.empty(2 * n * N + offset, device="cuda")
        out = flat[offset:].view(2, n, N)
        state, lg = torch.empty(n, N, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
        rows = T - t0

        def check(t, key, lkey, l):
            ls.ls_table_read(t, state, lg)
            close(state[rows].cpu().numpy(), ref[key][:, l], T)
            np.testing.assert_allclose(lg[rows].cpu().numpy(), ref[lkey][:, l], rtol=1e-6, atol=1e-6)
        ls.ls_forward(ctx, fw, 0)
        check(fw, "alpha", "logF", 0)
        ls.ls_forward(ctx, fw, 1)
        check(fw, "alpha", "logF", 1)
        ls.ls_forward(ctx, fw, 4, [2, 4], out)
        close(out[0][rows].cpu().numpy(), ref["alpha"][:, 2], T)
        close(out[1][rows].cpu().numpy(), ref["alpha"][:, 4], T)
        check(fw, "alpha", "logF", 4)
        ls.ls_backward(ctx, bw, L - 1)
        check(bw, "beta", "logG", L - 1)
        ls.ls_backward(ctx, bw, L - 2)
        check(bw, "beta", "logG", L - 2)
        ls.ls_backward(ctx, bw, L - 4, [L - 3, L - 4], out)
        close(out[0][rows].cpu().numpy(), ref["beta"][:, L - 3], T)
        close(out[1][rows].cpu().numpy(), ref["beta"][:, L - 4], T)
        check(bw, "beta", "logG", L - 4)
    finally:
        for t in tabs:
            ls.ls_table_destroy(t)
        ls.ls_destroy(ctx)
