"""One target per CTA of 8 warps, the whole state in registers (N in (20480, 40960]): distances of the fused
pipeline and resumed tables against the FP64 oracle on sampled targets, at the edges of every slice width,
with scalar and per-locus mu."""
import numpy as np
import pytest

import oracle
from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N,mu_kind", [(20481, "scalar"), (24576, "locus"), (24577, "scalar"), (28672, "scalar"),
                                       (28673, "locus"), (32769, "scalar"), (36865, "scalar"), (40960, "locus")])
def test_sampled_targets(ls, N, mu_kind):
    import torch
    L = 34  # past one fold of the log scales and several staged blocks
    w = synth.make_workload("ls_n50000_l20000", N=N, L=L, seed=N, founders=100)
    mu = 1e-4 if mu_kind == "scalar" else np.random.default_rng(N).uniform(1e-5, 1e-2, L)
    loci = np.array([0, 20, L - 1], dtype=np.int32)
    T = np.unique(np.r_[0, N // 3, N - 1]).astype(np.int32)
    ref = oracle.run(w["h"], w["rho"], mu, loci, targets=T, want=("post", "alpha", "llf"))
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], mu)
        d = torch.empty(len(loci), N, N, device="cuda")
        ls.ls_run_all(ctx, loci, d)
        for k in range(len(loci)):
            want = oracle.distance_block(ref["post"][:, k, :], T)
            got = d[k][T][:, T].cpu().numpy().astype(np.float64)
            assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(np.abs(want), 1.0))
        del d
        t = ls.ls_table_create(ctx, ls.LS_FWD, N - 40, N)
        try:
            out = torch.empty(40, N, device="cuda")
            ls.ls_forward(ctx, t, 12)
            ls.ls_forward(ctx, t, L - 1)  # resumed from the table
            ls.ls_table_read(t, out)
            a = out[39].cpu().numpy()
            big = ref["alpha"][-1, 2] > 1e-30
            assert np.all(np.abs(a - ref["alpha"][-1, 2])[big] <= 2e-4 * ref["alpha"][-1, 2][big])
        finally:
            ls.ls_table_destroy(t)
    finally:
        ls.ls_destroy(ctx)
