"""Small data sets run forward and backward side by side: the same distances, log-likelihood and status
as one after the other, bit for bit, at the limits of the rule (N = 1216), across calls that grow the
scratch, on a user's stream, under capture, with a prior matrix and with per-locus mu."""
import os

import numpy as np
import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def in_turn(ls, ctx, loci, d, **kw):
    os.environ["LS_TAIL_OVERLAP"] = "0"
    try:
        return ls.ls_run_all(ctx, loci, d, **kw)
    finally:
        del os.environ["LS_TAIL_OVERLAP"]


@pytest.mark.parametrize("N,kind", [(2, "mu"), (33, "scalar"), (200, "prior"), (200, "mu"), (1003, "scalar"), (1216, "scalar"),
                                    (1217, "scalar")])
def test_same_results_as_one_after_the_other(ls, N, kind):
    import torch
    L = 40
    w = synth.make_workload("ls_n200_l1000", N=N, L=L, seed=N, founders=min(N, 20))
    mu = np.random.default_rng(N).uniform(1e-4, 0.7, L) if kind == "mu" else w["mu"]
    Pi = torch.from_numpy(synth.gamma_prior_f32(N, N)).cuda() if kind == "prior" else None
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], mu, Pi)
        for D in (1, 4, 2):
            loci = synth.decode_loci(L, D)
            a, b = (torch.empty(D, N, N, device="cuda") for _ in range(2))
            sa, sb = (torch.empty(N, dtype=torch.int32, device="cuda") for _ in range(2))
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                ra = ls.ls_run_all(ctx, loci, a, status_out=sa)
            stream.synchronize()
            rb = in_turn(ls, ctx, loci, b, status_out=sb)
            torch.cuda.synchronize()
            assert ra == rb and torch.equal(a, b) and torch.equal(sa, sb)
        assert ls.ls_run_all(ctx, [], torch.empty(0, N, N, device="cuda")) == in_turn(ls, ctx, [], torch.empty(0, N, N, device="cuda"))
    finally:
        ls.ls_destroy(ctx)


@pytest.mark.parametrize("warm", [False, True])
def test_capture(ls, warm):
    import torch
    N, L = 150, 30
    w = synth.make_workload("ls_n200_l1000", N=N, L=L, seed=5)
    loci = synth.decode_loci(L, 3)
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        a, b = (torch.zeros(3, N, N, device="cuda") for _ in range(2))
        if warm:  # the scratch is there before the capture
            ls.ls_run_all(ctx, loci, a)
            a.zero_()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            ls.ls_run_all(ctx, loci, a, want_pac=False)
        graph.replay()
        torch.cuda.synchronize()
        in_turn(ls, ctx, loci, b)
        assert torch.equal(a, b)
        del graph
    finally:
        ls.ls_destroy(ctx)
