"""Rows that start off a 16-byte boundary (N not a multiple of four) at the limits of every row kernel that takes
them (and next to them): posteriors of caller-held rows against float64, decoded distances against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N", [2045, 2047, 2049, 5118, 5119, 5121, 10236, 10237, 10238, 10239, 10240, 10241, 20477, 20478, 20481, 32765, 32766, 32769])
def test_posterior_rows(ls, N):
    import torch
    T, t0 = 5, N - 5
    g = torch.Generator(device="cuda").manual_seed(N)
    a, b = (torch.rand(T, N, device="cuda", generator=g) for _ in range(2))
    a[0] = 0.0  # a zero normaliser: p = eps for every donor
    flat = torch.full((T * N + 2,), -7.0, device="cuda")
    ctx = ls.ls_create(np.zeros((1, N), dtype=np.uint8))
    try:
        ls.ls_posterior_rows(ctx, a, b, t0, flat[:T * N].view(T, N))
        got = flat.cpu().double()
    finally:
        ls.ls_destroy(ctx)
    assert (got[T * N:] == -7.0).all()  # nothing behind the last row
    got = got[:T * N].view(T, N)
    ref = a.cpu().double() * b.cpu().double()
    ref[torch.arange(T), torch.arange(t0, t0 + T)] = 0.0
    ref[1:] /= ref[1:].sum(1, keepdim=True)
    ref[0] = 2.0 ** -52
    ref[0, t0] = 0.0
    # an FP32 sum of N positive terms in tree order and four roundings per entry
    assert torch.all((got - ref).abs() <= 2e-6 * ref)


@pytest.mark.parametrize("N", [2046, 2047, 2049, 5117, 5118, 5119, 5121])
def test_decoded_distances(ls, N):
    import torch
    L, loci = 6, [0, 3, 5]
    w = synth.make_workload("ls_n10000_l10000", N=N, L=L, seed=N)
    rows = np.unique(np.r_[0, 1, 31, 32, N - 2, N - 1, np.random.default_rng(N).integers(0, N, 30)]).astype(np.int32)
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], 1e-3)
        d = torch.empty(len(loci), N, N, device="cuda")
        assert ls.ls_run_all(ctx, loci, d)[0] == 0
        at = torch.from_numpy(rows).long().cuda()
        got = d[:, at][:, :, at].cpu().numpy()
    finally:
        ls.ls_destroy(ctx)
    post = oracle.run(w["h"], w["rho"], 1e-3, loci, targets=rows)["post"]
    for k in range(len(loci)):
        # relative errors of a posterior of some 1e-5 at most (an FP32 sum of N terms and a dozen roundings a
        # locus) move half a logarithm by half of that
        np.testing.assert_allclose(got[k], oracle.distance_block(post[:, k], rows), rtol=1e-6, atol=2e-5)
