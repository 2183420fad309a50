"""Posteriors of caller-held rows (one row per CTA in registers, or two passes) against float64 at the
limits of every variant: row lengths on and off the quad grid, buffers off a 16-byte boundary, a zero
normaliser, and the target's own entry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("N", [2, 4, 5, 2048, 2052, 5120, 5124, 20480, 20484, 32768, 32772])
@pytest.mark.parametrize("offset", [0, 1])
def test_posterior_rows(ls, N, offset):
    import torch
    T, t0 = min(N, 5), max(0, N - 5)
    h = np.zeros((1, N), dtype=np.uint8)
    g = torch.Generator(device="cuda").manual_seed(N)
    flat = torch.zeros(3, T * N + 4, device="cuda")
    a, b, p = (f[offset:offset + T * N].view(T, N) for f in flat)
    a.copy_(torch.rand(T, N, device="cuda", generator=g))
    b.copy_(torch.rand(T, N, device="cuda", generator=g))
    a[0] = 0.0  # a zero normaliser: p = eps for every donor
    ctx = ls.ls_create(h)
    try:
        ls.ls_posterior_rows(ctx, a, b, t0, p)
        got = p.cpu().double()
    finally:
        ls.ls_destroy(ctx)
    ref = a.cpu().double() * b.cpu().double()
    ref[torch.arange(T), torch.arange(t0, t0 + T)] = 0.0
    ref[1:] /= ref[1:].sum(1, keepdim=True)
    ref[0] = 2.0 ** -52
    ref[0, t0] = 0.0
    # an FP32 sum of N positive terms in tree order and four roundings per entry
    assert torch.all((got - ref).abs() <= 2e-6 * ref)
