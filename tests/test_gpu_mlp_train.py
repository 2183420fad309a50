"""Gradient and Adam training of the proposal network at the edges of its row tiles (64 rows, whole
grids of CTAs, splits of dW2) against the float64 oracle."""
import numpy as np
import pytest

import oracle.proposal as op

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def problem(n, seed):
    rng = np.random.default_rng(seed)
    p = (rng.normal(0, 1, op.N_PARAMS) * 0.15).astype(np.float32)
    return p, rng.random((n, 8)).astype(np.float32), rng.random(n).astype(np.float32)


# one row; around a 64-row tile; around one split of 128 rows; more tiles than resident CTAs (304), ragged
@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 129, 1000, 304 * 64 + 1])
def test_gradient_row_tiles(ls, n):
    import torch
    p, X, y = problem(n, n)
    m = ls.ls_mlp_create(p)
    try:
        # an input whose rows start off a 16-byte boundary
        flat = torch.empty(8 * n + 1, device="cuda")
        Xd = flat[1:].view(n, 8)
        Xd.copy_(torch.from_numpy(X))
        g, loss = ls.ls_mlp_grad(m, Xd, torch.from_numpy(y).cuda())
    finally:
        ls.ls_mlp_destroy(m)
    rl, rg = op.mlp_loss_grad(p.astype(np.float64), X.astype(np.float64), y.astype(np.float64))
    # FP32 products and sums of 256 terms of either sign: about sqrt(256) 2^-24 of the terms' size
    assert abs(loss - rl) <= 1e-5 * rl
    assert float(np.linalg.norm(g - rg)) <= 1e-5 * float(np.linalg.norm(rg))


# every tile height (2, 4, 6, 7, 8 rows a warp) with its most CTAs, ragged
@pytest.mark.parametrize("n", [15, 17, 304 * 16, 304 * 32 - 5, 304 * 48 - 1, 304 * 56 - 3, 304 * 64])
def test_gradient_tile_heights(ls, n):
    import torch
    p, X, y = problem(n + n // 8 + 50, n)
    # rows with a pre-activation at the kink of a ReLU are left out: FP32 and float64 may take different
    # sides there, which moves the gradient by a row's whole share of a unit
    W1, b1, W2, b2, _, _ = op.unpack(p)
    Z1 = X.astype(np.float64) @ W1 + b1
    Z2 = np.maximum(Z1, 0.0) @ W2 + b2
    keep = np.flatnonzero((np.abs(Z1).min(1) > 1e-5) & (np.abs(Z2).min(1) > 1e-5))[:n]
    assert len(keep) == n
    X, y = X[keep], y[keep]
    m = ls.ls_mlp_create(p)
    try:
        g, loss = ls.ls_mlp_grad(m, torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    finally:
        ls.ls_mlp_destroy(m)
    rl, rg = op.mlp_loss_grad(p.astype(np.float64), X.astype(np.float64), y.astype(np.float64))
    assert abs(loss - rl) <= 1e-5 * rl
    # FP32 products and sums of 256 terms of either sign: about sqrt(256) 2^-24 of the terms' size
    assert float(np.linalg.norm(g - rg)) <= 1e-5 * float(np.linalg.norm(rg))


@pytest.mark.parametrize("n,batch", [(5, 64), (1000, 100), (3000, 777)])
def test_training_matches_adam_in_float64(ls, n, batch):
    import torch
    steps, lr, seed = 3, 1e-3, 12345
    p, X, y = problem(n, 7 + n)
    m = ls.ls_mlp_create(p)
    try:
        loss = ls.ls_mlp_train(m, torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), steps, batch, lr, seed)
        w = ls.ls_mlp_get(m)
    finally:
        ls.ls_mlp_destroy(m)
    mask = (1 << 64) - 1
    state, q = seed, p.astype(np.float64)
    m1, m2 = np.zeros_like(q), np.zeros_like(q)
    for it in range(1, steps + 1):
        rows = np.empty(batch, dtype=np.int64)
        for r in range(batch):  # splitmix64, modulo the number of rows
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            rows[r] = (z ^ (z >> 31)) % n
        rl, g = op.mlp_loss_grad(q, X[rows].astype(np.float64), y[rows].astype(np.float64))
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        q = q - lr * (m1 / (1 - 0.9 ** it)) / (np.sqrt(m2 / (1 - 0.999 ** it)) + 1e-8)
    assert abs(loss - rl) <= 1e-5 * rl  # the last of three steps is the tail
    # an update is lr g / |g| in its first step: a gradient entry's relative error (1e-5 of the norm
    # spread over entries of all sizes) enters it directly
    assert float(np.linalg.norm(w - q)) <= 1e-3 * float(np.linalg.norm(q - p))
