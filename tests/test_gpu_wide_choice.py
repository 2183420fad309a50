"""N in (20480, 40960]: calls of few loci per row transfer run the kernel with its state in registers and shared
memory, long ones the wide register tile.  Each against the other over the calls that take them (the moves of a
table, with stored rows; the fused pipeline) at the edges of every width, with both kinds of mu."""
import os

import numpy as np
import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def pinned(variant, f):
    if variant:
        os.environ["LS_PROP_VARIANT"] = variant
    try:
        return f()
    finally:
        os.environ.pop("LS_PROP_VARIANT", None)


def close(a, b):
    # the same FP32 recursion in another order of summation: the row sums differ by a few roundings a locus, which
    # the normalisation takes out again
    big = b.abs() > 1e-30
    return bool(((a - b).abs()[big] <= 2e-5 * b.abs()[big]).all())


@pytest.mark.parametrize("mu_kind", ["scalar", "locus"])
@pytest.mark.parametrize("N,quads", [(20481, 24), (24576, 24), (24577, 28), (28673, 32), (32769, 36), (36865, 40), (40960, 40)])
def test_tile_and_large_n_kernel_agree(ls, N, quads, mu_kind):
    import torch
    L, T = 70, 5
    w = synth.make_workload("ls_n50000_l20000", N=N, L=L, seed=N, founders=100)
    mu = 1e-4 if mu_kind == "scalar" else np.random.default_rng(N).uniform(1e-5, 1e-2, L)
    hyb = "1,16,%d" % (12 + 2 * ((-(-N // 2048) - 11) // 2))
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], mu)
        for kind, move in ((ls.LS_FWD, ls.ls_forward), (ls.LS_BWD, ls.ls_backward)):
            first, steps = (0, [3, 5, 66, 69]) if kind == ls.LS_FWD else (L - 1, [66, 64, 3, 0])
            stored = [40, 41, 66] if kind == ls.LS_FWD else [40, 39, 3]
            got = {}
            for variant in (None, "1,8,%d" % quads, hyb):
                def run():
                    t = ls.ls_table_create(ctx, kind, N - T, N)
                    try:
                        out, s = torch.empty(T, N, device="cuda"), torch.empty(3, T, N, device="cuda")
                        log = torch.empty(T, dtype=torch.float64, device="cuda")
                        move(ctx, t, first)
                        for k, to in enumerate(steps):
                            move(ctx, t, to, stored if k == 2 else None, s if k == 2 else None)
                        ls.ls_table_read(t, out, log)
                        torch.cuda.synchronize()
                        return out, s, log
                    finally:
                        ls.ls_table_destroy(t)
                got[variant] = pinned(variant, run)
            ref = got[hyb]
            for v in (None, "1,8,%d" % quads):
                assert close(got[v][0], ref[0]) and close(got[v][1], ref[1])
                assert torch.allclose(got[v][2], ref[2], rtol=1e-6, atol=1e-6 * L)
    finally:
        ls.ls_destroy(ctx)
