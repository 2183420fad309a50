"""Two threads, each with a context of its own size on a stream of its own: every call returns what it returns
alone (kernels shared by both sizes are launched with different amounts of shared memory)."""
import threading

import numpy as np
import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


def in_threads(calls, rounds):
    """calls: one function per thread, called `rounds` times at once and compared with its first result."""
    import torch
    want = [f() for f in calls]
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(calls))

    def run(k):
        try:
            start.wait()
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds):
                    got = calls[k]()
                    torch.cuda.current_stream().synchronize()
                    assert torch.equal(got, want[k])
        except BaseException as e:  # seen by the main thread
            errors.append(e)

    ts = [threading.Thread(target=run, args=(k,)) for k in range(len(calls))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]


def contexts(ls, sizes, L):
    out = []
    for N in sizes:
        w = synth.make_workload("ls_n10000_l10000", N=N, L=L, seed=N)
        ctx = ls.ls_create(w["h"])
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        out.append(ctx)
    return out


def test_widened_sets(ls):
    import torch
    sizes, L, K = (60, 3000), 40, 8
    ctxs = contexts(ls, sizes, L)

    def call(k):
        N = sizes[k]
        g = torch.Generator(device="cuda").manual_seed(N)
        idx = torch.sort(torch.rand(N, 2, N - 1, device="cuda", generator=g).argsort(dim=2)[:, :, :K], dim=2).values
        idx = (idx + (idx >= torch.arange(N, device="cuda").view(N, 1, 1))).int().contiguous()
        d = torch.empty(1, N, N, device="cuda")
        torch.cuda.synchronize()

        def f():
            ls.ls_sparse_run_all(ctxs[k], idx, K, 20, [L // 2], d, lookahead=2)
            return d.clone()
        return f

    try:
        in_threads([call(0), call(1)], 300)
    finally:
        for c in ctxs:
            ls.ls_destroy(c)


@pytest.mark.parametrize("sizes,L,loci", [((16500, 20000), 40, 30), ((21000, 40900), 20, 12)])
def test_table_moves(ls, sizes, L, loci):
    import torch
    ctxs = contexts(ls, sizes, L)
    tables = [ls.ls_table_create(c, ls.LS_FWD, 0, 4) for c in ctxs]

    def call(k):
        a = torch.empty(4, sizes[k], device="cuda")

        def f():
            ls.ls_table_reset(tables[k])
            ls.ls_forward(ctxs[k], tables[k], loci)
            ls.ls_table_read(tables[k], a)
            return a.clone()
        return f

    try:
        in_threads([call(0), call(1)], 500)
    finally:
        for t in tables:
            ls.ls_table_destroy(t)
        for c in ctxs:
            ls.ls_destroy(c)


def test_gradients(ls):
    import torch
    sizes, L, K = (9100, 10000), 12, 2
    ctxs = contexts(ls, sizes, L)

    def call(k):
        def f():
            return torch.tensor(ls.ls_pac_grad(ctxs[k], synth.rho_intervals(L, K), K, 0, 3)[3])
        return f

    try:
        in_threads([call(0), call(1)], 300)
    finally:
        for c in ctxs:
            ls.ls_destroy(c)
