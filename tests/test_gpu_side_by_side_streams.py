"""Small data sets, several calls of one context in flight at once (from one thread or two, each on a stream
of its own): the same distances as one call after the other, bit for bit."""
import os
import threading

import pytest

from paper_2212_11403_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("threads", [1, 2])
@pytest.mark.parametrize("N,L", [(200, 300), (1003, 60)])
def test_calls_on_two_streams(ls, N, L, threads):
    import torch
    w = synth.make_workload("ls_n200_l1000", N=N, L=L, seed=N, founders=20)
    ctx = ls.ls_create(w["h"])
    try:
        ls.ls_set_params(ctx, w["rho"], w["mu"])
        sets = [[k, L // 2 - k, L - 1 - k] for k in range(8)]  # another set of decode loci in every call
        want = []
        os.environ["LS_TAIL_OVERLAP"] = "0"
        try:
            for loci in sets:
                want.append(torch.empty(3, N, N, device="cuda"))
                ls.ls_run_all(ctx, loci, want[-1])
        finally:
            del os.environ["LS_TAIL_OVERLAP"]
        got = [torch.zeros_like(x) for x in want]
        streams = [torch.cuda.Stream() for _ in range(2)]
        torch.cuda.synchronize()
        errors = []

        def calls(which):
            try:
                for k, loci in enumerate(sets):
                    if k % threads == which:
                        with torch.cuda.stream(streams[k % 2]):
                            ls.ls_run_all(ctx, loci, got[k], want_pac=False)
            except Exception as e:  # seen by the main thread
                errors.append(e)

        if threads == 1:
            calls(0)
        else:
            ts = [threading.Thread(target=calls, args=(i,)) for i in range(threads)]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        torch.cuda.synchronize()
        assert not errors
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    finally:
        ls.ls_destroy(ctx)
