"""Status words of calls of one context in flight on two streams (from one thread or two): each call's own, with
and without side-by-side directions, asynchronous and with a PAC."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ls():
    from paper_2212_11403_gb300 import ls as m
    return m


@pytest.mark.parametrize("threads,want_pac", [(1, False), (2, False), (2, True)])
@pytest.mark.parametrize("N,L", [(200, 40), (200, 300), (2003, 40)])
def test_status_words_of_calls_in_flight(ls, N, L, threads, want_pac):
    import torch
    h = (np.random.default_rng(N).random((L, 5)) < 0.5).astype(np.uint8)[:, np.arange(N) % 5]
    h[L // 2] = 0  # an allele that one target alone has: with mu = 0 every donor of it ends there
    h[L // 2, N // 3] = 1
    ctx = ls.ls_create(np.ascontiguousarray(h))
    try:
        ls.ls_set_params(ctx, np.full(L - 1, 1e-3), 0.0)
        d = [torch.empty(1, N, N, device="cuda") for _ in range(2)]
        first = torch.zeros(N, dtype=torch.int32, device="cuda")
        rc0 = ls.ls_run_all(ctx, [L // 4], d[0], status_out=first)[0]
        torch.cuda.synchronize()
        assert rc0 == ls.LS_WARN_UNDERFLOW and int(first[N // 3]) & ls.LS_STATUS_UNDERFLOW
        calls = 60
        got = torch.zeros(calls, N, dtype=torch.int32, device="cuda")
        rcs = [rc0] * calls
        streams = [torch.cuda.Stream() for _ in range(2)]
        torch.cuda.synchronize()
        errors = []

        def run(which):
            try:
                for k in range(calls):
                    if k % threads == which:
                        with torch.cuda.stream(streams[k % 2]):
                            rc = ls.ls_run_all(ctx, [L // 4], d[k % 2], want_pac=want_pac, status_out=got[k])[0]
                        if want_pac:
                            rcs[k] = rc
            except Exception as e:  # seen by the main thread
                errors.append(e)

        if threads == 1:
            run(0)
        else:
            ts = [threading.Thread(target=run, args=(i,)) for i in range(threads)]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        torch.cuda.synchronize()
        assert not errors
        assert rcs == [rc0] * calls
        assert torch.equal(got, first.expand(calls, N))
    finally:
        ls.ls_destroy(ctx)
