"""GPU test of host threads that check traces over different numbers of
variables at the same time, each on a stream of its own: kernels whose shared
memory grows with the variables start in every thread, and each gets the
results it gets alone."""
import threading
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def trace_k(amc, n_vars):
    rng = np.random.default_rng(n_vars)
    n = (1 << 22) + 5
    op = torch.from_numpy(rng.choice(np.array([0, 1, 3, 4 | 0, 4 | 1], np.uint8), n)).cuda()
    var = torch.from_numpy(rng.integers(0, n_vars, n).astype(np.int32)).cuda()
    ws = torch.empty(int(amc.lib().amc_check_trace_k_workspace(n, n_vars)) + 256, dtype=torch.uint8, device="cuda")
    return lambda: amc.check_trace_k(op, var, n_vars, 2, workspace=ws[(-ws.data_ptr()) % 256:])


def guarded(amc, n_vars):
    rng = np.random.default_rng(n_vars)
    n = 300_000
    ks = torch.from_numpy((rng.choice(np.array([0, 1, 4], np.uint8), n) | rng.integers(0, 2, n).astype(np.uint8) << 4)).cuda()
    var = torch.from_numpy(rng.integers(0, n_vars, n).astype(np.int32)).cuda()
    ws = torch.empty(int(amc.lib().amc_check_guarded_trace_workspace(n, n_vars)) + 256, dtype=torch.uint8, device="cuda")
    return lambda: amc.check_trace(ks, var, n_vars, guarded=True, workspace=ws[(-ws.data_ptr()) % 256:])


def epochs(amc, n_vars):
    rng = np.random.default_rng(n_vars)
    n = (1 << 22) + 5
    ks = torch.from_numpy((rng.integers(0, 5, n).astype(np.uint8) | rng.integers(0, 2, n).astype(np.uint8) << 4)).cuda()
    var = torch.from_numpy(rng.integers(0, n_vars, n).astype(np.int32)).cuda()
    ws = torch.empty(int(amc.lib().amc_check_trace_workspace(n, n_vars)) + 256, dtype=torch.uint8, device="cuda")
    return lambda: amc.check_trace(ks, var, n_vars, workspace=ws[(-ws.data_ptr()) % 256:])


@pytest.mark.parametrize("make,few,many", [(trace_k, 1000, 300_000), (guarded, 9000, 60_000), (epochs, 20_000, 1 << 20)])
def test_two_threads(amc, monkeypatch, make, few, many):
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")                     # the reduce / carry / apply path
    monkeypatch.setenv("AMC_TRACE_GRAPH", "0")                           # no replay: every call launches
    calls = [make(amc, few), make(amc, many)]
    want = [{k: v.clone() for k, v in c().items()} for c in calls]       # alone, and the size class tuned
    torch.cuda.synchronize()
    assert amc.sync_status() == 0
    bad, go = [], threading.Barrier(2)

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            try:
                go.wait()
                end = time.monotonic() + 2.0
                while time.monotonic() < end and not bad:
                    for _ in range(8):
                        got = calls[i]()
                    s.synchronize()
                bad.extend((i, k) for k in got if not torch.equal(got[k], want[i][k]))
            except Exception as e:  # noqa: BLE001
                bad.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
    assert amc.sync_status() == 0
