"""GPU parity of the epoch path around the candidate slots: chunks of 1,024 ops
with exactly as many ops on variables that are not stuck as there are slots (half
of a chunk in epochs of at most 2^24 ops, a quarter in longer ones), one fewer,
and one more, which rechecks the epoch whole; arrays that start off the filter's
vector alignment.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
STUCK, ALIVE = 4096, 30_000


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("epoch,per_chunk", [
    (1 << 16, 256), (1 << 16, 257), (1 << 16, 511), (1 << 16, 512), (1 << 16, 513),
    (1 << 24, 512), ((1 << 24) + 1024, 256), ((1 << 24) + 1024, 257),
])
def test_slots(amc, oracle_mod, monkeypatch, epoch, per_chunk):
    first = 4096
    monkeypatch.setenv("AMC_SCAN_TAIL", f"12,{max(16, (epoch - 1).bit_length())}")
    rng = np.random.default_rng(per_chunk)
    n = first + epoch
    ks = rng.choice(np.array([0, 1, 2, 3, 4, 16, 17, 18, 19, 20], np.uint8), n)
    var = rng.integers(0, STUCK, n).astype(np.int32)
    ks[:first] = 16                                    # reads where nothing is valid: variables 0 to 4,095 are stuck
    var[:first] = np.arange(first)
    live = np.zeros((epoch // 1024, 1024), bool)
    live[:, :per_chunk - 1] = True
    live[epoch // 2048, :per_chunk] = True             # the most in one chunk in the middle
    live = np.concatenate([np.zeros(first, bool), live.ravel()])
    ks[live] = np.where(rng.random(int(live.sum())) < 0.999, 1, ks[live])      # CPU writes, a few others
    var[live] = STUCK + rng.integers(0, ALIVE, int(live.sum()))
    exp = oracle_mod.check_trace(ks, var, STUCK + ALIVE, None)
    out = amc.check_trace(torch.from_numpy(ks).cuda(), torch.from_numpy(var).cuda(), STUCK + ALIVE)
    assert amc.sync_status() == 0
    assert np.array_equal(out["step_status"].cpu().numpy(), exp[0])
    assert np.array_equal(out["final_status"].cpu().numpy(), exp[1])
    assert np.array_equal(out["var_first_fault"].cpu().numpy(), exp[2])
    assert int(out["first_fault"].cpu()[0]) == exp[3]


@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (4, 4, 4), (3, 2, 1)])
def test_alignment(amc, oracle_mod, monkeypatch, shift):
    """kind_side, var and step_status so many elements off a 256-byte boundary."""
    monkeypatch.setenv("AMC_SCAN_TAIL", "13,-1")
    rng = np.random.default_rng(5)
    n, nv = 100_003, 20_000
    ks = rng.choice(np.array([0, 1, 2, 3, 4, 5, 16, 17, 18, 19, 20, 21], np.uint8), n)
    var = (nv * rng.random(n) ** 3).astype(np.int32)
    exp = oracle_mod.check_trace(ks, var, nv, None)
    d_ks = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")[shift[0]:shift[0] + n]
    d_var = torch.zeros(n + 8, dtype=torch.int32, device="cuda")[shift[1]:shift[1] + n]
    d_ks.copy_(torch.from_numpy(ks))
    d_var.copy_(torch.from_numpy(var))
    out = dict(step_status=torch.empty(n + 8, dtype=torch.uint8, device="cuda")[shift[2]:shift[2] + n],
               final_status=torch.empty(nv, dtype=torch.uint8, device="cuda"),
               var_first_fault=torch.empty(nv, dtype=torch.int32, device="cuda"),
               first_fault=torch.empty(1, dtype=torch.int64, device="cuda"))
    amc.check_trace(d_ks, d_var, nv, out=out)
    assert amc.sync_status() == 0
    assert np.array_equal(out["step_status"].cpu().numpy(), exp[0])
    assert np.array_equal(out["final_status"].cpu().numpy(), exp[1])
    assert np.array_equal(out["var_first_fault"].cpu().numpy(), exp[2])
    assert int(out["first_fault"].cpu()[0]) == exp[3]


@pytest.mark.parametrize("mix", [[0.002, 0.6, 0.1, 0.1, 0.198], [0.2, 0.4, 0.15, 0.15, 0.1]])
def test_statuses_in_place(amc, oracle_mod, monkeypatch, mix):
    """Requests of a session whose statuses are read and written in one buffer:
    variables with runs over several sort tiles of the first part."""
    import test_serve
    import workloads

    monkeypatch.setenv("AMC_SCAN_TAIL", "16,-1")
    rng = np.random.default_rng(17)
    nv = 20_000
    reqs = []
    for n in (200_003, 70_001, 150_000):
        ks, var = workloads.trace_random(rng, n, nv, p=mix)
        var[rng.random(n) < 0.3] = 11                  # a run of a third of the ops
        reqs.append((0, ks, var))
    sessions = [(0, nv, reqs)]
    exp, fin = test_serve.oracle_results(oracle_mod, sessions)
    got, got_fin = test_serve.run_server(amc, sessions, 2, True)
    for k, (step, ff, _) in exp.items():
        assert got[k]["error"] == 0
        assert np.array_equal(got[k]["status"], step), k
        assert got[k]["first_fault"] == ff, k
    assert np.array_equal(got_fin[0], fin[0])
