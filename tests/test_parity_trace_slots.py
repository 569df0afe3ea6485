"""GPU parity of the epoch path around the candidate slots: chunks of 1,024 ops
with exactly as many ops on variables that are not stuck as there are slots (half
of a chunk in epochs of at most 2^24 ops, a quarter in longer ones), one fewer,
and one more, which rechecks the epoch whole.  Bit-exact against the oracle."""
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
