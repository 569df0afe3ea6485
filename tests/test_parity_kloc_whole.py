"""GPU parity of the k-location check in epochs that are kept whole (at least
7/8 of their ops on variables that are not stuck): all of them, the share just
below and just above 7/8, ragged ends, one epoch kept whole and the next one not,
inputs off their alignment, and bad input in an epoch that is kept whole."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
KL_F = 0x80
N = 1 << 23                 # from here on in epochs: [2^21, 2^23), [2^23, ...)


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def writes(rng, n, k):
    return np.where(rng.random(n) < 0.9, 1 | rng.integers(0, k, n) << 2, 3).astype(np.uint8)


def check(amc, oracle_mod, op, var, n_vars, k, st, off=0):
    exp = oracle_mod.check_trace_k(op, var, n_vars, k, st)
    n = op.size
    o = torch.empty(n + off, dtype=torch.uint8, device="cuda")[off:].copy_(torch.from_numpy(op))
    v = torch.empty(n + off, dtype=torch.int32, device="cuda")[off:].copy_(torch.from_numpy(var))
    out = amc.check_trace_k(o, v, n_vars, k, None if st is None else torch.from_numpy(st).cuda())
    assert amc.sync_status() == 0
    for key, e in zip(("step_status", "final_status", "var_first_fault"), exp[:3]):
        assert np.array_equal(out[key].cpu().numpy(), e), key
    assert int(out["first_fault"].cpu()[0]) == exp[3]


@pytest.mark.parametrize("n, n_vars, k, stuck, off", [
    (N - 1, 77, 3, 0.0, 0),
    (N, 1, 2, 0.0, 0),
    (N + 1, 1 << 20, 7, 0.0, 0),
    (N + 511, 33_333, 4, 0.0, 1),
    (N + 513, 1000, 4, 0.11, 0),                           # kept whole
    (N + 16 * 512 + 7, 1000, 4, 0.14, 3),                  # compacted
])
def test_kept_whole(amc, oracle_mod, n, n_vars, k, stuck, off):
    # written variables never get stuck; a share of them is from the start
    rng = np.random.default_rng(n + n_vars)
    st = np.full(n_vars, 1, np.uint8)
    st[:int(stuck * n_vars)] = KL_F
    check(amc, oracle_mod, writes(rng, n, k), rng.integers(0, n_vars, n).astype(np.int32), n_vars, k, st, off)


def test_faults_in_an_epoch_kept_whole(amc, oracle_mod):
    # nothing but writes up to 2^22; then reads that get most variables stuck inside
    # the epoch that is kept whole, so that the next one is not
    rng = np.random.default_rng(8)
    n, n_vars, k = N + 100_001, 5000, 4
    op, var = writes(rng, n, k), rng.integers(0, n_vars, n).astype(np.int32)
    at = rng.integers(N // 2, N, 200_000)
    op[at] = rng.integers(0, k, at.size).astype(np.uint8) << 2
    check(amc, oracle_mod, op, var, n_vars, k, None)


@pytest.mark.parametrize("what", ["op", "id"])
def test_bad_input_kept_whole(amc, what):
    rng = np.random.default_rng(9)
    op, var = writes(rng, N, 4), rng.integers(0, 1000, N).astype(np.int32)
    if what == "op":
        op[N - 3] = 1 << 5                                 # r with a second location
    else:
        var[N - 3] = 1000
    amc.check_trace_k(torch.from_numpy(op).cuda(), torch.from_numpy(var).cuda(), 1000, 4)
    assert amc.sync_status() == (amc.E_INVALID if what == "op" else amc.E_RANGE)
    assert amc.sync_status() == 0
