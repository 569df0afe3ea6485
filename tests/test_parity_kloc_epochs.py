"""GPU parity of the k-location check in epochs: the sizes around the one it
starts at (2^22 ops), few and the most variables it takes (2^20) and one more,
traces where nearly nothing and where nearly everything is kept, initial
statuses, inputs off their alignment, and bad input in an epoch.  Bit-exact
against the oracle."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu
KL_F = 0x80
N = 1 << 22


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def trace(rng, n, n_vars, k, kinds, zipf):
    kind = rng.choice(4, size=n, p=kinds)
    a = rng.integers(0, k, n)
    b = (a + rng.integers(1, k, n)) % k
    op = np.where(kind == 3, 3, np.where(kind == 2, kind | a << 2 | b << 5, kind | a << 2)).astype(np.uint8)
    var = np.searchsorted(workloads.zipf_cdf(n_vars), rng.random(n)) if zipf else rng.integers(0, n_vars, n)
    return op, np.minimum(var, n_vars - 1).astype(np.int32)


MIXED, WRITES, NOOPS = (0.4, 0.2, 0.3, 0.1), (0.0, 0.9, 0.0, 0.1), (0.0, 0.0, 0.0, 1.0)


@pytest.mark.parametrize("n, n_vars, k, kinds, zipf, init, off", [
    (N - 1, 5000, 4, MIXED, True, False, 0),
    (N, 5000, 4, MIXED, True, True, 0),
    (N + 1, 1, 3, (0.0, 0.5, 0.0, 0.5), False, False, 0),
    (N + 16_385, 33, 2, MIXED, False, True, 1),
    (N + 77, 40_000, 7, WRITES, False, True, 0),           # nothing gets stuck: every op is kept
    (N + 5, 300_000, 5, NOOPS, True, False, 3),
    ((1 << 23) + 1, 1 << 20, 4, MIXED, True, True, 0),
    ((1 << 23) + 1, (1 << 20) + 1, 4, MIXED, True, False, 0),
])
def test_epochs(amc, oracle_mod, n, n_vars, k, kinds, zipf, init, off):
    rng = np.random.default_rng(n + n_vars)
    op, var = trace(rng, n, n_vars, k, kinds, zipf)
    st = None
    if init:
        st = rng.integers(0, 1 << k, n_vars).astype(np.uint8)
        st[rng.random(n_vars) < 0.1] = KL_F
    exp = oracle_mod.check_trace_k(op, var, n_vars, k, st)
    dev = torch.device("cuda")
    o = torch.empty(n + off, dtype=torch.uint8, device=dev)[off:].copy_(torch.from_numpy(op))
    v = torch.empty(n + off, dtype=torch.int32, device=dev)[off:].copy_(torch.from_numpy(var))
    out = amc.check_trace_k(o, v, n_vars, k, None if st is None else torch.from_numpy(st).to(dev))
    assert amc.sync_status() == 0
    for key, e in zip(("step_status", "final_status", "var_first_fault"), exp[:3]):
        assert np.array_equal(out[key].cpu().numpy(), e), key
    assert int(out["first_fault"].cpu()[0]) == exp[3]


@pytest.mark.parametrize("what", ["op", "id"])
def test_bad_input_in_an_epoch(amc, what):
    rng = np.random.default_rng(5)
    op, var = trace(rng, N, 1000, 4, MIXED, True)
    if what == "op":
        op[N - 3] = 1 << 5                                 # r with a second location
    else:
        var[N - 3] = 1000
    amc.check_trace_k(torch.from_numpy(op).cuda(), torch.from_numpy(var).cuda(), 1000, 4)
    assert amc.sync_status() == (amc.E_INVALID if what == "op" else amc.E_RANGE)
    assert amc.sync_status() == 0
