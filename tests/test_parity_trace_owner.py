"""GPU parity of the owner-sorted reduce / carry / apply kernels at the sizes
where they can go wrong: one op, a tile and one op around it, the size where
the tiles grow from 1,024 to 4,096 ops, one variable, variable counts around
the owner counts (128 and 256) and the limits of the two variants (8,192 and
65,536), statuses shared between the input and the output, and guarded traces
whose GT / EN pairs lie across tile ends.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

EDGE = 152 * 6 * 4096          # from here tiles of 4,096 ops


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def run(amc, ks, var, n_vars, init=None, guarded=False):
    dev = torch.device("cuda")
    out = amc.check_trace(torch.from_numpy(ks).to(dev), torch.from_numpy(var).to(dev), n_vars,
                          None if init is None else torch.from_numpy(init).to(dev), guarded=guarded)
    return out, amc.sync_status()


def same(out, step, final, vff, ff):
    assert np.array_equal(out["step_status"].cpu().numpy(), step)
    assert np.array_equal(out["final_status"].cpu().numpy(), final)
    assert np.array_equal(out["var_first_fault"].cpu().numpy(), vff)
    assert int(out["first_fault"].cpu()[0]) == ff


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("n, n_vars", [(1, 3000), (1023, 1), (1024, 127), (1025, 128), (4095, 2500), (4097, 257),
                                       (70_000, 8192), (70_001, 8193), (70_000, 65_536), (EDGE - 1, 511),
                                       (EDGE, 512), (EDGE + 1, 2049)])
def test_sizes(amc, oracle_mod, monkeypatch, n, n_vars, wide):
    monkeypatch.setenv("AMC_TRACE_CANDIDATE", "4")            # the reduce / carry / apply path at any size
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    rng = np.random.default_rng(n + n_vars)
    ks, var = workloads.trace_random(rng, n, n_vars, p=[0.03, 0.5, 0.1, 0.1, 0.27])
    var[-1] = n_vars - 1
    init = rng.integers(0, 5, n_vars).astype(np.uint8)
    out, rc = run(amc, ks, var, n_vars, init)
    assert rc == 0
    same(out, *oracle_mod.check_trace(ks, var, n_vars, init))


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("n_arrays, n_calls", [(3, 700), (300, 40_000), (4096, 120_000), (6000, 30_000)])
def test_guarded(amc, oracle_mod, monkeypatch, n_arrays, n_calls, wide):
    # about a third of the statements are GTs, so tiles end between a GT and
    # its EN; 120,000 calls translate to more than EDGE statements
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    w = workloads.vectorpu_calls(seed=71, n_arrays=n_arrays, space=n_arrays << 12, n_calls=n_calls, drop_p=0.01)
    exp = oracle_mod.vectorpu(**w)
    tile = 4096 if wide == "1" or exp["var"].size >= EDGE else 1024
    if n_calls > 1000:
        assert ((exp["kind_side"][tile - 1::tile] & 15) == 6).any()
    out, rc = run(amc, exp["kind_side"], exp["var"], 2 * w["arr_start"].size, guarded=True)
    assert rc == 0
    same(out, exp["step_status"], exp["final_status"], exp["var_first_fault"], exp["first_fault"])


# (op byte, variable) pairs put at a position: each is malformed
GT, EN = 6, 7
BAD_PAIRS = {
    "no_en": [(GT, 1), (0, 2)],
    "other_side": [(GT, 1), (EN | 16, 2)],
    "own_variable": [(GT, 1), (EN, 1)],
    "last_op": [(GT, 1)],
}


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("at", [10, 1023, 4095])
@pytest.mark.parametrize("pair", sorted(BAD_PAIRS))
def test_malformed_guards(amc, monkeypatch, pair, at, wide):
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    n = at + 1 if pair == "last_op" else 9000
    ks = np.full(n, 1, np.uint8)
    var = (np.arange(n) % 300).astype(np.int32)
    for k, (b, v) in enumerate(BAD_PAIRS[pair]):
        ks[at + k], var[at + k] = b, v
    _, rc = run(amc, ks, var, 300, guarded=True)
    assert rc == amc.E_INVALID
    ks[at] = 1                                                # without the GT the trace is fine
    if pair != "last_op":
        ks[at + 1] = 0 if (ks[at + 1] & 15) != EN else ks[at + 1]
    _, rc = run(amc, ks, var, 300, guarded=True)
    assert rc == 0
