"""GPU parity of the one-CTA trace check: stretches of no, one, a whole and a
ragged batch of 32 ops, of as many as stay in registers (128 ops a warp: 4,096 in
all) and one more, up to its longest; variable counts around the id's bits, the
carry's two forms (128 variables) and the most; batches of one variable; initial
statuses; bad input.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1024, 1025, 4095, 4096, 4097, 8192, 65_535, 65_536])
@pytest.mark.parametrize("n_vars", [1, 2, 3, 16, 17, 127, 128, 129, 2047, 2048])
def test_small(amc, oracle_mod, monkeypatch, n, n_vars):
    monkeypatch.setenv("AMC_TRACE_CANDIDATE", "0")               # the path by size
    rng = np.random.default_rng(n * 4096 + n_vars)
    ks = rng.choice(np.array([0, 1, 2, 3, 4, 5, 16, 17, 18, 19, 20, 21], np.uint8), n,
                    p=[.02, .3, .05, .05, .1, .05, .02, .16, .05, .05, .1, .05])
    var = rng.integers(0, n_vars, n).astype(np.int32)
    var[n // 3:n // 2] = n_vars - 1                              # one variable for a while
    init = rng.integers(0, 5, n_vars).astype(np.uint8) if n % 2 else None
    assert amc.trace_plan(n, n_vars, init is not None)[0] == "small"
    exp = oracle_mod.check_trace(ks, var, n_vars, init)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    out = amc.check_trace(t(ks), t(var), n_vars, None if init is None else t(init))
    assert amc.sync_status() == 0
    assert np.array_equal(out["step_status"].cpu().numpy(), exp[0])
    assert np.array_equal(out["final_status"].cpu().numpy(), exp[1])
    assert np.array_equal(out["var_first_fault"].cpu().numpy(), exp[2])
    assert int(out["first_fault"].cpu()[0]) == exp[3]


@pytest.mark.parametrize("n", [100, 5000])
@pytest.mark.parametrize("bad,code", [(("var", 16), "E_RANGE"), (("var", -1), "E_RANGE"), (("ks", 6), "E_INVALID"),
                                      (("ks", 0x21), "E_INVALID")])
def test_bad_input(amc, n, bad, code):
    ks = torch.zeros(n, dtype=torch.uint8, device="cuda")
    var = torch.zeros(n, dtype=torch.int32, device="cuda")
    (var if bad[0] == "var" else ks)[n - 2] = bad[1]
    assert amc.sync_status() == 0
    amc.check_trace(ks, var, 16)
    assert amc.sync_status() == getattr(amc, code)
    assert amc.sync_status() == 0
