"""GPU parity of the owner-sorted trace check where a few owners have most of the
tiles' ops, whose ops are then walked in pieces: lists around the length from
which on, one and several such owners, all ops on one, owners of one and of many
variables, guarded traces with their GT / EN pairs across pieces and tiles,
malformed guards; and that such a trace takes no multiple of an even one's time.
Bit-exact against the oracle."""
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


def same(out, step, final, vff, ff):
    assert np.array_equal(out["step_status"].cpu().numpy(), step)
    assert np.array_equal(out["final_status"].cpu().numpy(), final)
    assert np.array_equal(out["var_first_fault"].cpu().numpy(), vff)
    assert int(out["first_fault"].cpu()[0]) == ff


def check(amc, oracle_mod, ks, var, n_vars, init=None):
    t = lambda a: None if a is None else torch.from_numpy(a).cuda()  # noqa: E731
    out = amc.check_trace(t(ks), t(var), n_vars, t(init))
    assert amc.sync_status() == 0
    same(out, *oracle_mod.check_trace(ks, var, n_vars, init))


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("n, n_vars, hot, share", [
    (5000, 1, 1, 1.0), (70_003, 2, 2, 1.0), (4096, 31, 31, 1.0), (70_001, 4096, 1, 0.9), (70_001, 8192, 8, 0.9),
    (70_001, 8192, 40, 1.0), (EDGE + 5, 8192, 16, 0.8), (EDGE + 1, 300, 3, 0.5), (EDGE + 77, 65_536, 1, 0.95),
    (300_001, 65_536, 20, 0.7)])
def test_hot_variables(amc, oracle_mod, monkeypatch, n, n_vars, hot, share, wide):
    monkeypatch.setenv("AMC_TRACE_CANDIDATE", "4")            # the reduce / carry / apply path at any size
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    rng = np.random.default_rng(n + n_vars + hot)
    ks, var = workloads.trace_random(rng, n, n_vars, p=[0.03, 0.5, 0.1, 0.1, 0.27])
    ids = rng.choice(n_vars, size=hot, replace=False).astype(np.int32)
    at = rng.random(n) < share
    var[at] = ids[rng.integers(0, hot, int(at.sum()))]
    check(amc, oracle_mod, ks, var, n_vars, rng.integers(0, 5, n_vars).astype(np.uint8))


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("more", [-1, 0, 1, 2, 32, 33])
@pytest.mark.parametrize("n_vars", [128, 5000])
def test_list_lengths(amc, oracle_mod, monkeypatch, more, n_vars, wide):
    # the variables of one owner have `length` ops in the tile, the others few; lists
    # of more than 256 and 4 for each of an owner's bytes are walked in pieces
    monkeypatch.setenv("AMC_TRACE_CANDIDATE", "4")
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    no = 256 if wide == "1" else 128
    length = 256 + 4 * (-(-n_vars // (4 * no)) * 4) + more
    rng = np.random.default_rng(length)
    v = np.arange(n_vars)
    owner = (v + 37 * (v // no)) % no
    mine, others = v[owner == 5], v[owner != 5]
    n = 1000
    ks, _ = workloads.trace_random(rng, n, n_vars, p=[0.03, 0.5, 0.1, 0.1, 0.27])
    var = others[np.arange(n) % others.size].astype(np.int32)
    var[rng.choice(n, size=length, replace=False)] = mine[rng.integers(0, mine.size, length)]
    check(amc, oracle_mod, ks, var, n_vars)


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("n_arrays, n_calls, hot, share", [(1, 60_000, 1, 1.0), (40, 60_000, 1, 0.9), (4000, 60_000, 3, 0.9),
                                                           (4000, 1_300_000, 2, 0.8), (30_000, 60_000, 1, 0.9)])
def test_guarded(amc, oracle_mod, monkeypatch, n_arrays, n_calls, hot, share, wide):
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    rng = np.random.default_rng(n_arrays + hot)
    w = workloads.vectorpu_calls(seed=72, n_arrays=n_arrays, space=n_arrays << 10, n_calls=n_calls, len_log2=(2.0, 9.0),
                                 max_opnds=1, drop_p=0.01)
    at = rng.random(n_calls) < share
    w["opnd_array"][at] = rng.choice(n_arrays, size=hot, replace=False)[rng.integers(0, hot, int(at.sum()))]
    exp = oracle_mod.vectorpu(**w)
    out = amc.check_trace(torch.from_numpy(exp["kind_side"]).cuda(), torch.from_numpy(exp["var"]).cuda(), 2 * n_arrays,
                          guarded=True)
    assert amc.sync_status() == 0
    same(out, exp["step_status"], exp["final_status"], exp["var_first_fault"], exp["first_fault"])


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("at", [3, 150, 1023, 4095, 6000])
@pytest.mark.parametrize("pair", [[(6, 1), (0, 2)], [(6, 1), (7 | 16, 2)], [(6, 1), (7, 1)], [(6, 2), (7, 2)]])
def test_malformed_guards(amc, monkeypatch, pair, at, wide):
    # every op before and after on variables 1 and 2, so that the GT and what
    # follows it lie in lists that are walked in pieces
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")
    monkeypatch.setenv("AMC_SCAN_DENSE_SORT", wide)
    n = 9000
    ks = np.full(n, 1, np.uint8)
    var = (1 + np.arange(n) % 2).astype(np.int32)
    for k, (b, v) in enumerate(pair):
        ks[at + k], var[at + k] = b, v
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    amc.check_trace(t(ks), t(var), 300, guarded=True)
    assert amc.sync_status() == amc.E_INVALID
    ks[at], var[at], ks[at + 1], var[at + 1] = 6, 1, 7, 2       # a pair: the trace is fine
    amc.check_trace(t(ks), t(var), 300, guarded=True)
    assert amc.sync_status() == 0


def test_time_of_a_hot_array(amc, monkeypatch):
    # 9 of 10 transfers on one array of 1,000: 10 times as long as spread evenly when
    # its owner's thread walked them alone
    monkeypatch.setenv("AMC_GUARDED_CANDIDATE", "1")
    A, m = 1000, 2_000_000
    rng = np.random.default_rng(3)

    def us(x):
        side = (rng.integers(0, 2, m) << 4).astype(np.uint8)
        ks = torch.from_numpy(np.stack([6 | side, 7 | side, 1 | side, 1 | side], 1).reshape(-1).astype(np.uint8)).cuda()
        var = torch.from_numpy(np.stack([x, A + x, A + x, x], 1).reshape(-1).astype(np.int32)).cuda()
        amc.check_trace(ks, var, 2 * A, guarded=True)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            amc.check_trace(ks, var, 2 * A, guarded=True)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        return best

    x = rng.integers(0, A, m)
    even, hot = us(x), us(np.where(rng.random(m) < 0.9, 0, x))
    assert hot < 4 * even, (even, hot)
