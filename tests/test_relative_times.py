"""GPU tests of times relative to each other on the same device, where a rule
that chooses a path by size once took a multiple of the other path's time."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def us(f):
    """The least time of a call, after two untimed ones."""
    f()
    f()
    best = 1e9
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def batch(amc, *parts):
    """Check of the programs of several workloads as one batch."""
    bs = [workloads.programs(**p) for p in parts]
    off = np.concatenate([[0], np.cumsum(np.concatenate([np.diff(b["prog_tok_off"]) for b in bs]))]).astype(np.int64)
    a = [torch.from_numpy(np.concatenate([b["tok"] for b in bs])).cuda(),
         torch.from_numpy(np.concatenate([b["payload"] for b in bs])).cuda(), torch.from_numpy(off).cuda(),
         torch.from_numpy(np.concatenate([b["prog_nvars"] for b in bs])).cuda()]
    return us(lambda: amc.check_batch(*a))


def test_few_variables_without_constructs(amc):
    # one chain a program against 64: 7.2 times, 3.7 with stretches of ops
    flat = dict(n_progs=64, seed=31, median=40000.0, sigma=0.1, p_if=0.0, p_while=0.0)
    one, many = batch(amc, dict(flat, vars_lo=1, vars_hi=1)), batch(amc, dict(flat, vars_lo=64, vars_hi=64))
    assert one < 5.5 * many, (one, many)


def test_both_kinds_at_the_same_time(amc):
    # programs evaluated by variables and programs left token by token: the sum of
    # their times, one after the other
    short = dict(n_progs=40, seed=32, median=40000.0, sigma=0.05, vars_lo=4, vars_hi=4)
    long = dict(n_progs=40, seed=33, median=4000.0, sigma=0.05, vars_lo=4097, vars_hi=4200)
    a, b, both = batch(amc, short), batch(amc, long), batch(amc, short, long)
    assert both < 0.93 * (a + b), (a, b, both)


def test_writes_to_few_variables(amc):
    # 5 M writes over 100 variables against 4 M: 2.2 times in epochs, 1.2 sorted whole
    def k(n):
        rng = np.random.default_rng(n)
        op = torch.ones(n, dtype=torch.uint8, device="cuda")
        var = torch.from_numpy(rng.integers(0, 100, n).astype(np.int32)).cuda()
        return us(lambda: amc.check_trace_k(op, var, 100, 3))

    few, more = k(4_000_000), k(5_000_000)
    assert more < 1.7 * few, (few, more)
