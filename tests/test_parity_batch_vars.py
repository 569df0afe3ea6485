"""GPU parity of the relation mode variable by variable: few variables (long
chains, nearly every op sharing its construct with another), deep nesting, more
constructs than shared memory holds, programs around the longest and the widest
that are evaluated this way (65,535 tokens, 4,096 variables) next to ones that
are not, all six op kinds, and malformed programs at window ends.  Bit-exact
against the oracle."""
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


def run(amc, tok, payload, off, nv):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    out = amc.check_batch(t(tok), t(payload), t(off), t(nv))
    return out, amc.sync_status()


def check(amc, oracle_mod, tok, payload, off, nv):
    step, final, pff = oracle_mod.check_batch(tok, payload, off, nv)
    out, rc = run(amc, tok, payload, off, nv)
    assert rc == 0
    assert np.array_equal(out["step_mask"].cpu().numpy(), step)
    assert np.array_equal(out["final_mask"].cpu().numpy(), final)
    assert np.array_equal(out["prog_first_fault"].cpu().numpy(), pff)


CASES = {
    "few_variables": dict(n_progs=300, vars_lo=1, vars_hi=4, median=400.0, p_if=0.1, p_while=0.08),
    "forty_variables": dict(n_progs=300, vars_lo=20, vars_hi=60, median=1500.0),
    "deep": dict(n_progs=200, vars_lo=8, vars_hi=200, median=900.0, p_if=0.15, p_while=0.1, max_depth=8),
    "many_constructs": dict(n_progs=20, vars_lo=100, vars_hi=4096, median=9000.0, p_if=0.3, p_while=0.1, max_branch=6,
                            max_body=6),
    "straight": dict(n_progs=64, vars_lo=1, vars_hi=4096, median=700.0, p_if=0.0, p_while=0.0),
    "tiny": dict(n_progs=2000, vars_lo=1, vars_hi=3, median=3.0, p_if=0.3, p_while=0.3, max_branch=2, max_body=2),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_programs(amc, oracle_mod, case):
    b = workloads.programs(seed=91, **CASES[case])
    tok = b["tok"].copy()
    rng = np.random.default_rng(92)
    ops = np.nonzero((tok & 15) <= 4)[0]
    pw = ops[rng.random(ops.size) < 0.1]
    tok[pw] = (tok[pw] & 0x10) | 5                             # partial writes among them
    check(amc, oracle_mod, tok, b["payload"], b["prog_tok_off"], b["prog_nvars"])


def test_around_the_limits(amc, oracle_mod):
    # lengths of 65,534 to 65,537 tokens and 4,095 to 4,097 variables, a While
    # over the second half of each, one batch
    rng = np.random.default_rng(93)
    toks, pays, lens, nvs = [], [], [], []
    for n in (65_534, 65_535, 65_536, 65_537, 100):
        for nv in (4095, 4096, 4097):
            t = (rng.choice(6, n, p=[0.3, 0.3, 0.1, 0.1, 0.15, 0.05]) | rng.integers(0, 2, n) << 4).astype(np.uint8)
            p = rng.integers(0, nv, n).astype(np.int32)
            a = n // 2
            t[a], p[a] = 10, n - 2 - a
            t[n - 1], p[n - 1] = 11, 0
            toks.append(t), pays.append(p), lens.append(n), nvs.append(nv)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    check(amc, oracle_mod, np.concatenate(toks), np.concatenate(pays), off, np.array(nvs, np.int32))


IF, ELSE, WHILE, END = 8, 9, 10, 11
MALFORMED = {  # (token, payload) pairs
    "end_first": [(END, 0), (0, 0)],
    "else_alone": [(0, 0), (ELSE, 0), (END, 0)],
    "if_without_else": [(IF, 1), (0, 0), (END, 0)],
    "else_in_while": [(WHILE, 2), (0, 0), (ELSE, 0), (END, 0)],
    "short_while": [(WHILE, 1), (0, 0), (0, 0), (END, 0)],
    "long_while": [(WHILE, 9), (0, 0), (END, 0)],
    "negative": [(WHILE, -1), (END, 0)],
    "crossing": [(WHILE, 3), (WHILE, 3), (0, 0), (0, 0), (END, 0), (END, 0)],
    "open": [(WHILE, 1), (0, 0)],
    "side_on_end": [(WHILE, 1), (0, 0), (END | 16, 0)],
    "unknown": [(12, 0)],
    "guarded_transfer": [(6, 0)],
    "nine_deep": [(WHILE, 16 - 2 * i) for i in range(9)] + [(END, 0)] * 9,
}


@pytest.mark.parametrize("at", [0, 29, 62])
@pytest.mark.parametrize("case", sorted(MALFORMED))
def test_malformed(amc, case, at):
    bad = MALFORMED[case]
    tok = np.array([0] * at + [b & 0xFF for b, _ in bad], np.uint8)
    pay = np.array([0] * at + [v for _, v in bad], np.int32)
    _, rc = run(amc, tok, pay, np.array([0, tok.size], np.int64), np.array([4], np.int32))
    assert rc == amc.E_INVALID
    # a well-formed program of the same ops is accepted
    _, rc = run(amc, np.zeros(at + 1, np.uint8), np.zeros(at + 1, np.int32), np.array([0, at + 1], np.int64),
                np.array([4], np.int32))
    assert rc == 0


def test_id_out_of_range(amc):
    tok, pay = np.zeros(100, np.uint8), np.zeros(100, np.int32)
    pay[70] = 4
    _, rc = run(amc, tok, pay, np.array([0, 100], np.int64), np.array([4], np.int32))
    assert rc == amc.E_RANGE
