"""GPU parity of the path-sensitive relation mode for programs of at most 256
variables: one warp with four variables a lane at a time, or, for the programs
that are long against the rest of the batch, one warp per 32 variables.
Variable counts around a lane's four, a warp's 32 and the limit; nesting below
the levels kept in shared memory; all six op kinds; many ops on the guard, loops
that run again, ops on one variable side by side; malformed programs of both
kinds.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu
IF, ELSE, WHILE, END = 8, 9, 10, 11


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def run(amc, b):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    out = amc.check_batch_guarded(t(b["tok"]), t(b["payload"]), t(b["prog_tok_off"]), t(b["prog_nvars"]),
                                  t(b["prog_guard"]))
    return out, amc.sync_status()


def check(amc, oracle_mod, b):
    step, final, pff = oracle_mod.check_batch_guarded(b["tok"], b["payload"], b["prog_tok_off"], b["prog_nvars"],
                                                      b["prog_guard"])
    out, rc = run(amc, b)
    assert rc == 0
    assert np.array_equal(out["step_mask"].cpu().numpy(), step)
    assert np.array_equal(out["final_mask"].cpu().numpy(), final)
    assert np.array_equal(out["prog_first_fault"].cpu().numpy(), pff)


@pytest.mark.parametrize("nv", [1, 2, 3, 4, 5, 31, 32, 33, 64, 127, 128, 129, 255, 256, 257])
@pytest.mark.parametrize("median", [150.0, 4000.0])           # below and above the shortest shared length
def test_variable_counts(amc, oracle_mod, nv, median):
    b = workloads.programs_guarded(n_progs=24, seed=100 + nv, median=median, vars_lo=nv, vars_hi=nv, p_if=0.08,
                                   p_while=0.06, max_depth=8, max_branch=20, max_body=30)
    rng = np.random.default_rng(nv)
    tok = b["tok"]
    ops = np.nonzero((tok & 15) <= 4)[0]
    pw = ops[rng.random(ops.size) < 0.1]
    tok[pw] = (tok[pw] & 0x10) | 5
    prog = np.repeat(np.arange(24), np.diff(b["prog_tok_off"]))
    on_g = ops[rng.random(ops.size) < 0.05]
    b["payload"][on_g] = np.maximum(b["prog_guard"][prog[on_g]], 0)
    check(amc, oracle_mod, b)


def test_shared_with_short(amc, oracle_mod):
    """Long programs in a batch of short ones, with and without a guard."""
    b = [workloads.programs_guarded(n_progs=n, seed=s, median=m, vars_lo=16, vars_hi=300)
         for n, s, m in ((2000, 131, 60.0), (6, 132, 20000.0), (2000, 133, 90.0))]
    check(amc, oracle_mod, dict(
        tok=np.concatenate([x["tok"] for x in b]), payload=np.concatenate([x["payload"] for x in b]),
        prog_tok_off=np.concatenate([[0], np.cumsum(np.concatenate([np.diff(x["prog_tok_off"]) for x in b]))]),
        prog_nvars=np.concatenate([x["prog_nvars"] for x in b]),
        prog_guard=np.concatenate([x["prog_guard"] for x in b])))


@pytest.mark.parametrize("before", [0, 31, 5000])
@pytest.mark.parametrize("case,code", [("range", "E_RANGE"), ("else", "E_INVALID"), ("end", "E_INVALID"),
                                       ("open", "E_INVALID"), ("token", "E_INVALID"), ("deep", "E_INVALID")])
def test_malformed(amc, before, case, code):
    tail = {"range": ([4, 4], [40, 0]), "else": ([IF, 4, ELSE, END, END], [1, 0, 1, 0, 0]),
            "end": ([WHILE, 4, END, 4], [2, 0, 0, 0]), "open": ([WHILE, 4], [1, 0]), "token": ([6, 4], [0, 0]),
            "deep": ([WHILE] * 9 + [END] * 9, list(range(16, -2, -2)) + [0] * 9)}[case]
    n = before + len(tail[0])
    b = dict(tok=np.array([4] * before + tail[0], np.uint8), payload=np.array([0] * before + tail[1], np.int32),
             prog_tok_off=np.array([0, n]), prog_nvars=np.array([40], np.int32), prog_guard=np.array([0], np.int32))
    assert amc.sync_status() == 0
    assert run(amc, b)[1] == getattr(amc, code)
    assert amc.sync_status() == 0
