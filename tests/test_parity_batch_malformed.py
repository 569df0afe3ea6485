"""GPU parity of relation mode over batches that hold malformed programs: the
batch is refused, and the well-formed programs between the malformed ones still
get their sets, bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

NOOP, IF, ELSE, WHILE, END = 4, 8, 9, 10, 11
DEEP = dict(vars_lo=1, vars_hi=9, median=60.0, p_if=0.3, p_while=0.2, max_depth=8, max_branch=6, max_body=6)


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def programs(n, seed):
    """[(tok, payload, n_vars)] of n well-formed programs full of constructs."""
    b = workloads.programs(n, seed=seed, **DEEP)
    off = b["prog_tok_off"]
    return [(b["tok"][off[i]:off[i + 1]], b["payload"][off[i]:off[i + 1]], int(b["prog_nvars"][i])) for i in range(n)]


def run(amc, tok, payload, off, nv):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    out = amc.check_batch(t(tok), t(payload), t(off), t(nv))
    return {k: v.cpu().numpy() for k, v in out.items()}, amc.sync_status()


def offsets(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


def check_among(amc, oracle_mod, progs, good):
    """The batch of progs is refused; the programs with good[i] as the oracle has them."""
    off, voff = offsets([p[0].size for p in progs]), offsets([p[2] for p in progs])
    out, rc = run(amc, np.concatenate([p[0] for p in progs]), np.concatenate([p[1] for p in progs]), off,
                  np.array([p[2] for p in progs], np.int32))
    assert rc == amc.E_INVALID
    keep = [p for p, g in zip(progs, good) if g]
    step, final, pff = oracle_mod.check_batch(np.concatenate([p[0] for p in keep]), np.concatenate([p[1] for p in keep]),
                                              offsets([p[0].size for p in keep]), np.array([p[2] for p in keep], np.int32))
    cut = lambda a, o: np.concatenate([a[o[i]:o[i + 1]] for i in range(len(progs)) if good[i]])  # noqa: E731
    assert np.array_equal(cut(out["step_mask"], off), step)
    assert np.array_equal(cut(out["final_mask"], voff), final)
    assert np.array_equal(out["prog_first_fault"][np.array(good)], pff)


@pytest.mark.parametrize("opener", [IF, WHILE])
@pytest.mark.parametrize("n_open,n_ops", [(1, 1), (2, 1), (8, 1), (8, 2), (7, 23), (8, 56)])
def test_open_constructs(amc, oracle_mod, opener, n_open, n_ops):
    # constructs that are never closed, more of them than pairs of tokens, before
    # and after programs that are well-formed, at odd and even tokens
    tok = np.array([opener] * n_open + [NOOP] * n_ops, np.uint8)
    pay = np.array([0] * n_open + [0] * n_ops, np.int32)
    progs, good = [], []
    for i, p in enumerate(programs(1500, seed=94)):
        progs += [(tok, pay, 1), p] + ([(tok[:0], pay[:0], 1)] if i % 3 else [(tok[-1:], pay[-1:], 1)])
        good += [False, True, True]
    check_among(amc, oracle_mod, progs, good)


@pytest.mark.parametrize("n_tokens_more", [0, 70_000])
def test_common_tokens(amc, oracle_mod, n_tokens_more):
    # offsets that go back, so that two programs have tokens in common, offsets
    # before the first and behind the last token: refused, and the programs that
    # share nothing as the oracle has them
    good = programs(40, seed=95)
    tok, pay = np.concatenate([p[0] for p in good]), np.concatenate([p[1] for p in good])
    a = offsets([p[0].size for p in good])
    n = int(a[-1])
    more = np.full(200 + n_tokens_more, NOOP, np.uint8)
    tok, pay = np.concatenate([tok, more]), np.concatenate([pay, np.zeros(more.size, np.int32)])
    back = [n + 100, n + 50, n + 150, -5, n + 150, 1 << 40, n, tok.size]
    off = np.concatenate([a, np.array(back, np.int64)])
    nv = np.array([p[2] for p in good] + [1] * len(back), np.int32)
    out, rc = run(amc, tok, pay, off, nv)
    assert rc == amc.E_INVALID
    step, final, pff = oracle_mod.check_batch(tok[:n], pay[:n], a, nv[:40])
    assert np.array_equal(out["step_mask"][:n], step)
    assert np.array_equal(out["final_mask"][:int(nv[:40].sum())], final)
    assert np.array_equal(out["prog_first_fault"][:40], pff)
