"""GPU parity of relation mode over batches of which some programs are evaluated
by variables and others, which are too long or have too many variables, token by
token beside them: the same sets and first faults as the oracle has."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu
DEEP = dict(p_if=0.12, p_while=0.08, max_depth=8, max_branch=16, max_body=24)


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def parts(*kw):
    """[(tok, payload, n_vars)] of several workloads, dealt in turn."""
    lists = []
    for k in kw:
        b = workloads.programs(**k)
        off = b["prog_tok_off"]
        lists.append([(b["tok"][off[i]:off[i + 1]], b["payload"][off[i]:off[i + 1]], int(b["prog_nvars"][i]))
                      for i in range(len(off) - 1)])
    out = []
    while any(lists):
        out += [p.pop() for p in lists if p]
    return out


def check(amc, oracle_mod, progs):
    off = np.concatenate([[0], np.cumsum([p[0].size for p in progs])]).astype(np.int64)
    a = [np.concatenate([p[0] for p in progs]), np.concatenate([p[1] for p in progs]), off,
         np.array([p[2] for p in progs], np.int32)]
    out = amc.check_batch(*[torch.from_numpy(x).cuda() for x in a])
    assert amc.sync_status() == 0
    for key, e in zip(("step_mask", "final_mask", "prog_first_fault"), oracle_mod.check_batch(*a)):
        assert np.array_equal(out[key].cpu().numpy(), e), key


@pytest.mark.parametrize("few", [1, 3])
def test_many_variables_beside(amc, oracle_mod, few):
    # 4,097 and more variables: token by token
    check(amc, oracle_mod, parts(dict(n_progs=300, seed=21, median=400.0, vars_lo=4097, vars_hi=4600, **DEEP),
                                 dict(n_progs=900, seed=22, median=300.0, vars_lo=few, vars_hi=40, **DEEP)))


def test_long_programs_beside(amc, oracle_mod):
    # more than 65,535 tokens: cut into segments
    check(amc, oracle_mod, parts(dict(n_progs=5, seed=23, median=70000.0, sigma=0.1, vars_lo=3, vars_hi=200),
                                 dict(n_progs=400, seed=24, median=700.0, vars_lo=1, vars_hi=300, **DEEP)))


@pytest.mark.parametrize("nv", [1, 2, 33])
@pytest.mark.parametrize("p_if,p_while", [(0.0, 0.0), (0.004, 0.0), (0.002, 0.002), (0.02, 0.01)])
def test_few_constructs(amc, oracle_mod, nv, p_if, p_while):
    # stretches of ops in no construct, none to several hundred ops long
    progs = parts(dict(n_progs=200, seed=25, median=900.0, vars_lo=nv, vars_hi=nv, p_if=p_if, p_while=p_while),
                  dict(n_progs=40, seed=26, median=31.0, sigma=0.2, vars_lo=nv, vars_hi=nv, p_if=0.0, p_while=0.0))
    check(amc, oracle_mod, progs)
