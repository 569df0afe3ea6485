"""GPU parity of the path-sensitive relation mode around the length from which a
program alone goes to a warp per 32 variables (1,024 tokens): one program, its
guard alone, a few and the most variables."""
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


@pytest.mark.parametrize("nv", [1, 17, 33, 256])
@pytest.mark.parametrize("n_tokens", [1023, 1024, 1025, 2048])
def test_one_program(amc, oracle_mod, nv, n_tokens):
    # of one longer program, cut between top-level statements, and Noops behind it
    b = workloads.programs_guarded(1, seed=nv, median=1400.0, sigma=0.01, vars_lo=nv, vars_hi=nv)
    tok, pay = b["tok"], b["payload"]
    kind = tok & 15
    depth = np.cumsum(np.where((kind == 8) | (kind == 10), 1, 0) - (kind == 11))
    cut = int(np.nonzero(depth[:n_tokens] == 0)[0][-1]) + 1
    more = n_tokens - cut
    tok = np.concatenate([tok[:cut], np.full(more, 4, np.uint8)])
    pay = np.concatenate([pay[:cut], np.zeros(more, np.int32)])
    a = [tok, pay, np.array([0, n_tokens], np.int64), b["prog_nvars"], b["prog_guard"]]
    out = amc.check_batch_guarded(*[torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a])
    assert amc.sync_status() == 0
    for key, e in zip(("step_mask", "final_mask", "prog_first_fault"), oracle_mod.check_batch_guarded(*a)):
        assert np.array_equal(out[key].cpu().numpy(), e), key
