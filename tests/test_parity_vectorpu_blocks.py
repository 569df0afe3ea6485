"""GPU parity of the translation's blocks of 128 calls: a thread per list entry
where a block's calls fit its areas, a thread per call where they do not (calls
of more than four operands, more list entries or statements than the areas
hold), blocks of one call and ragged last blocks, lists that share arrays, and
outputs that do not start on a 16-byte boundary.  Bit-exact against the
oracle, with and without overlap inference."""
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


CASES = {
    # arrays, space, log2 lengths, calls, most operands
    "one_call": (64, 1 << 16, (8.0, 14.0), 1, 4),
    "ragged": (500, 1 << 20, (8.0, 15.0), 128 * 9 + 1, 4),
    "shared_lists": (12, 1 << 12, (8.0, 11.0), 3000, 4),         # every pair of lists has arrays in common
    "long_lists": (400, 1 << 14, (10.0, 13.0), 700, 4),          # more entries than a block copies
    "some_long": (2000, 1 << 20, (4.0, 17.0), 4000, 4),          # blocks of both kinds
    "six_operands": (300, 1 << 20, (8.0, 14.0), 2000, 6),
    "no_overlap": (50, 1 << 28, (1.0, 2.0), 1000, 4),
}


@pytest.mark.parametrize("infer", [True, False])
@pytest.mark.parametrize("case", sorted(CASES))
def test_translation(amc, oracle_mod, case, infer):
    A, space, lens, calls, most = CASES[case]
    w = workloads.vectorpu_calls(seed=83, n_arrays=A, space=space, n_calls=calls, len_log2=lens, max_opnds=most,
                                 drop_p=0.05)
    exp = oracle_mod.vectorpu(**w, infer_overlap=infer)
    dev = torch.device("cuda")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    args = [t(w[k]) for k in ("arr_start", "arr_len", "call_side", "call_off", "opnd_array", "opnd_mode")]
    n = exp["kind_side"].size
    got = amc.translate_vectorpu(*args, infer_overlap=infer)
    # the same into buffers one statement off their alignment
    out = dict(kind_side=torch.zeros(n + 8, dtype=torch.uint8, device=dev)[1:n + 1],
               var=torch.zeros(n + 8, dtype=torch.int32, device=dev)[1:n + 1],
               call_first_op=torch.empty(calls + 1, dtype=torch.int64, device=dev),
               n_dev=torch.empty(1, dtype=torch.int64, device=dev))
    off = amc.translate_vectorpu(*args, infer_overlap=infer, known_n=n, out=out)
    assert amc.sync_status() == 0
    for g in (got, off):
        assert g["n"] == n and int(g["n_dev"].cpu()[0]) == n
        assert np.array_equal(g["kind_side"].cpu().numpy(), exp["kind_side"])
        assert np.array_equal(g["var"].cpu().numpy(), exp["var"])
