"""GPU parity of the overlap lists: all pairs up to 8,192 arrays, the sort by
range start above, at counts around that limit and around a warp's 32, with
ranges that touch, nest and repeat, the last possible index and one array that
overlaps all others; the number of entries and the translation read from them,
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("A", [1, 2, 31, 32, 33, 257, 8191, 8192, 8193])
def test_lists(amc, oracle_mod, A):
    rng = np.random.default_rng(A)
    start = rng.integers(0, 8 * A, A).astype(np.int32)
    length = rng.integers(1, 17, A).astype(np.int32)
    start[A // 2], length[A // 2] = 0, 2 ** 31 - 1             # overlaps every other
    start[A - 1], length[A - 1] = 2 ** 31 - 2, 1               # ends at the last index
    if A > 2:
        start[1], length[1] = start[0], length[0]
    end = start.astype(np.int64) + length
    entries = 0
    for a in range(A):
        entries += int(((start < end[a]) & (start[a] < end)).sum()) - 1
    calls = 300
    used = [rng.choice(A, min(A, int(rng.integers(1, 4))), replace=False) for _ in range(calls)]
    w = dict(arr_start=start, arr_len=length, call_side=rng.integers(0, 2, calls).astype(np.uint8),
             call_off=np.cumsum([0] + [len(u) for u in used]).astype(np.int32),
             opnd_array=np.concatenate(used).astype(np.int32),
             opnd_mode=rng.integers(1, 4, sum(len(u) for u in used)).astype(np.uint8))
    exp = oracle_mod.vectorpu(**w, infer_overlap=True)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    args = [t(w[k]) for k in ("arr_start", "arr_len", "call_side", "call_off", "opnd_array", "opnd_mode")]
    assert int(amc.vectorpu_overlap_pairs(args[0], args[1]).item()) == entries
    got = amc.translate_vectorpu(*args, infer_overlap=True)
    assert amc.sync_status() == 0
    assert np.array_equal(got["kind_side"].cpu().numpy(), exp["kind_side"])
    assert np.array_equal(got["var"].cpu().numpy(), exp["var"])
