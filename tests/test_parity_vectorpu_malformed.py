"""GPU test of the translation over malformed arrays: negative starts and ends
past 2^31 are refused, and counting and emission still agree, so that the
statements fill the counted room exactly and nothing behind it is written."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("more", [5, 2])              # operands of the last call: a thread per call, or per entry
@pytest.mark.parametrize("n_arrays", [400, 9000])     # all pairs tested, lists by sort and sweep
@pytest.mark.parametrize("kind", ["negative", "wrapping"])
def test_counted_room(amc, kind, n_arrays, more):
    rng = np.random.default_rng(96)
    start = rng.integers(0, 1 << 20, n_arrays).astype(np.int32)
    length = rng.integers(1, 1 << 10, n_arrays).astype(np.int32)
    k = np.arange(64)
    if kind == "negative":      # even ids end below 0, odd ones reach over it: they meet, but not as listed by start
        start[:64], length[:64] = np.where(k % 2, -10, -100 - k), np.where(k % 2, 20, 95)
    else:                       # ends past 2^31 - 1
        start[:64], length[:64] = 0x7FFFFF00 - k, np.where(k % 2, 0x200, 8)
    n_calls = 128
    # one declared written operand among R ones, of the malformed arrays
    opnd = [np.array([2 * (c % 31) + 1, 2 * (c % 31), 2 * ((c + 7) % 31) + 64 * (c % 2), 100 + c % 50][:2 + c % 3])
            for c in range(n_calls - 1)] + [np.array([200, 201, 202, 203, 204][:more])]
    mode = [np.array([3, 1, 1, 1][:o.size] if i < n_calls - 1 else [1] * more) for i, o in enumerate(opnd)]
    off = np.concatenate([[0], np.cumsum([o.size for o in opnd])])
    t = lambda a, d: torch.from_numpy(np.ascontiguousarray(a).astype(d)).cuda()  # noqa: E731
    args = [t(start, np.int32), t(length, np.int32), t(rng.integers(0, 2, n_calls), np.uint8), t(off, np.int32),
            t(np.concatenate(opnd), np.int32), t(np.concatenate(mode), np.uint8)]
    got = amc.translate_vectorpu(*args, out_cap=1 << 20)
    assert amc.sync_status() == amc.E_INVALID
    n, pad = got["n"], 4096
    first = got["call_first_op"].cpu().numpy()
    assert n == first[-1] and np.all(np.diff(first) >= 0)
    ks = torch.full((n + pad,), 0xFF, dtype=torch.uint8, device="cuda")
    var = torch.full((n + pad,), -7, dtype=torch.int32, device="cuda")
    out = dict(kind_side=ks[:n], var=var[:n], call_first_op=torch.empty(n_calls + 1, dtype=torch.int64, device="cuda"),
               n_dev=torch.empty(1, dtype=torch.int64, device="cuda"))
    amc.translate_vectorpu(*args, known_n=n, out=out)
    assert amc.sync_status() == amc.E_INVALID
    assert bool((ks[n:] == 0xFF).all()) and bool((var[n:] == -7).all())
    assert bool((ks[:n] != 0xFF).all()) and bool((var[:n] >= 0).all())
    assert torch.equal(ks[:n], got["kind_side"]) and torch.equal(var[:n], got["var"])
