"""GPU tests of how well-declaredness calls are dealt to warps: a few long calls
go to a warp each, and calls with many written arrays match the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amc():
    import paper_1910_11110_gb300 as m
    m.build()
    return m


def calls(n_calls, n_decls, locs, reads_every=0, gap=False):
    """n_calls calls that write every location of n_decls W arrays each; with gap,
    call c leaves out one location of its (c mod n_decls)-th array."""
    n_arrays = n_calls + n_decls
    tok_off, tok, pay, am_off, am, mode = [0], [], [], [0], [], []
    for c in range(n_calls):
        for d in range(n_decls):
            for i in range(locs):
                if gap and d == c % n_decls and i == c % locs:
                    continue
                tok.append(1)
                pay.append((c + d) * locs + i)
            am.append(c + d)
            mode.append(3 if reads_every and d % reads_every == 0 else 2)
        tok_off.append(len(tok))
        am_off.append(len(am))
    return dict(arr_loc_off=np.arange(n_arrays + 1, dtype=np.int64) * locs,
                loc_owner=np.repeat(np.arange(n_arrays), locs).astype(np.int32), call_tok_off=np.array(tok_off, np.int64),
                tok=np.array(tok, np.uint8), payload=np.array(pay, np.int32), call_am_off=np.array(am_off, np.int64),
                am_array=np.array(am, np.int32), am_mode=np.array(mode, np.uint8))


def run(amc, w):
    t = {k: torch.from_numpy(v).cuda() for k, v in w.items()}
    return lambda: amc.check_well_declared(t["arr_loc_off"], t["loc_owner"], t["call_tok_off"], t["tok"], t["payload"],
                                           t["call_am_off"], t["am_array"], t["am_mode"])


@pytest.mark.parametrize("n_decls", [1, 4, 5, 6, 31, 32])
@pytest.mark.parametrize("locs,reads_every", [(1, 0), (7, 3), (100, 0)])
def test_many_written_arrays(amc, oracle_mod, n_decls, locs, reads_every):
    w = calls(37, n_decls, locs, reads_every, gap=True)
    out = run(amc, w)()
    assert amc.sync_status() == 0
    exp = oracle_mod.well_declared(**w)
    got = (out["violations"].cpu().numpy().astype(np.uint32), out["first_bad"].cpu().numpy(), out["first_unmet"].cpu().numpy())
    for e, g in zip(exp, got):
        assert np.array_equal(e, g)


def test_long_calls_side_by_side(amc):
    # 64 calls of 4,000 tokens on 152 SMs take about as long as one (eight times as
    # long when a warp took eight of them one after another)
    def us(f):
        f()
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                f()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 250)
        return best

    one, many = us(run(amc, calls(1, 2, 2000))), us(run(amc, calls(64, 2, 2000)))
    assert many < 3 * one, (one, many)
