"""Cases for timing the checker: what a user has it do, through its public entry points.

Every case is one call (or the two calls that belong together: translate, then check) on inputs that are already on
the GPU, as a program that records or generates them there has them.  The inputs are drawn on the GPU from the seed
alone, with the distributions of this repository's workloads (Zipf ids, its kind mixes, its array lengths, modes,
program shapes and lifetimes); sizes are those of its workloads, smaller ones of the same kinds, and odd ones.

Every output is a status code, a mask, an index or a count: whole numbers, the same for every correct implementation.
"""
import math
import random

import numpy as np
import torch

import paper_1910_11110_gb300 as amc

DEV = "cuda"
MIXES = {  # r, w, Push, Pull, Noop
    "uniform": (0.2, 0.2, 0.2, 0.2, 0.2),
    "mixed": (0.40, 0.20, 0.15, 0.15, 0.10),
    "low_fault": (0.02, 0.60, 0.05, 0.05, 0.28),
}
MODES = (0.5, 0.3, 0.2)  # R, W, RW
DROP = 1e-4              # annotations dropped


def listed():
    return [
        # the smallest call in use: a unit-test sized trace over a few variables, where the launch is the time
        {"name": "trace_4k", "path": "trace", "ops": 4096, "vars": 16, "ids": "uniform", "mix": "uniform", "init": False},
        # one trace request of a session that keeps its statuses between requests
        {"name": "trace_session", "path": "trace", "ops": 300_007, "vars": 2_011, "ids": "uniform", "mix": "mixed",
         "init": True},
        # a recorded run of ordinary length over many variables, hot and cold
        {"name": "trace_zipf_16m", "path": "trace", "ops": (1 << 24) + 77, "vars": 1 << 20, "ids": "zipf", "mix": "mixed",
         "init": False},
        # the longest recorded run: the trace of the headline benchmark
        {"name": "trace_zipf_1g", "path": "trace", "ops": 1 << 30, "vars": 1 << 20, "ids": "zipf", "mix": "mixed",
         "init": False},
        # a long run of a program that is mostly right, continued from known statuses, ragged sizes
        {"name": "trace_low_fault", "path": "trace", "ops": 150_000_001, "vars": 1_000_003, "ids": "zipf",
         "mix": "low_fault", "init": True},
        # a component program over many overlapping arrays: translation and guarded check
        {"name": "vectorpu", "path": "vectorpu", "arrays": 4096, "calls": 5_000_011, "infer": True},
        # the same for a short component program, where launches and the host read count
        {"name": "vectorpu_small", "path": "vectorpu", "arrays": 64, "calls": 3_001, "infer": True},
        # a component program that creates and deletes partial vectors as it runs
        {"name": "lifetimes", "path": "lifetimes", "vectors": 16, "pvectors": 16_384, "calls": 1_000_003},
        # a batch of structured programs in relation mode
        {"name": "programs", "path": "programs", "progs": 100_000, "vars_lo": 64, "vars_hi": 4096, "guarded": False},
        # the same with conditions on a guard variable that are evaluated
        {"name": "programs_guarded", "path": "programs", "progs": 20_000, "vars_lo": 16, "vars_hi": 256, "guarded": True},
        # the static check of function bodies against their declarations, a whole code base at once
        {"name": "well_declared", "path": "well_declared", "arrays": 4096, "calls": 1 << 20},
        # a recorded run on a node with several accelerators
        {"name": "trace_k4", "path": "trace_k", "ops": 100_000_007, "vars": 1 << 20, "k": 4},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(("trace", "trace", "trace", "vectorpu", "vectorpu", "lifetimes", "programs", "programs",
                       "well_declared", "trace_k"))
    if path == "trace":
        if rng.random() < 0.5:    # one session's request, or a short run
            return {"path": path, "ops": size(1 << 10, 1 << 24), "vars": rng.randint(16, 4096), "ids": "uniform",
                    "mix": rng.choice(("uniform", "mixed")), "init": rng.random() < 0.5}
        return {"path": path, "ops": size(1 << 20, 1 << 29), "vars": size(1 << 13, 1 << 20), "ids": "zipf",
                "mix": rng.choice(("mixed", "low_fault")), "init": rng.random() < 0.5}
    if path == "vectorpu":
        return {"path": path, "arrays": size(32, 4096), "calls": size(1 << 10, 5_000_011), "infer": rng.random() < 0.8}
    if path == "lifetimes":
        return {"path": path, "vectors": rng.randint(2, 16), "pvectors": size(256, 16_384), "calls": size(1 << 14, 1_000_003)}
    if path == "programs":
        if rng.random() < 0.5:
            return {"path": path, "progs": size(1, 20_000), "vars_lo": 16, "vars_hi": 256, "guarded": True}
        return {"path": path, "progs": size(1, 100_000), "vars_lo": 64, "vars_hi": 4096, "guarded": False}
    if path == "well_declared":
        return {"path": path, "arrays": size(64, 4096), "calls": size(1 << 10, 1 << 20)}
    return {"path": path, "ops": size(1 << 14, 100_000_007), "vars": size(1 << 10, 1 << 20), "k": rng.randint(2, 7)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _uniform(g, lo, hi, n, dtype=torch.int64):
    """n whole numbers in [lo, hi]."""
    return torch.randint(lo, hi + 1, (n,), generator=g, device=DEV, dtype=dtype)


def _kinds(g, n, mix):
    cdf = torch.tensor(np.cumsum(mix)[:-1], dtype=torch.float32, device=DEV)
    return torch.searchsorted(cdf, torch.rand(n, generator=g, device=DEV), right=True, out_int32=True).to(torch.uint8)


def _ids(g, n, n_vars, ids):
    """Variable ids: uniform, or Zipf(1.05) by inverse CDF with the heavy ids first."""
    if ids == "uniform":
        return _uniform(g, 0, n_vars - 1, n, torch.int32)
    out = torch.empty(n, dtype=torch.int32, device=DEV)
    w = torch.arange(1, n_vars + 1, dtype=torch.float64, device=DEV) ** -1.05
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    for lo in range(0, n, 1 << 27):
        u = torch.rand(min(1 << 27, n - lo), generator=g, device=DEV, dtype=torch.float64)
        out[lo:lo + u.numel()] = torch.searchsorted(cdf, u, out_int32=True).clamp_(max=n_vars - 1)
    return out


def _trace(case, g):
    n, nv = case["ops"], case["vars"]
    ks = torch.empty(n, dtype=torch.uint8, device=DEV)
    for lo in range(0, n, 1 << 27):
        m = min(1 << 27, n - lo)
        ks[lo:lo + m] = _kinds(g, m, MIXES[case["mix"]]) | (_uniform(g, 0, 1, m, torch.uint8) << 4)
    # statuses that an earlier trace left behind: any valid pair, a few of them stuck
    init = None
    if case["init"]:
        init = _uniform(g, 1, 3, nv, torch.uint8)
        init[torch.rand(nv, generator=g, device=DEV) < 0.02] = amc.ST_F
    return {"ks": ks, "var": _ids(g, n, nv, case["ids"]), "vars": nv, "init": init}


def _trace_k(case, g):
    n, k = case["ops"], case["k"]
    cdf = torch.tensor([0.4, 0.6, 0.9], dtype=torch.float32, device=DEV)      # r, w, copy, Noop
    kind = torch.searchsorted(cdf, torch.rand(n, generator=g, device=DEV), right=True, out_int32=True).to(torch.uint8)
    a = _uniform(g, 0, k - 1, n, torch.uint8)
    b = (a + _uniform(g, 1, k - 1, n, torch.uint8)) % k
    op = torch.where(kind == 3, kind, kind | (a << 2) | torch.where(kind == 2, b << 5, torch.zeros_like(b)))
    return {"op": op, "var": _ids(g, n, case["vars"], "zipf"), "vars": case["vars"], "k": k}


def _lengths(g, n):
    return torch.exp2(torch.rand(n, generator=g, device=DEV) * 8 + 8).to(torch.int64)


def _distinct(counts, width, pick):
    """[calls, width] ids from pick(mask), the first counts[c] of row c distinct, and which of them are used."""
    got = pick(torch.ones((counts.numel(), width), dtype=torch.bool, device=DEV))
    used = torch.arange(width, device=DEV)[None, :] < counts[:, None]
    while True:
        dup = torch.zeros_like(used)
        for j in range(1, width):
            for i in range(j):
                dup[:, j] |= got[:, j] == got[:, i]
        dup &= used
        if not bool(dup.any()):
            return got, used
        got[dup] = pick(dup)[dup]


def _modes(g, n):
    m = torch.searchsorted(torch.tensor([MODES[0], MODES[0] + MODES[1]], device=DEV),
                           torch.rand(n, generator=g, device=DEV), right=True, out_int32=True).to(torch.uint8) + 1
    m[torch.rand(n, generator=g, device=DEV) < DROP] |= 0x80
    return m


def _offsets(counts, dtype=torch.int64):
    off = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=off[1:])
    return off.to(dtype)


def _vectorpu(case, g):
    """The number of statements depends on which arrays overlap and on the operands: those are the case's own, and the
    seed numbers the arrays, orders the calls and draws their sides."""
    own = _gen(1)
    A, C = case["arrays"], case["calls"]
    space = 4096 * A                      # the density of 4,096 arrays over 2^24 elements
    start = _uniform(own, 0, space - 1, A)
    length = torch.minimum(_lengths(own, A), space - start)
    counts = _uniform(own, 1, 4, C)
    opnd, used = _distinct(counts, 4, lambda m: _uniform(own, 0, A - 1, m.numel()).view(m.shape))
    mode = _modes(own, 4 * C).view(C, 4)
    number = torch.randperm(A, generator=g, device=DEV)
    at = torch.argsort(number)
    order = torch.randperm(C, generator=g, device=DEV)
    used = used[order]
    return {"start": start[at].to(torch.int32), "len": length[at].to(torch.int32),
            "side": _uniform(g, 0, 1, C, torch.uint8), "off": _offsets(counts[order], torch.int32),
            "opnd": number[opnd[order]][used].to(torch.int32), "mode": mode[order][used], "infer": case["infer"]}


def _lifetimes(case, g):
    """As above: the seed numbers the arrays, may mirror the elements and draws the sides."""
    own = _gen(2)
    V, P, C, L = case["vectors"], case["pvectors"], case["calls"], 1 << 20
    born = torch.sort(_uniform(own, 0, C - 1, P)).values
    life = torch.empty(P, device=DEV).exponential_(16.0 / C, generator=own).to(torch.int64).clamp_(min=1)
    died = torch.minimum(born + life, torch.tensor(C, device=DEV))
    of = _uniform(own, 0, V - 1, P)
    at = _uniform(own, 0, L - 1, P)
    length = torch.minimum(_lengths(own, P), L - at)
    counts = _uniform(own, 1, 4, C)
    whole = torch.arange(V, device=DEV)
    calls = torch.arange(C, device=DEV)
    first = torch.searchsorted(born, calls - C // 4)                  # four mean lifetimes back
    upto = torch.searchsorted(born, calls, right=True)
    live = upto - torch.searchsorted(torch.sort(died).values, calls, right=True)

    def pick(m):      # one of the live arrays: a vector, or a pvector born lately that is not deleted yet
        row = m.nonzero()[:, 0]
        got = _uniform(own, 0, V - 1, row.numel())
        todo = (torch.rand(row.numel(), generator=own, device=DEV) * (V + live[row]) >= V).nonzero()[:, 0]
        for _ in range(24):
            r = row[todo]
            span = upto[r] - first[r]
            p = first[r] + (torch.rand(r.numel(), generator=own, device=DEV) * span).to(torch.int64)
            p = torch.minimum(p, (upto[r] - 1).clamp_(min=0))
            ok = (span > 0) & (born[p] <= r) & (died[p] > r)
            got[todo[ok]] = V + p[ok]
            todo = todo[~ok]
        out = torch.zeros(m.shape, dtype=torch.int64, device=DEV)
        out[m] = got
        return out

    opnd, used = _distinct(counts.clamp_(max=V), 4, pick)
    mode = _modes(own, 4 * C).view(C, 4)
    start = torch.cat((whole * L, of * L + at))
    length = torch.cat((torch.full_like(whole, L), length))
    parent = torch.cat((torch.full_like(whole, -1), of))
    born = torch.cat((torch.zeros_like(whole), born))
    died = torch.cat((torch.full_like(whole, C), died))
    number = torch.randperm(V + P, generator=g, device=DEV)
    back = torch.argsort(number)
    start = torch.where(torch.rand(1, generator=g, device=DEV) < 0.5, start, V * L - start - length)
    parent = torch.where(parent < 0, parent, number[parent.clamp(min=0)])
    i32 = lambda a: a[back].to(torch.int32)  # noqa: E731
    return {"start": i32(start), "len": i32(length), "parent": i32(parent), "born": i32(born), "died": i32(died),
            "side": _uniform(g, 0, 1, C, torch.uint8), "off": _offsets(counts, torch.int32),
            "opnd": number[opnd][used].to(torch.int32), "mode": mode[used]}


def _constructs(seed, count):
    """Ifs and Whiles nested to depth 4 (If .05, While .03 per node, branches of 0..32 and bodies of 1..64 leaf ops):
    their tokens (0 for a leaf op) and payloads, back to back, and where each begins."""
    r = random.Random(seed)
    tok, pay, off = [], [], [0]

    def if_(budget, depth):
        t = min(r.randint(0, 32), budget)
        e = min(r.randint(0, 32), budget - t)
        at = len(tok)
        tok.append(8), pay.append(0)
        body(t, depth + 1)
        other = len(tok)
        tok.append(9), pay.append(0)
        body(e, depth + 1)
        pay[at], pay[other] = other - at - 1, len(tok) - other - 1
        tok.append(11), pay.append(0)
        return t + e

    def while_(budget, depth):
        b = min(r.randint(1, 64), budget)
        at = len(tok)
        tok.append(10), pay.append(0)
        body(b, depth + 1)
        pay[at] = len(tok) - at - 1
        tok.append(11), pay.append(0)
        return b

    def body(budget, depth):
        while budget > 0:
            u = r.random() if depth < 4 else 1.0
            if u < 0.05:
                budget -= if_(budget, depth)
            elif u < 0.08:
                budget -= while_(budget, depth)
            else:
                tok.append(0), pay.append(0)
                budget -= 1

    for _ in range(count):
        (if_ if r.random() < 0.625 else while_)(1 << 20, 0)
        off.append(len(tok))
    return tok, pay, off


def _programs(case, g):
    """The statements' lengths and the programs' sizes are the case's own, so that the token count is; the seed orders
    both and draws the operations, their variables and the conditions."""
    own = _gen(3)
    P, K = case["progs"], 512
    tok, pay, off = _constructs(3, K)
    # item 0 is a leaf op, item k the construct k - 1
    b_tok = torch.tensor([0] + tok, dtype=torch.uint8, device=DEV)
    b_pay = torch.tensor([0] + pay, dtype=torch.int32, device=DEV)
    b_off = torch.tensor([0, 1] + [1 + o for o in off[1:]], dtype=torch.int64, device=DEV)
    b_len = b_off[1:] - b_off[:-1]
    nv = _uniform(own, case["vars_lo"], case["vars_hi"], P, torch.int32)[torch.randperm(P, generator=g, device=DEV)]
    leaves = torch.exp(torch.randn(P, generator=own, device=DEV) * 0.7356 + math.log(2048.0)).clamp_(1, 1 << 20)
    items = (leaves / 3.5).to(torch.int64).clamp_(min=1)          # a top-level statement has 3.5 leaf ops on average
    item_off = _offsets(items[torch.randperm(P, generator=g, device=DEV)])
    n_items = int(item_off[-1])
    item = torch.where(torch.rand(n_items, generator=own, device=DEV) < 0.08, _uniform(own, 1, K, n_items),
                       torch.zeros(1, dtype=torch.int64, device=DEV))
    item = item[torch.randperm(n_items, generator=g, device=DEV)]
    at = _offsets(b_len[item])
    tok_off = at[item_off]
    n = int(at[-1])
    src = torch.repeat_interleave(b_off[item] - at[:-1], b_len[item], output_size=n)
    src += torch.arange(n, device=DEV)
    t, payload = b_tok[src], b_pay[src]
    del src, item, at
    prog = torch.repeat_interleave(torch.arange(P, dtype=torch.int32, device=DEV), tok_off[1:] - tok_off[:-1], output_size=n)
    leaf = t == 0
    op = _kinds(g, n, MIXES["mixed"]) | (_uniform(g, 0, 1, n, torch.uint8) << 4)
    var = (torch.rand(n, generator=g, device=DEV) * nv[prog]).to(torch.int32)
    var = torch.minimum(var, nv[prog] - 1)
    t = torch.where(leaf, op, t)
    payload = torch.where(leaf, var, payload)
    s = {"nv": nv, "tok_off": tok_off, "var_off": _offsets(nv)}
    if case["guarded"]:
        # a guard variable that only writes flip; each If tests it (isValid, remIsValid) or is opaque
        s["guard"] = (torch.rand(P, generator=g, device=DEV) * nv).to(torch.int32).clamp_(max=case["vars_hi"] - 1)
        s["guard"] = torch.minimum(s["guard"], nv - 1)
        t = torch.where(t == 8, t | (_uniform(g, 0, 2, n, torch.uint8) << 4), t)
        wr = torch.where(torch.rand(n, generator=g, device=DEV) < 0.7, 1, 4).to(torch.uint8)
        t = torch.where(leaf & (payload == s["guard"][prog]), (t & 0x10) | wr, t)
    s["tok"], s["payload"] = t, payload
    return s


def _well_declared(case, g):
    A, C = case["arrays"], case["calls"]
    lens = _uniform(g, 1, 64, A)
    a_off = _offsets(lens)
    owner = torch.repeat_interleave(torch.arange(A, dtype=torch.int32, device=DEV), lens)
    nd = _uniform(g, 1, 4, C)
    am, used = _distinct(nd, 4, lambda m: _uniform(g, 0, A - 1, m.numel()).view(m.shape))
    am = am[used].to(torch.int32)
    D = am.numel()
    call = torch.repeat_interleave(torch.arange(C, device=DEV), nd)
    side = _uniform(g, 0, 1, C, torch.uint8)[call] << 4
    mode = _modes(g, D) & 3
    flawed = torch.rand(D, generator=g, device=DEV) < 0.004       # about one call in a hundred
    u = torch.rand(D, generator=g, device=DEV)
    w = mode == 2
    # what the body does for each declaration: 0 writes every location, 1 in both branches of an If, 2 in a While only
    # (a flaw), 3 reads, or reads and writes, 4 the same in a While; some with a Noop after it, or a flaw in its place
    what = torch.where(w, torch.where(flawed & (u < 0.5), 2, torch.where(u < 0.3, 1, 0)), torch.where(u < 0.2, 4, 3))
    n1 = lens[am.long()]
    reads = _uniform(g, 1, 4, D) * torch.where((mode == 3) & (torch.rand(D, generator=g, device=DEV) < 0.75), 2, 1)
    inner = torch.where(w, n1, reads)
    size = torch.where(what == 1, 2 * inner + 3, torch.where((what == 2) | (what == 4), inner + 2, inner))
    tail = (flawed & (what != 2)) | (torch.rand(D, generator=g, device=DEV) < 0.2)
    seg_off = _offsets(size + tail)
    n = int(seg_off[-1])
    seg = torch.repeat_interleave(torch.arange(D, device=DEV), size + tail, output_size=n)
    j = torch.arange(n, device=DEV) - seg_off[seg]
    sw, si, sz, sd = what[seg], inner[seg], size[seg], side[seg]
    wrapped = (sw == 1) | (sw == 2) | (sw == 4)
    q = j - wrapped.to(torch.int64)                                   # place inside the first branch or body
    q = torch.where((sw == 1) & (j > si + 1), j - si - 2, q)          # ... or inside the second branch
    base = a_off[am.long()][seg]
    two = (sw >= 3) & (mode[seg] == 3)
    loc = torch.where(sw >= 3, base + (torch.rand(n, generator=g, device=DEV) * lens[am.long()][seg]).to(torch.int64)
                      .clamp_(max=63), base + q)
    loc = torch.minimum(loc, a_off[am.long() + 1][seg] - 1)
    kind = torch.where(sw < 3, 1, torch.where(two, q & 1, 0)).to(torch.uint8)
    tok, payload = kind | sd, loc
    bad = flawed[seg]
    for at, t, v in (((j == 0) & wrapped, torch.where(sw == 1, 8, 10), si), ((sw == 1) & (j == si + 1), 9, si),
                     (wrapped & (j == sz - 1), 11, 0),
                     (j == sz, torch.where(bad, _uniform(g, 0, 2, n), 4).to(torch.uint8) | sd,
                      torch.where(bad, _uniform(g, 0, owner.numel() - 1, n), base))):
        tok = torch.where(at, torch.as_tensor(t, device=DEV).to(torch.uint8), tok)
        payload = torch.where(at, torch.as_tensor(v, device=DEV), payload)
    am_off = _offsets(nd)
    return {"a_off": a_off, "owner": owner, "tok_off": seg_off[am_off], "tok": tok, "payload": payload.to(torch.int32),
            "am_off": am_off, "am": am, "mode": mode | side}


def prepare(case, seed):
    g, path = _gen(seed), case["path"]
    make = {"trace": _trace, "trace_k": _trace_k, "vectorpu": _vectorpu, "lifetimes": _lifetimes,
            "programs": _programs, "well_declared": _well_declared}
    s = make[path](case, g)
    s["path"] = path
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    path = s["path"]
    if path == "trace":
        return amc.check_trace(s["ks"], s["var"], s["vars"], s["init"])
    if path == "trace_k":
        return amc.check_trace_k(s["op"], s["var"], s["vars"], s["k"])
    if path == "vectorpu":
        t = amc.translate_vectorpu(s["start"], s["len"], s["side"], s["off"], s["opnd"], s["mode"],
                                   infer_overlap=s["infer"])
        out = amc.check_trace(t["kind_side"], t["var"], 2 * s["start"].numel(), guarded=True)
        return [out, t["kind_side"], t["var"], t["call_first_op"]]
    if path == "lifetimes":
        t = amc.translate_vectorpu_lifetimes(s["start"], s["len"], s["parent"], s["born"], s["died"], s["side"],
                                             s["off"], s["opnd"], s["mode"])
        out = amc.check_inherited_trace(t["kind_side"], t["var"], s["start"].numel(), s["parent"], t["arr_probe"])
        return [out, t["kind_side"], t["var"], t["call_first_op"], t["arr_probe"]]
    if path == "programs" and "guard" in s:
        return amc.check_batch_guarded(s["tok"], s["payload"], s["tok_off"], s["nv"], s["guard"], s["var_off"])
    if path == "programs":
        return amc.check_batch(s["tok"], s["payload"], s["tok_off"], s["nv"], s["var_off"])
    return amc.check_well_declared(s["a_off"], s["owner"], s["tok_off"], s["tok"], s["payload"], s["am_off"], s["am"],
                                   s["mode"])


def work(case):
    """Inputs read once and outputs written once; one transition per op for the operations."""
    path = case["path"]
    if path == "trace":
        n, v = case["ops"], case["vars"]
        return {"bytes": 6 * n + (6 if case["init"] else 5) * v, "flops": n}
    if path == "trace_k":
        return {"bytes": 6 * case["ops"] + 5 * case["vars"], "flops": case["ops"]}
    if path in ("vectorpu", "lifetimes"):
        C = case["calls"]
        # 2.5 operands a call, half of them written; a written array carries its m overlapping ones along: three
        # statements for the shadow, one for the projection.  Out come 6 bytes a statement and 8 a call.
        mean = (2.0 ** 16 - 2.0 ** 8) / (8 * math.log(2.0))
        if path == "vectorpu":
            A, live = case["arrays"], 0
            m = 2 * mean / 4096
            each = 3.9 + 0.5 * m * (4 if case["infer"] else 1)
        else:
            A, live = case["vectors"] + case["pvectors"], case["pvectors"] / 16
            m = 2 * mean * live / (case["vectors"] << 20) + 1
            each = 3.9 + 0.5 * m * 4
        n = 2.5 * each * C
        return {"bytes": 17.5 * C + 14 * A + 7 * n + 8 * C, "flops": n}
    if path == "programs":
        tokens, nv = 3_300.0 * case["progs"], (case["vars_lo"] + case["vars_hi"]) / 2 * case["progs"]
        return {"bytes": 6 * tokens + nv + 28 * case["progs"], "flops": tokens}
    tokens = 38.4 * case["calls"]
    return {"bytes": 5 * tokens + case["calls"] * (32 + 2.5 * 5), "flops": tokens}


def exact(case, seed):
    """Statuses, masks, indices and counts: no output is a rounded number that 64 bits would give more exactly."""
    return None
