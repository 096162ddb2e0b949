"""The work that a program hands to this library, as cases to be measured.

Three integer tables as the tests and the benchmark draw them: D (a dimension),
M (its keys 4i + U{0..3}, a reference into D and a date) and F (facts that
refer to M, with a price, a discount and a date).  A case is one call, or the
few calls that belong together, through the package's public functions:

* ``plan``      the three-table query (filter, join, group by, top-k) over
                resident tables, ``pq_run_plan``;
* ``aggfirst``  the query that groups F first and filters on the sum;
* ``batch``     many such queries over slices of the same tables at once,
                ``pq_run_batch`` (how a server answers its clients);
* ``stream``    the query over packed columns in pinned host memory;
* ``filter``    one predicate, or two joined by AND through a selection vector;
* ``partition`` the radix partition ahead of an exchange;
* ``join``      hash-join build and probe, the matches put in probe order;
* ``groupby``   group-by SUM, then ORDER BY sum LIMIT k.

The operators leave pairs and groups in no defined order, so the join and the
group-by cases put them where their rows belong (by probe row, by M row), as a
program that goes on working with them does.
"""
import math

import torch

import paper_2512_02862_gb300 as pq

DTYPES = {"int8": torch.int8, "int32": torch.int32, "int64": torch.int64}
DATES = 2406        # M.date is uniform over 0..2405
M_DATE, F_DATE = 1200, 1200   # the query's cuts


def listed():
    return [
        # A dashboard query on small tables: one call, its result awaited.
        # Launches and latency are what it costs.
        dict(name="plan_small", kind="plan", n_d=15_000, n_m=150_000, n_f=600_000,
             fk="clustered", pass_all=False, k=10, pinned=False),
        # The ordinary analytical query: every column resident, 1.5 GB read.
        dict(name="plan_x100", kind="plan", n_d=1_500_000, n_m=15_000_000, n_f=60_000_000,
             fk="clustered", pass_all=False, k=10, pinned=True),
        # Skewed foreign keys in no order, nothing filtered out: every F row
        # joins, and there are millions of groups.
        dict(name="plan_skew", kind="plan", n_d=4_000_000, n_m=40_000_000, n_f=200_000_000,
             fk="zipf", pass_all=True, k=10, pinned=True),
        # Large orders: group all of F, keep the groups over a threshold.
        dict(name="aggfirst_x100", kind="aggfirst", n_d=1_500_000, n_m=15_000_000,
             n_f=60_000_000, having=4_000_000_000, k=10),
        # A server's batch: 64 queries over slices whose sizes are lognormal,
        # each with constants of its own.
        dict(name="batch_64", kind="batch", n_d=1_500_000, n_m=15_000_000, n_f=60_000_000,
             queries=64, k=10),
        # Tables kept packed in host memory: each query moves them over the link.
        dict(name="stream_packed", kind="stream", n_d=500_000, n_m=5_000_000, n_f=20_000_000,
             k=10),
        # Filter pushed into a scan of a large date column.
        dict(name="filter_x100", kind="filter", n=60_000_000, type="int32", second=False),
        # Two predicates on a small, odd-sized chunk.
        dict(name="filter_and", kind="filter", n=1_000_003, type="int32", second=True),
        # Partition by join key for 64 receivers: the key and one wide column.
        dict(name="partition_64", kind="partition", n=60_000_000, key="int64",
             payload="int64", log2p=6),
        # Out-of-core fan-out with all columns of F, an odd number of rows.
        dict(name="partition_1024", kind="partition", n=20_000_003, key="int64",
             payload="int64,int8,int32", log2p=10),
        # Foreign-key join: build on M, probe with F.
        dict(name="join_x100", kind="join", n_b=15_000_000, n_p=60_000_000, fk="clustered",
             gap=4, half=False),
        # GROUP BY M key ORDER BY sum DESC LIMIT 10 over all of F.
        dict(name="groupby_x100", kind="groupby", n_m=15_000_000, n=60_000_000,
             fk="clustered", gap=4, k=10),
    ]


def draw(rng):
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1

    kind = rng.choice(["plan", "plan", "plan", "aggfirst", "batch", "stream", "filter", "filter",
                       "partition", "partition", "join", "groupby"])
    k = rng.choice([1, 5, 10, 10, 20, 64])
    if kind == "plan":
        n_f = size(100_000, 150_000_000)
        return dict(kind=kind, n_d=max(64, n_f // 40), n_m=n_f // 4, n_f=n_f,
                    fk=rng.choice(["clustered", "zipf"]), pass_all=rng.random() < 0.4,
                    k=rng.choice([1, 5, 10, 10, 20]), pinned=n_f > 2_000_000)
    if kind == "aggfirst":
        n_f = size(1_000_000, 60_000_000)
        return dict(kind=kind, n_d=n_f // 40, n_m=n_f // 4, n_f=n_f,
                    having=rng.choice([1_000_000_000, 2_000_000_000, 3_000_000_000]), k=10)
    if kind == "batch":
        n_f = size(8_000_000, 60_000_000)
        return dict(kind=kind, n_d=n_f // 40, n_m=n_f // 4, n_f=n_f,
                    queries=rng.randint(8, 128), k=10)
    if kind == "stream":
        n_f = size(2_000_000, 20_000_000)
        return dict(kind=kind, n_d=n_f // 40, n_m=n_f // 4, n_f=n_f, k=10)
    if kind == "filter":
        return dict(kind=kind, n=size(10_000, 60_000_000), type=rng.choice(list(DTYPES)),
                    second=rng.random() < 0.4)
    if kind == "partition":
        return dict(kind=kind, n=size(100_000, 60_000_000), key=rng.choice(["int32", "int64"]),
                    payload=rng.choice(["int64", "int32", "int8,int32", "int64,int8,int32"]),
                    log2p=rng.randint(2, 12))
    if kind == "join":
        n_p = size(100_000, 60_000_000)
        return dict(kind=kind, n_b=n_p // 4, n_p=n_p, fk=rng.choice(["clustered", "zipf"]),
                    gap=rng.choice([4, 64]), half=rng.random() < 0.5)
    n = size(100_000, 60_000_000)
    return dict(kind="groupby", n_m=n // 4, n=n, fk=rng.choice(["clustered", "zipf"]),
                gap=rng.choice([4, 64]), k=k)


# ------------------------------------------------------------------ inputs ----
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, n, dtype):
    """n values of U{lo..hi}."""
    return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=dtype)


def _m_keys(g, n_m, gap):
    """gap * i + U{0..gap-1}: ascending, unique, with gaps."""
    return torch.arange(n_m, device="cuda") * gap + _uniform(g, 0, gap - 1, n_m, torch.int64)


def _references(g, n_f, n_m, fk):
    """The M row of each F row: runs of 1..7 rows in M order, from the start
    again when M is used up (clustered), or Zipf(1.0) ranks spread over M
    (zipf).  Also the first F row of each M row (clustered)."""
    if fk == "zipf":
        # Ranks by the inverse of the logarithmic distribution function.
        u = torch.rand(n_f, generator=g, device="cuda", dtype=torch.float64)
        rank = ((u * math.log(n_m + 1)).exp_().long() - 1).clamp_(0, n_m - 1)
        a = 7_368_787
        while math.gcd(a, n_m) != 1:
            a += 2
        return rank.mul_(a).add_(12_345).remainder_(n_m), None
    reps = _uniform(g, 1, 7, n_m, torch.int64)
    starts = torch.zeros(n_m + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(reps, 0, out=starts[1:])
    at = torch.repeat_interleave(reps)
    while at.numel() < n_f:
        at = torch.cat([at, at[:n_f - at.numel()]])
    return at[:n_f].contiguous(), starts


def _tables(case, seed):
    """D, M, F as dicts of columns, and the M row of each F row."""
    g = _generator(seed)
    n_d, n_m, n_f = case["n_d"], case["n_m"], case["n_f"]
    D = dict(key=torch.arange(1, n_d + 1, device="cuda", dtype=torch.int32),
             seg=_uniform(g, 0, 4, n_d, torch.int8))
    M = dict(key=_m_keys(g, n_m, 4), dref=_uniform(g, 1, n_d, n_m, torch.int32),
             date=_uniform(g, 0, DATES - 1, n_m, torch.int32))
    at, starts = _references(g, n_f, n_m, case.get("fk", "clustered"))
    F = dict(mkey=M["key"][at], price=_uniform(g, 90_000, 10_500_000, n_f, torch.int64),
             disc=_uniform(g, 0, 10, n_f, torch.int8),
             date2=M["date"][at] + _uniform(g, 1, 121, n_f, torch.int32))
    return D, M, F, at, starts


def _query(case):
    """The query's predicates, as make_plan takes them."""
    if case.get("pass_all"):
        return dict(d_op="all", m_op="all", f_op="all")
    return dict(seg=1, m_date_lt=M_DATE, f_date_gt=F_DATE)


def _slices(case, seed, starts):
    """The batch's queries: (M row range, F row range, seg, date cut).  F sizes
    are lognormal around 500k rows; slices start on multiples of 16 rows."""
    g = _generator(seed + 1)
    n, n_m, n_f = case["queries"], case["n_m"], min(case["n_f"], int(starts[-1]))
    z = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    want = (z * 1.5 + math.log(500_000)).exp().clamp_(10_000, n_f // 2).long()
    a = _uniform(g, 0, n_m - 1, n, torch.int64) // 16 * 16
    f0 = starts[a] // 16 * 16
    f0 = torch.minimum(f0, torch.full_like(f0, (n_f - 16) // 16 * 16))
    f1 = torch.minimum(f0 + want, torch.full_like(f0, n_f))
    b = torch.searchsorted(starts, f1)
    b = torch.minimum((b + 15) // 16 * 16, torch.full_like(b, n_m))
    seg, cut = _uniform(g, 0, 4, n, torch.int64), _uniform(g, 200, 2200, n, torch.int64)
    rows = torch.stack([a, (b - a).clamp_(min=0), f0, f1 - f0, seg, cut], 1)
    return [tuple(r) for r in rows.tolist()]


def _join_inputs(case, seed):
    """Build keys and values, probe keys, and where each probe row's match is
    in the build side (-1: none).  half: only every other M row is built."""
    g = _generator(seed)
    keys = _m_keys(g, case["n_b"], case["gap"])
    at, _ = _references(g, case["n_p"], case["n_b"], case["fk"])
    step = 2 if case["half"] else 1
    build = keys[::step].contiguous()
    vals = _uniform(g, 1, case["n_b"], build.numel(), torch.int64)
    return build, vals, keys[at], torch.where(at % step == 0, at // step, -1)


def _filter_inputs(case, seed):
    """The column, its cut, and the second predicate's column (if any).  The
    rows are a shuffle of the same rows for every seed, so that the number of
    rows that pass does not depend on it."""
    lo, hi, cut = {"int8": (0, 10, 4), "int32": (0, DATES + 120, F_DATE),
                   "int64": (90_000, 10_500_000, 8_000_000)}[case["type"]]
    i = torch.randperm(case["n"], generator=_generator(seed), device="cuda")
    col = (lo + (i * 7_919) % (hi - lo + 1)).to(DTYPES[case["type"]])
    second = (((i * 2_654_435_761) >> 16) % 11).to(torch.int8) if case["second"] else None
    return col, cut, second


def _partition_inputs(case, seed):
    g = _generator(seed)
    n = case["n"]
    key = _m_keys(g, max(1, n // 4), 4)[_references(g, n, max(1, n // 4), "clustered")[0]]
    make = {"int64": lambda: _uniform(g, 90_000, 10_500_000, n, torch.int64),
            "int32": lambda: _uniform(g, 0, DATES + 120, n, torch.int32),
            "int8": lambda: _uniform(g, 0, 10, n, torch.int8)}
    return key.to(DTYPES[case["key"]]), [make[t]() for t in case["payload"].split(",")]


def _groupby_inputs(case, seed):
    g = _generator(seed)
    keys = _m_keys(g, case["n_m"], case["gap"])
    at, _ = _references(g, case["n"], case["n_m"], case["fk"])
    return keys[at], _uniform(g, 90_000, 10_500_000, case["n"], torch.int64), keys, at


# ------------------------------------------------------------- the calls ----
_work_stream = None


def _stream():
    """The program's one work stream."""
    global _work_stream
    if _work_stream is None:
        _work_stream = torch.cuda.Stream()
    return _work_stream


def prepare(case, seed):
    kind, s = case["kind"], _stream()
    st = dict(case=case, kind=kind)
    if kind in ("plan", "aggfirst", "batch"):
        D, M, F, _, starts = _tables(case, seed)
        ctx = pq.Context(arena_bytes=(4 << 30) if case["n_f"] <= 60_000_000 else (8 << 30))
        torch.cuda.synchronize()
        T = [pq.pq_load_columns(ctx, list(t.values()), stream=s) for t in (D, M, F)]
        if kind == "batch":
            st["plans"] = [pq.make_plan(*T, seg=seg, m_date_lt=cut, f_date_gt=cut, k=case["k"],
                                        rows=dict(m=(m0, mn), f=(f0, fn)))
                           for m0, mn, f0, fn, seg, cut in _slices(case, seed, starts)]
            st["res"] = pq.pinned_results(case["queries"])
        else:
            st["plan"] = pq.make_plan(*T, k=case["k"], having=case.get("having"), **_query(case))
            st["res"] = pq.pinned_results(1) if case.get("pinned", True) else None
    elif kind == "stream":
        D, M, F, _, _ = _tables(case, seed)
        ctx = pq.Context(chunk_bytes=64 << 20, ring_slots=6, copy_streams=3)
        T = [pq.pq_load_columns(ctx, [pq.pq_pack_column(c.cpu()) for c in t.values()],
                                mode=pq.PQ_STREAMING, stream=s) for t in (D, M, F)]
        st["plan"] = pq.make_plan(*T, k=case["k"], **_query(case))
        st["res"] = pq.pinned_results(1)
    else:
        ctx = pq.Context()
        if kind == "filter":
            st["col"], st["cut"], st["col2"] = _filter_inputs(case, seed)
        elif kind == "partition":
            st["key"], st["pay"] = _partition_inputs(case, seed)
        elif kind == "join":
            st["build"], st["vals"], st["probe"], _ = _join_inputs(case, seed)
        elif kind == "groupby":
            st["key"], st["val"], _, _ = _groupby_inputs(case, seed)
        torch.cuda.synchronize()
    st["ctx"] = ctx
    return st


def _record(res, k):
    """The fields of one result record; `res` in pinned memory is read where
    it lies, once the stream has passed the call."""
    b = res._buf.view(torch.int64)
    return dict(n=b[0:1], ngroups=b[1:2], keys=b[2:2 + k], sums=b[2 + pq.PQ_MAX_K:][:k],
                status=res._buf.view(torch.int32)[4 + 4 * pq.PQ_MAX_K:][:1], hits=b[131:132])


def run(st):
    case, kind, ctx, s = st["case"], st["kind"], st["ctx"], _stream()
    if kind in ("plan", "aggfirst", "stream"):
        if st["res"] is None:  # the call waits and returns the record
            r = pq.pq_run_plan(ctx, st["plan"], stream=s)
            d = r.as_dict()
            return dict(n=int(r.n), ngroups=d["ngroups"], keys=d["keys"], sums=d["sums"],
                        status=d["status"], hits=int(r.hits))
        pq.pq_run_plan(ctx, st["plan"], st["res"][0], stream=s)
        return _record(st["res"], case["k"])
    if kind == "batch":
        # A server hands its clients the rows that each result holds (`hits`
        # counts the probe's inputs, which a hash-table plan has more of).
        pq.pq_run_batch(ctx, st["plans"], st["res"], stream=s)
        ctx.sync(s)
        b = st["res"]._buf.view(torch.int64).view(case["queries"], -1)
        k, kmax = case["k"], pq.PQ_MAX_K
        held = torch.arange(k)[None, :] < b[:, :1]
        return dict(n=b[:, 0].clone(), ngroups=b[:, 1].clone(),
                    keys=torch.where(held, b[:, 2:2 + k], 0),
                    sums=torch.where(held, b[:, 2 + kmax:2 + kmax + k], 0))
    with torch.cuda.stream(s):
        if kind == "filter":
            sel, cnt = pq.pq_filter(ctx, st["col"], ">", st["cut"], stream=s)
            if st["col2"] is not None:
                sel, cnt = pq.pq_filter(ctx, st["col2"], "<=", 6, sel_in=sel, d_n_in=cnt,
                                        stream=s)
            return sel[:int(cnt)]
        if kind == "partition":
            key, pay, off = pq.pq_partition(ctx, st["key"], st["pay"], log2P=case["log2p"],
                                            stream=s)
            return dict(key=key, pay=pay, offsets=off)
        if kind == "join":
            n_p = case["n_p"]
            ht = pq.pq_join_build(ctx, st["build"], st["vals"], stream=s)
            rows, vals, cnt = pq.pq_join_probe(ctx, ht, st["probe"], cap=n_p, stream=s)
            ht.free(s)
            pairs = int(cnt)
            joined = torch.full((n_p,), -1, dtype=torch.int64, device="cuda")
            return dict(pairs=pairs, joined=joined.scatter_(0, rows[:pairs], vals[:pairs]))
        keys, sums, cnt = pq.pq_groupby_sum(ctx, st["key"], st["val"], cap=case["n_m"], stream=s)
        g = int(cnt)
        top_k, top_s, _ = pq.pq_topk(ctx, keys[:g], sums[:g], case["k"], stream=s)
        by_row = torch.zeros(case["n_m"], dtype=torch.int64, device="cuda")
        by_row.scatter_(0, keys[:g] // case["gap"], sums[:g])
        return dict(groups=g, sums=by_row, top_keys=top_k, top_sums=top_s)


# -------------------------------------------------------------- the results ----
def _top(keys, sums, k):
    """The first k of (keys, sums) by sum descending, key ascending."""
    order = torch.argsort(keys, stable=True)
    order = order[torch.argsort(sums[order], descending=True, stable=True)][:k]
    return keys[order], sums[order]


def _exact_plan(case, D, M, F, at, q, seg=1, m0=0, mn=None, f0=0, fn=None):
    """ngroups, hits, keys, sums of the query over M and F row ranges, by M row."""
    n_m = case["n_m"]
    mn, fn = n_m if mn is None else mn, case["n_f"] if fn is None else fn
    a, f = at[f0:f0 + fn], {c: v[f0:f0 + fn] for c, v in F.items()}
    keep_m = torch.zeros(n_m, dtype=torch.bool, device="cuda")
    keep_m[m0:m0 + mn] = True
    if q is not None:
        keep_m &= (M["date"] < q[0]) & (D["seg"] == seg)[(M["dref"] - 1).long()]
    keep_f = f["date2"] > q[1] if q is not None else torch.ones_like(f["date2"], dtype=torch.bool)
    rev = f["price"] * (100 - f["disc"].long())
    having = case.get("having")
    hit = keep_f if having is not None else keep_f & keep_m[a]
    sums = torch.zeros(n_m, dtype=torch.int64, device="cuda")
    sums.index_add_(0, a[hit], rev[hit])
    seen = torch.zeros(n_m, dtype=torch.bool, device="cuda")
    seen[a[hit]] = True
    if having is not None:
        seen &= keep_m & (sums > having)
    keys, vals = _top(M["key"][seen], sums[seen], case["k"])
    return int(seen.sum()), int(hit.sum()), keys, vals


def exact(case, seed):
    kind = case["kind"]
    if kind in ("plan", "aggfirst", "stream"):
        D, M, F, at, _ = _tables(case, seed)
        q = None if case.get("pass_all") else (M_DATE, F_DATE)
        groups, hits, keys, sums = _exact_plan(case, D, M, F, at, q)
        out = dict(n=keys.numel(), ngroups=groups, keys=keys, sums=sums, status=0, hits=hits)
        if not case.get("pinned", True):
            out["keys"], out["sums"] = keys.tolist(), sums.tolist()
        return out
    if kind == "batch":
        D, M, F, at, starts = _tables(case, seed)
        out = dict(n=[], ngroups=[], keys=[], sums=[])
        for m0, mn, f0, fn, seg, cut in _slices(case, seed, starts):
            groups, _, keys, sums = _exact_plan(case, D, M, F, at, (cut, cut), seg, m0, mn, f0,
                                                fn)
            pad = [0] * (case["k"] - keys.numel())
            for name, v in (("n", keys.numel()), ("ngroups", groups),
                            ("keys", keys.tolist() + pad), ("sums", sums.tolist() + pad)):
                out[name].append(v)
        return {name: torch.tensor(v) for name, v in out.items()}
    if kind == "filter":
        col, cut, col2 = _filter_inputs(case, seed)
        keep = col > cut
        return torch.nonzero(keep if col2 is None else keep & (col2 <= 6)).flatten()
    if kind == "partition":
        key, pay = _partition_inputs(case, seed)
        # Fibonacci hashing in wrapping 64-bit arithmetic: the top bits.
        h = key.long() * (0x9E3779B97F4A7C15 - (1 << 64))
        p = 1 << case["log2p"]
        bucket = (h >> (64 - case["log2p"])) & (p - 1)
        order = torch.argsort(bucket, stable=True)
        offsets = torch.zeros(p + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(torch.bincount(bucket, minlength=p), 0, out=offsets[1:])
        return dict(key=key[order], pay=[c[order] for c in pay], offsets=offsets)
    if kind == "join":
        _, vals, _, match = _join_inputs(case, seed)
        return dict(pairs=int((match >= 0).sum()),
                    joined=torch.where(match >= 0, vals[match.clamp(min=0)], -1))
    _, val, keys, at = _groupby_inputs(case, seed)
    sums = torch.zeros(case["n_m"], dtype=torch.int64, device="cuda").index_add_(0, at, val)
    seen = torch.zeros(case["n_m"], dtype=torch.bool, device="cuda")
    seen[at] = True
    top_k, top_s = _top(keys[seen], sums[seen], case["k"])
    return dict(groups=int(seen.sum()), sums=sums, top_keys=top_k, top_sums=top_s)


def work(case):
    """Bytes of one pass: every input read once, every output written once."""
    kind = case["kind"]
    size = {"int8": 1, "int32": 4, "int64": 8}
    if kind in ("plan", "aggfirst"):
        b = 21 * case["n_f"] + 16 * case["n_m"] + 5 * case["n_d"]
    elif kind == "batch":
        # Each query's slices (800k F rows on average) and the shared D.
        rows = case["queries"] * min(1_200_000, case["n_f"] // 4)
        b = 21 * rows + 16 * rows // 4 + 5 * case["n_d"]
    elif kind == "stream":
        # Packed widths of the columns: F 13 + 24 + 4 + 12 bits a row, M 14 + 20 + 12, D 12 + 3.
        b = (53 * case["n_f"] + 46 * case["n_m"] + 15 * case["n_d"]) // 8
    elif kind == "filter":
        share = {"int8": 6 / 11, "int32": 0.525, "int64": 0.24}[case["type"]]
        n = case["n"]
        b = size[case["type"]] * n + 8 * n * share * (7 / 11 if case["second"] else 1)
        b += n * share if case["second"] else 0
    elif kind == "partition":
        row = size[case["key"]] + sum(size[t] for t in case["payload"].split(","))
        b = 2 * row * case["n"] + 8 * ((1 << case["log2p"]) + 1)
    elif kind == "join":
        b = 16 * case["n_b"] // (2 if case["half"] else 1) + (8 + 8) * case["n_p"]
    else:
        b = 16 * case["n"] + 8 * case["n_m"]
    return {"bytes": float(b), "flops": 0.0}
