"""Operators at the sizes where their kernels change shape: edges of warp
tiles and blocks, the rules that choose between kernels, scratch that does
not fit.  Everything is an integer and compared for equality with the
oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = pq.Context(arena_bytes=6 << 30)
    yield c
    c.close()


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check_filter(ctx, stream, a, op, c, off=0, sel=None, d_n=None):
    x = dev(a)[off:]
    y = None if sel is None else dev(sel)
    n_dev = None if d_n is None else torch.tensor([d_n], device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        out, cnt = pq.pq_filter(ctx, x, op, c, sel_in=y, d_n_in=n_dev, stream=stream)
        ctx.sync(stream)
    want = oracle.filter(a[off:], op, c, sel if d_n is None else sel[:d_n])
    assert int(cnt.item()) == len(want)
    assert np.array_equal(out[:len(want)].cpu().numpy(), want)


# One warp tile is 512 rows, one block of the single launch 32 of them.
@pytest.mark.parametrize("dt", [np.int8, np.int32, np.int64])
@pytest.mark.parametrize("n", [511, 512, 513, 16383, 16384, 16385, 24_577, 3_000_011])
@pytest.mark.parametrize("off", [0, 1])
def test_filter_tile_edges(ctx, stream, dt, n, off):
    rng = np.random.default_rng(n + off)
    info = np.iinfo(dt)
    a = rng.integers(-50, 50, size=n + off).astype(dt)
    a[rng.integers(0, n, size=20)] = info.min  # the type's extremes
    a[rng.integers(0, n, size=20)] = info.max
    for op, c in ((">", 0), ("<=", int(info.min)), (">=", int(info.max)), ("!=", 7),
                  ("<", -2**63), (">", 2**40), ("all", 0)):
        check_filter(ctx, stream, a, op, c, off)


@pytest.mark.parametrize("n,held", [(512, 512), (16384, 16383), (16385, 513), (200_001, 0),
                                    (200_001, 131_073), (3_000_011, 2_999_999)])
def test_filter_selection_edges(ctx, stream, n, held):
    rng = np.random.default_rng(n)
    a = rng.integers(0, 100, size=2 * n).astype(np.int8)
    sel = np.sort(rng.choice(2 * n, size=n, replace=False)).astype(np.int64)
    check_filter(ctx, stream, a, "<", 50, sel=sel)
    check_filter(ctx, stream, a, "<", 50, sel=sel, d_n=held)


def test_filter_without_room_for_its_bits(stream):
    """9M rows keep 1.1 MB of predicate bits; the arena is the smallest allowed."""
    small = pq.Context(arena_bytes=1 << 20)
    a = np.random.default_rng(5).integers(0, 100, size=9_000_001).astype(np.int32)
    check_filter(small, stream, a, "<", 37)
    small.close()


def check_groupby(ctx, stream, k, v, cap=None, off=0):
    want = oracle.groupby_sum(k[off:], v[off:])
    cap = len(want[0]) if cap is None else cap
    x, y = dev(k)[off:], dev(v)[off:]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ok, os_, ng = pq.pq_groupby_sum(ctx, x, y, cap=cap, stream=stream)
        ctx.sync(stream)
    g = int(ng.item())
    assert g == len(want[0])
    gk, gs = ok[:g].cpu().numpy(), os_[:g].cpu().numpy()
    order, worder = np.argsort(gk), np.argsort(want[0])
    assert np.array_equal(gk[order], want[0][worder])
    assert np.array_equal(gs[order], want[1][worder])


N_GB = 1 << 20  # from here on the key order is looked at


def runs_of(rng, n, longest):
    """Ascending keys (with gaps) in runs of 1..longest rows."""
    m = min(n, 4 * n // (longest + 1) + 64)  # runs enough for n rows
    reps = rng.integers(1, longest + 1, size=m)
    reps[-1] += max(0, n - int(reps.sum()))
    keys = np.cumsum(rng.integers(1, 9, size=m))
    return np.repeat(keys, reps)[:n].astype(np.int64)


@pytest.mark.parametrize("longest", [1, 7, 300, 200_000])
@pytest.mark.parametrize("n", [N_GB - 1, N_GB, N_GB + 1, 3_000_017])
@pytest.mark.parametrize("off", [0, 1])
def test_groupby_in_key_order(ctx, stream, longest, n, off):
    """Runs that end at, span and cross the shares of the warps."""
    rng = np.random.default_rng(n + longest)
    k = runs_of(rng, n, longest) - 1000
    check_groupby(ctx, stream, k, rng.integers(-10**12, 10**12, size=n), off=off)


@pytest.mark.parametrize("kt,vt", [(np.int32, np.int8), (np.int8, np.int32), (np.int32, np.int64)])
def test_groupby_in_key_order_types(ctx, stream, kt, vt):
    rng = np.random.default_rng(2)
    n = N_GB + 777
    k = np.sort(rng.integers(-100, 100, size=n)).astype(kt) if kt == np.int8 else \
        runs_of(rng, n, 5).astype(kt)
    v = rng.integers(np.iinfo(vt).min // 2, np.iinfo(vt).max // 2, size=n).astype(vt)
    check_groupby(ctx, stream, k, (v >> 20).astype(vt) if vt == np.int64 else v)


# A late part after one descent: rows of groups seen before and of new ones.
@pytest.mark.parametrize("tail", [1, 129, 100_000, 700_000])
@pytest.mark.parametrize("new", [False, True])
def test_groupby_with_a_late_part(ctx, stream, tail, new):
    rng = np.random.default_rng(tail)
    n = 2 * N_GB
    k = runs_of(rng, n, 4)
    k[n - tail:] = np.sort(rng.integers(0, k[n - tail - 1] + (1000 if new else 0), size=tail))
    k[n - tail] = 0 if new else k[0]  # the descent
    check_groupby(ctx, stream, k, rng.integers(0, 10**9, size=n))


@pytest.mark.parametrize("kind", ["all-equal", "two-descents", "reversed", "zipf", "zipf-sparse",
                                  "uniform-sparse", "cancelling", "wrapping"])
def test_groupby_other_orders(ctx, stream, kind):
    rng = np.random.default_rng(17)
    n = N_GB + 4321
    v = rng.integers(-10**9, 10**9, size=n)
    k = runs_of(rng, n, 4)
    if kind == "all-equal":
        k[:] = -5
    elif kind == "two-descents":
        k = np.concatenate([k[:n // 3], k[:n // 3], k[:n - 2 * (n // 3)]])
    elif kind == "reversed":
        k = k[::-1].copy()
    elif kind.startswith("zipf"):
        k = np.exp(rng.random(n) * np.log(200_000)).astype(np.int64) * 7919 % 200_003
        k = k * 1000 - 10**7 if kind == "zipf-sparse" else k
    elif kind == "uniform-sparse":
        k = rng.integers(-2**62, 2**62, size=n // 4)[rng.integers(0, n // 4, size=n)]
    elif kind == "cancelling":  # sums of exactly 0 are groups too
        k = np.repeat(np.arange(n // 2 + 1), 2)[:n]
        v = np.where(np.arange(n) % 2 == 0, 7, -7)
    elif kind == "wrapping":  # frequent group whose low words carry often
        k = np.where(rng.random(n) < 0.7, 3, k)
        v = rng.integers(2**31, 2**40, size=n) * rng.choice([-1, 1], size=n)
    check_groupby(ctx, stream, k, v)


@pytest.mark.parametrize("order", ["runs", "late", "zipf"])
def test_groupby_capacity_is_counted(ctx, stream, order):
    rng = np.random.default_rng(3)
    n = N_GB + 5
    k = runs_of(rng, n, 4)
    if order == "late":
        k[-1000:] = np.arange(1000) * 3
    elif order == "zipf":
        k = np.exp(rng.random(n) * np.log(100_000)).astype(np.int64)
    groups = len(np.unique(k))
    with torch.cuda.stream(stream):
        ok, os_, ng = pq.pq_groupby_sum(ctx, dev(k), dev(k), cap=groups - 7, stream=stream)
        with pytest.raises(pq.PQError) as e:
            ctx.sync(stream)
    assert e.value.status == pq.PQ_ERR_CAPACITY and int(ng.item()) == groups


@pytest.mark.parametrize("cap", [1, 1000, "half", "less one", "groups", "more"])
def test_groupby_unordered_range_above_the_table(ctx, stream, cap):
    """Keys in no order over a range of 4 keys per row: a hash table sized for
    cap groups, whose place the slot array takes when there are more."""
    rng = np.random.default_rng(23)
    n = N_GB + 77
    k = rng.integers(0, n // 8, size=n) * 32 - 5_000_000
    v = rng.integers(-10**9, 10**9, size=n)
    wk, ws, _ = oracle.groupby_sum(k, v)
    groups = len(wk)
    cap = {"half": groups // 2, "less one": groups - 1, "groups": groups,
           "more": groups + 100}.get(cap, cap)
    with torch.cuda.stream(stream):
        ok, os_, ng = pq.pq_groupby_sum(ctx, dev(k), dev(v), cap=cap, stream=stream)
        if cap < groups:
            with pytest.raises(pq.PQError) as e:
                ctx.sync(stream)
            assert e.value.status == pq.PQ_ERR_CAPACITY
        else:
            ctx.sync(stream)
    assert int(ng.item()) == groups
    m = min(cap, groups)
    gk, gs = ok[:m].cpu().numpy(), os_[:m].cpu().numpy()
    at = np.searchsorted(wk, gk)
    assert len(np.unique(gk)) == m
    assert np.array_equal(wk[at], gk) and np.array_equal(ws[at], gs)


def test_groupby_reserved_key_in_order(ctx, stream):
    k = np.sort(np.random.default_rng(1).integers(-50, 50, size=N_GB))
    k[0] = np.iinfo(np.int64).min
    with torch.cuda.stream(stream):
        ok, os_, ng = pq.pq_groupby_sum(ctx, dev(k), dev(k), cap=1000, stream=stream)
        with pytest.raises(pq.PQError) as e:
            ctx.sync(stream)
    assert e.value.status == pq.PQ_ERR_RESERVED_KEY
    assert int(ng.item()) == len(np.unique(k)) - 1


# Blocks with 8 pairs and more per thread read the sums first.
@pytest.mark.parametrize("n", [2047, 2048, 2049, 700_001, 2_500_000])
@pytest.mark.parametrize("kind", ["random", "equal", "few", "ascending"])
def test_topk_sums_first(ctx, stream, n, kind):
    rng = np.random.default_rng(n)
    keys = rng.permutation(n).astype(np.int64) - n // 2
    sums = {"random": rng.integers(-2**62, 2**62, size=n), "equal": np.full(n, -3),
            "few": rng.integers(0, 5, size=n), "ascending": np.arange(n) * 3}[kind].astype(np.int64)
    for k in (1, 10, 32, 33):
        with torch.cuda.stream(stream):
            ok, os_, nout = pq.pq_topk(ctx, dev(keys), dev(sums), k, stream=stream)
            ctx.sync(stream)
        wk, ws = oracle.topk(keys, sums, k)
        assert int(nout.item()) == len(wk)
        assert np.array_equal(ok[:len(wk)].cpu().numpy(), wk)
        assert np.array_equal(os_[:len(wk)].cpu().numpy(), ws)


N_HT = 1 << 18  # build keys from which lines of the table may follow the key order


def join_keys(rng, kind, n):
    i = np.arange(n, dtype=np.int64)
    if kind == "gap4":
        return 4 * i + rng.integers(0, 4, size=n) - 2 * n
    if kind == "gap1000":
        return 1000 * i + rng.integers(0, 1000, size=n)
    if kind == "dense":
        return i - n // 3
    if kind == "two-scales":    # regions of dense ids
        return (i // 500 << 40) + i % 500
    if kind == "dense-groups":  # even in the large, crowded in the small
        return (i // 64) * 256 + i % 64
    if kind == "outliers":      # dense ids and a few keys far away
        k = i.copy()
        k[::1000] = rng.integers(-2**62, 2**62, size=len(k[::1000]))
        return k
    if kind == "half-sparse":   # the sample's spacing fits neither half
        return np.where(i < n // 2, i, i * 5000)
    if kind == "random":
        return rng.integers(-2**62, 2**62, size=n)
    if kind == "equal-low-bits":
        return i << 34
    if kind == "repeated":      # lines fill up with copies of a key
        return np.repeat(4 * np.arange(n // 5 + 1), 5)[:n]
    if kind == "few-repeated-much":
        return np.where(rng.random(n) < 0.001, 4 * 77, 4 * i)
    raise ValueError(kind)


@pytest.mark.parametrize("n", [N_HT - 1, N_HT, N_HT + 12_345])
@pytest.mark.parametrize("kind", ["gap4", "gap1000", "dense", "two-scales", "dense-groups", "outliers",
                                  "half-sparse", "random", "equal-low-bits", "repeated",
                                  "few-repeated-much"])
def test_join_key_order(ctx, stream, n, kind):
    rng = np.random.default_rng(n)
    build = join_keys(rng, kind, n)
    if kind in ("dense", "random"):
        rng.shuffle(build)
    vals = rng.integers(-10**12, 10**12, size=n)
    probe = np.concatenate([build[rng.integers(0, n, size=20_011)],
                            build[:500] + 1, build[-500:] - 1, np.array([0, 2**62, -2**62])])
    wr, wv = oracle.join(build, probe, vals)
    with torch.cuda.stream(stream):
        ht = pq.pq_join_build(ctx, dev(build), dev(vals), stream=stream)
        rows, got, cnt = pq.pq_join_probe(ctx, ht, dev(probe), cap=len(wr) + 5, stream=stream)
        ht.free(stream)
        ctx.sync(stream)
    c = int(cnt.item())
    assert c == len(wr)
    rows, got = rows[:c].cpu().numpy(), got[:c].cpu().numpy()
    order, worder = np.lexsort((got, rows)), np.lexsort((wv, wr))
    assert np.array_equal(rows[order], wr[worder]) and np.array_equal(got[order], wv[worder])


def test_join_key_order_int32_row_ids(ctx, stream):
    rng = np.random.default_rng(4)
    n = N_HT + 3
    build = (rng.permutation(n) * 3 - n).astype(np.int32)
    probe = np.arange(-n, 2 * n, dtype=np.int32)
    wr, wv = oracle.join(build, probe)
    with torch.cuda.stream(stream):
        ht = pq.pq_join_build(ctx, dev(build), None, load_factor=0.9, stream=stream)
        rows, got, cnt = pq.pq_join_probe(ctx, ht, dev(probe), cap=len(wr), stream=stream)
        ht.free(stream)
        ctx.sync(stream)
    assert int(cnt.item()) == len(wr)
    order = np.argsort(rows.cpu().numpy())
    assert np.array_equal(rows.cpu().numpy()[order], wr)
    assert np.array_equal(got.cpu().numpy()[order], wv)


def check_partition(ctx, stream, key, pays, log2P, off=0):
    want_k, want_p, want_o = oracle.partition(key[off:], log2P, [p[off:] for p in pays])
    k, ps = dev(key)[off:], [dev(p)[off:] for p in pays]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        gk, gp, go = pq.pq_partition(ctx, k, ps, log2P=log2P, stream=stream)
        ctx.sync(stream)
    assert np.array_equal(go.cpu().numpy(), want_o)
    assert np.array_equal(gk.cpu().numpy(), want_k)
    for g, w in zip(gp, want_p):
        assert np.array_equal(g.cpu().numpy(), w)


def rows_for(rng, n, kt, pay, dist):
    hi = 2**31 - 1 if kt == np.int32 else 2**62
    key = rng.integers(-hi, hi, size=n) if dist == "uniform" else \
        np.where(rng.random(n) < 0.8, 12345, rng.integers(0, 5000, size=n))
    return key.astype(kt), [rng.integers(-100, 100, size=n).astype(t) for t in pay]


# Two passes by half the bucket number each: 1024 buckets from 320 MiB on,
# 2048 from 48 MiB, 4096 from 16 MiB; one pass below.
@pytest.mark.parametrize("log2P,n,kt,pay", [
    (10, 16_000_001, np.int64, (np.int64, np.int8, np.int32)),
    (10, 1_000_003, np.int64, (np.int64, np.int8, np.int32)),
    (11, 6_291_455, np.int32, (np.int32,)), (11, 6_291_456, np.int32, (np.int32,)),
    (12, 2_097_151, np.int64, ()), (12, 2_097_152, np.int64, ()),
    (12, 1_300_001, np.int64, (np.int8, np.int32, np.int8)),
    (8, 1_000_003, np.int32, (np.int32,)), (8, 1_000_003, np.int64, (np.int8,))])
@pytest.mark.parametrize("dist", ["uniform", "skewed"])
def test_partition_passes(ctx, stream, log2P, n, kt, pay, dist):
    check_partition(ctx, stream, *rows_for(np.random.default_rng(n), n, kt, pay, dist), log2P)


@pytest.mark.parametrize("log2P", [11, 12])
def test_partition_two_passes_unaligned(ctx, stream, log2P):
    key, pays = rows_for(np.random.default_rng(2), 5_000_001, np.int64, (np.int32, np.int8), "uniform")
    check_partition(ctx, stream, key, pays, log2P, off=1)


def test_partition_without_room_for_a_second_copy(stream):
    """40 MB of rows by 4096 buckets; the arena holds the counts, not the rows."""
    small = pq.Context(arena_bytes=32 << 20)
    key, pays = rows_for(np.random.default_rng(3), 2_500_000, np.int64, (np.int64,), "uniform")
    check_partition(small, stream, key, pays, 12)
    small.close()
