"""Plans large enough for the one-pass F phase: values where that pass differs
from the hit list (zero, negative and cancelling revenues, repeated M keys with
frequent groups, checked additions, row-by-row loads), and shares of M and of
F's dates on both sides of what chooses it.  Bit-exact against the oracle."""
import numpy as np
import pytest

import datagen
import oracle
from gpu_util import assert_same, load_tables, oracle_plan, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402

ALL = dict(d_op="all", m_op="all", f_op="all")
N = 1_600_003


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = pq.Context(arena_bytes=2 << 30)
    yield c
    c.close()


def check(ctx, D, M, F, k=10, off=0, **pred):
    stream = torch.cuda.Stream()
    if off:  # columns that start off a 16-byte boundary
        dev = {c: v[off:] for c, v in
               to_dev({c: np.concatenate([v[:off], v]) for c, v in F.items()}).items()}
    else:
        dev = to_dev(F)
    with torch.cuda.stream(stream):
        TD, TM, _, keep = load_tables(pq, ctx, D, M, F, stream=stream)
        TF = pq.pq_load_columns(ctx, [dev[c] for c in ("mkey", "price", "disc", "date2")],
                                stream=stream)
        plan = pq.make_plan(TD, TM, TF, k=k, **pred)
        want = oracle_plan(D, M, F, seg=pred.get("seg", 1), mc=pred.get("m_date_lt", 1200),
                           fc=pred.get("f_date_gt", 1200), k=k,
                           **{o: pred[o] for o in ("d_op", "m_op", "f_op") if o in pred})
        for _ in range(2):  # launched as a chain, then replayed from its graph
            res = pq.pq_run_plan(ctx, plan, stream=stream)
            ctx.sync(stream)
            assert_same(res.as_dict(), want, (pred, k))
        for t in (TD, TM, TF):
            t.free(stream)
        ctx.sync(stream)


def tables(seed, fk="clustered", n_m=N // 4):
    return datagen.make(max(8, n_m // 10), n_m, N, seed=seed, fk=fk)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("fk", ["clustered", "zipf"])
@pytest.mark.parametrize("kind", ["zero", "negative", "cancel", "mixed"])
def test_groups_without_positive_sums(ctx, kind, fk, off):
    D, M, F = tables(21, fk)
    rng = np.random.default_rng(4)
    if kind == "zero":
        F["price"][F["mkey"] % 2 == 0] = 0
        F["disc"][(F["mkey"] % 2 == 1) & (rng.random(N) < 0.3)] = 100
    elif kind == "negative":
        F["price"] = -F["price"]
    elif kind == "cancel":  # groups whose revenues add up to exactly 0
        F["price"][:] = 1000
        F["disc"][:] = 90
        F["price"][np.argsort(F["mkey"], kind="stable")[1::2]] *= -1
    else:
        F["price"] = rng.integers(-(10**6), 10**6, size=N)
        F["disc"] = rng.integers(-128, 128, size=N).astype(np.int8)
    check(ctx, D, M, F, k=64, off=off, **ALL)


# With an M key held thousands of times the bound on all sums no longer holds:
# every addition is checked.
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("fk", ["clustered", "zipf", "hot"])
@pytest.mark.parametrize("dups", ["one", "third", "often"])
def test_repeated_member_keys(ctx, fk, dups, off):
    D, M, F = tables(5, "clustered" if fk == "hot" else fk)
    rng = np.random.default_rng(6)
    if dups == "one":
        M["key"][1] = M["key"][0]
    elif dups == "often":
        M["key"][:3000] = M["key"][0]
    else:
        M["key"][1::3] = M["key"][::3][:len(M["key"][1::3])]
    if fk == "hot":
        # (the oracle adds a row once per copy of its key)
        F["mkey"][rng.random(N) < (0.02 if dups == "often" else 0.9)] = M["key"][0]
    F["price"][rng.random(N) < 0.4] *= -1
    check(ctx, D, M, F, k=64, off=off, **ALL)


def test_revenues_of_a_key_held_often_that_cancel(ctx):
    """A key held by 100000 M rows, 3200 F rows of it with large revenues of
    either sign in turn: each counts 100000 times, so that 40 of one sign leave
    int64, but every 32 rows in a row nearly cancel."""
    D, M, F = tables(7)
    M["key"][:100_000] = M["key"][0]
    F["mkey"][:3200] = M["key"][0]
    F["disc"][:3200] = 0
    F["price"][0:3200:2] = 24 * 10**9
    F["price"][1:3200:2] = -24 * 10**9 + 5
    check(ctx, D, M, F, **ALL)


@pytest.mark.parametrize("price", [2**40, 2**43])
def test_bound_that_does_not_hold(ctx, price):
    """Distinct M keys, but all rows times the largest price leave int64."""
    D, M, F = tables(6)
    F["price"][:] = price - np.arange(N)
    check(ctx, D, M, F, k=64, **ALL)


@pytest.mark.parametrize("price", [2**56, 24 * 10**9])
def test_overflow_of_a_repeated_key_is_reported(ctx, price):
    D, M, F = tables(2)
    M["key"][:100_000] = M["key"][0]
    F["mkey"][:64] = M["key"][0]
    F["price"][:64] = price
    F["disc"][:64] = 0
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        TD, TM, TF, keep = load_tables(pq, ctx, D, M, F, stream=stream)
        res = pq.pq_run_plan(ctx, pq.make_plan(TD, TM, TF, **ALL), stream=stream)
        assert res.status == pq.PQ_ERR_OVERFLOW
        with pytest.raises(pq.PQError):
            ctx.sync(stream)
    assert oracle.run_plan(D, M, F, k=10, **ALL)["status"] == pq.PQ_ERR_OVERFLOW


@pytest.mark.parametrize("fk", ["clustered", "zipf"])
@pytest.mark.parametrize("m_cut", [250, 320, 1200, 2406])
@pytest.mark.parametrize("f_cut", [-1, 300, 1200, 2300, 3000])
def test_shares_of_members_and_dates(ctx, fk, m_cut, f_cut):
    D, M, F = tables(9, fk)
    F["date2"] = np.random.default_rng(1).integers(0, 2406, size=N).astype(np.int32)
    check(ctx, D, M, F, d_op="all", m_date_lt=m_cut, f_date_gt=f_cut)
