"""Plans whose F rows mostly join (the one-pass F phase): bit-exact against the
oracle at the sizes and values where that pass changes shape -- step tails,
unaligned columns, row ranges, groups whose revenues are zero, negative or
cancel, repeated M keys, sums that need checked additions, hot groups -- and
on both sides of the member share that chooses it."""
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


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = pq.Context(arena_bytes=2 << 30)
    yield c
    c.close()


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


def check(ctx, stream, D, M, F, k=10, rows=None, off=0, hits=None, **pred):
    if off:  # columns that start off a 16-byte boundary
        pad = {c: np.concatenate([v[:off], v]) for c, v in F.items()}
        dev = {c: v[off:] for c, v in to_dev(pad).items()}
    else:
        dev = to_dev(F)
    with torch.cuda.stream(stream):
        TD, TM, _, keep = load_tables(pq, ctx, D, M, F, stream=stream)
        TF = pq.pq_load_columns(ctx, [dev[c] for c in ("mkey", "price", "disc", "date2")],
                                stream=stream)
        plan = pq.make_plan(TD, TM, TF, k=k, rows=rows, **pred)
        for _ in range(2):  # launched as a chain, then replayed from its graph
            res = pq.pq_run_plan(ctx, plan, stream=stream)
            ctx.sync(stream)
            want = oracle_plan(D, M, F, seg=pred.get("seg", 1), mc=pred.get("m_date_lt", 1200),
                               fc=pred.get("f_date_gt", 1200), k=k, rows=rows,
                               **{o: pred[o] for o in ("d_op", "m_op", "f_op") if o in pred})
            assert_same(res.as_dict(), want, (pred, k))
            if hits is not None:
                assert res.hits == hits
        for t in (TD, TM, TF):
            t.free(stream)
        ctx.sync(stream)


def tables(n_m, n_f, seed, fk="clustered"):
    return datagen.make(max(8, n_m // 10), n_m, n_f, seed=seed, fk=fk)


@pytest.mark.parametrize("n_f", [1, 3, 127, 128, 129, 1000, 100_003, 1_000_001])
@pytest.mark.parametrize("off", [0, 1])
def test_pass_all_sizes(ctx, stream, n_f, off):
    D, M, F = tables(max(4, n_f // 4), n_f, seed=n_f)
    check(ctx, stream, D, M, F, off=off, hits=n_f, **ALL)


@pytest.mark.parametrize("k", [1, 32, 33, 64])
@pytest.mark.parametrize("fk", ["clustered", "zipf"])
def test_skewed_and_clustered_keys(ctx, stream, k, fk):
    D, M, F = tables(200_000, 2_000_003, seed=3, fk=fk)
    check(ctx, stream, D, M, F, k=k, hits=2_000_003, **ALL)
    check(ctx, stream, D, M, F, k=k, d_op="all", m_op="all", f_date_gt=2000)
    check(ctx, stream, D, M, F, k=k, rows=dict(m=(1024, 150_000), f=(16, 1_500_001)), **ALL)


# M' from almost nothing to everything: both sides of the share of M rows
# from which F is scanned and aggregated in one pass.
@pytest.mark.parametrize("cut", [20, 250, 299, 302, 360, 1200, 3000])
def test_member_share(ctx, stream, cut):
    D, M, F = tables(100_000, 400_000, seed=9)
    check(ctx, stream, D, M, F, d_op="all", m_date_lt=cut, f_op="all")


@pytest.mark.parametrize("kind", ["zero", "negative", "cancel", "mixed"])
def test_groups_without_positive_sums(ctx, stream, kind):
    D, M, F = tables(5000, 60_000, seed=21)
    rng = np.random.default_rng(4)
    if kind == "zero":  # rows of revenue 0 only, in half the groups
        F["price"][F["mkey"] % 2 == 0] = 0
        F["disc"][(F["mkey"] % 2 == 1) & (rng.random(60_000) < 0.3)] = 100
    elif kind == "negative":
        F["price"] = -F["price"]
    elif kind == "cancel":  # groups whose revenues add up to exactly 0
        F["price"][:] = 1000
        F["disc"][:] = 90
        order = np.argsort(F["mkey"], kind="stable")
        F["price"][order[1::2]] *= -1
    else:
        F["price"] = rng.integers(-(10**6), 10**6, size=60_000)
        F["disc"] = rng.integers(-128, 128, size=60_000).astype(np.int8)
    check(ctx, stream, D, M, F, k=64, hits=60_000, **ALL)


def test_repeated_member_keys(ctx, stream):
    D, M, F = tables(20_000, 100_000, seed=5)
    M["key"][1::3] = M["key"][::3][:len(M["key"][1::3])]
    check(ctx, stream, D, M, F, **ALL)


@pytest.mark.parametrize("price,k", [(2**45, 10), (2**50, 64)])
def test_checked_additions(ctx, stream, price, k):
    """Rows times the largest price no longer stay below 2^63 together, but
    each group's sum does."""
    D, M, F = tables(50_000, 200_000, seed=6)
    F["price"][:] = price - np.arange(200_000)
    check(ctx, stream, D, M, F, k=k, hits=200_000, **ALL)


def test_one_hot_group(ctx, stream):
    D, M, F = tables(1000, 500_000, seed=8)
    F["mkey"][np.random.default_rng(1).random(500_000) < 0.9] = M["key"][17]
    check(ctx, stream, D, M, F, hits=500_000, **ALL)


def test_overflow_in_one_pass_is_reported(ctx, stream):
    D, M, F = tables(1000, 4000, seed=2)
    F["price"][:] = 2**56
    F["disc"][:] = 0
    with torch.cuda.stream(stream):
        TD, TM, TF, keep = load_tables(pq, ctx, D, M, F, stream=stream)
        res = pq.pq_run_plan(ctx, pq.make_plan(TD, TM, TF, **ALL), stream=stream)
        assert res.status == pq.PQ_ERR_OVERFLOW
        with pytest.raises(pq.PQError):
            ctx.sync(stream)
    assert oracle.run_plan(D, M, F, k=10, **ALL)["status"] == pq.PQ_ERR_OVERFLOW
