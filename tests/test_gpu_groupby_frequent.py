"""Group-by over unordered rows: with and without keys that come often, tables
smaller and larger than L2, more groups than the output holds, few rows.
Compared with the oracle as sets of groups."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = pq.Context(arena_bytes=4 << 30)
    yield c
    c.close()


def check(ctx, k, v, cap=None, capture=False):
    s = torch.cuda.Stream()
    dk, dv = torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda()
    order = np.argsort(k, kind="stable")
    uk, first = np.unique(k[order], return_index=True)
    want = np.add.reduceat(v[order].astype(np.int64), first)
    torch.cuda.synchronize()
    run = lambda: pq.pq_groupby_sum(ctx, dk, dv, len(uk) if cap is None else cap, stream=s)
    if capture:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
            gk, gs, cnt = run()
        with torch.cuda.stream(s):
            g.replay()
    else:
        with torch.cuda.stream(s):
            gk, gs, cnt = run()
    if cap is not None and cap < len(uk):
        with pytest.raises(pq.PQError) as e:
            ctx.sync(s)
        assert e.value.status == pq.PQ_ERR_CAPACITY and int(cnt.item()) == len(uk)
        return
    ctx.sync(s)
    assert int(cnt.item()) == len(uk)
    gk, gs = gk[:len(uk)].cpu().numpy(), gs[:len(uk)].cpu().numpy()
    at = np.argsort(gk)
    assert np.array_equal(gk[at], uk) and np.array_equal(gs[at], want)


def keys(rng, n, groups, gap, often):
    """Uniform keys; with `often` a fifth of the rows hold one of three keys."""
    k = rng.integers(0, groups, size=n) * gap - 12345
    if often:
        hot = rng.random(n) < 0.2
        k[hot] = rng.choice([-12345, 7 * gap - 12345, 2**40], size=int(hot.sum()))
    return k


@pytest.mark.parametrize("often", [False, True])
@pytest.mark.parametrize("n", [2**20 - 1, 2**20, 3_000_017])
@pytest.mark.parametrize("groups,gap", [(3, 1), (1000, 1), (1000, 64), (20_000, 100),
                                        (400_000, 1), (400_000, 10**6)])
def test_unordered(ctx, n, groups, gap, often):
    rng = np.random.default_rng(groups + n)
    k = keys(rng, n, groups, gap, often)
    if often:
        k[k == 2**40] = 11 * gap - 12345 if gap < 10**6 else 2**40
    check(ctx, k, rng.integers(-2**40, 2**40, size=n))


@pytest.mark.parametrize("often", [False, True])
@pytest.mark.parametrize("vt", [np.int8, np.int32, np.int64])
@pytest.mark.parametrize("off", [0, 1])
def test_narrow_values_and_unaligned_columns(ctx, often, vt, off):
    n = 1_500_001
    rng = np.random.default_rng(3)
    k = keys(rng, n + off, 30_000, 90, often)[off:]
    k[k == 2**40] = 5
    v = rng.integers(-100, 100, size=n + off).astype(vt)[off:]
    check(ctx, np.ascontiguousarray(k), np.ascontiguousarray(v))


@pytest.mark.parametrize("cap", [1000, 100_000])
def test_more_groups_than_the_table_holds(ctx, cap):
    """Frequent keys, a table for `cap` groups, 200000 of them in a dense range:
    the slot array takes over and counts them all."""
    n = 4_000_000
    rng = np.random.default_rng(9)
    k = rng.integers(0, 200_000, size=n) * 50
    k[rng.random(n) < 0.1] = 100
    check(ctx, k, rng.integers(0, 1000, size=n), cap=cap)


@pytest.mark.parametrize("often", [False, True])
def test_table_larger_than_l2(ctx, often):
    n = 9_000_000
    rng = np.random.default_rng(10)
    check(ctx, keys(rng, n, 9_000_000, 5000, often), rng.integers(-5, 5, size=n), cap=n)


@pytest.mark.parametrize("n", [1, 31, 1000, 300_007])
@pytest.mark.parametrize("groups", [1, 12, 5000])
def test_few_rows_captured(ctx, n, groups):
    rng = np.random.default_rng(n)
    k = rng.integers(0, groups, size=n) - 3
    check(ctx, k, rng.integers(-2**62, 2**62, size=n) // max(n, 1), capture=True)


def test_reserved_key_among_frequent_ones(ctx):
    n = 1_200_000
    rng = np.random.default_rng(2)
    k = keys(rng, n, 1000, 64, True)
    k[k == 2**40] = 0
    k[12345] = -2**63
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        pq.pq_groupby_sum(ctx, torch.from_numpy(k).cuda(), torch.from_numpy(k).cuda(), 2000,
                          stream=s)
        with pytest.raises(pq.PQError) as e:
            ctx.sync(s)
    assert e.value.status == pq.PQ_ERR_RESERVED_KEY
