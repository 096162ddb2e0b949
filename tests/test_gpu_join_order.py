"""The join's table over build keys whose order and spread choose its layout:
in key order (an even sample), crowded in one part, hashed, on both sides of
the size from which a sample is taken."""
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
    c = pq.Context(arena_bytes=2 << 30)
    yield c
    c.close()


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


def check_join(ctx, stream, build, vals, probe, cap=None, load_factor=0.0):
    """Every (probe row, build value) pair once, in any order."""
    at = np.argsort(build, kind="stable")
    lo = np.searchsorted(build[at], probe, "left")
    n = np.searchsorted(build[at], probe, "right") - lo
    rows = np.repeat(np.arange(len(probe)), n)
    first = np.repeat(np.cumsum(n) - n, n)
    want = vals[at][np.repeat(lo, n) + np.arange(len(rows)) - first]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    b, v, p = dev(build), dev(vals), dev(probe)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ht = pq.pq_join_build(ctx, b, v, load_factor=load_factor, stream=stream)
        r, w, cnt = pq.pq_join_probe(ctx, ht, p, len(rows) if cap is None else cap, stream=stream)
        ht.free(stream)
    if cap is not None and cap < len(rows):
        with pytest.raises(pq.PQError) as e:
            ctx.sync(stream)
        assert e.value.status == pq.PQ_ERR_CAPACITY and int(cnt.item()) == len(rows)
        return
    ctx.sync(stream)
    assert int(cnt.item()) == len(rows)
    r, w = r[:len(rows)].cpu().numpy(), w[:len(rows)].cpu().numpy()
    got, exp = np.lexsort((w, r)), np.lexsort((want, rows))
    assert np.array_equal(r[got], rows[exp]) and np.array_equal(w[got], want[exp])


def crowded(n, gap=40):
    """n ascending keys, the first quarter of them in a twelfth of the range:
    no 512th of the range holds more than three keys of a sample of 512, and
    the crowd has more keys than its part of the table has slots."""
    a, width = n // 4, n * gap // 12
    return np.concatenate([np.arange(a) * width // a,
                           width + np.arange(n - a) * (n * gap - width) // (n - a)])


@pytest.mark.parametrize("load_factor", [0.0, 0.9])
def test_keys_crowded_in_one_part(ctx, stream, load_factor):
    n = 2_000_000
    build = crowded(n)
    rng = np.random.default_rng(1)
    vals = rng.integers(0, 2**40, size=n)
    probe = np.concatenate([build[rng.integers(0, n, size=1_000_000)],
                            rng.integers(-100, n * 40 + 100, size=1_000_000)])
    check_join(ctx, stream, build, vals, probe, load_factor=load_factor)
