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


# Below and from the size on where a sample is taken; in key order, in no
# order, dense; with repeated keys; 4 or 8 bytes; a few million probes, some
# without a match.
@pytest.mark.parametrize("n", [3 * 2**18 - 1, 3 * 2**18, 1_200_007])
@pytest.mark.parametrize("kind", ["even", "even-int32", "dense", "shuffled", "repeated",
                                  "repeated-shuffled"])
def test_layouts(ctx, stream, n, kind):
    rng = np.random.default_rng(n)
    build = np.arange(n) * (1 if kind == "dense" else 5) - 1_000_000
    if kind != "dense":
        build += rng.integers(0, 5, size=n)
    if kind.startswith("repeated"):
        build[1::7] = build[::7][:len(build[1::7])]
    if kind.endswith("shuffled"):
        rng.shuffle(build)
    probe = rng.integers(build.min() - 1000, build.max() + 1000, size=3_000_001)
    probe[::2] = build[rng.integers(0, n, size=len(probe[::2]))]
    if kind.endswith("int32"):
        build, probe = build.astype(np.int32), probe.astype(np.int32)
    check_join(ctx, stream, build, rng.integers(-2**40, 2**40, size=n), probe)


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("cap", [1000, 2_999_999])
def test_small_output_at_millions_of_probes(ctx, stream, shuffled, cap):
    n = 1_100_000
    rng = np.random.default_rng(3)
    build = np.arange(n) * 4 + rng.integers(0, 4, size=n)
    probe = np.repeat(build, 3)[:3_000_000]
    if shuffled:
        rng.shuffle(build)
    check_join(ctx, stream, build, np.arange(n), probe, cap=cap)


def test_even_keys_with_strays(ctx, stream):
    """Keys far outside the sampled range, negative and positive, among even
    ones; probes that miss on both sides."""
    n = 2_000_000
    rng = np.random.default_rng(4)
    build = np.arange(n) * 8 + rng.integers(0, 8, size=n)
    at = rng.choice(np.setdiff1d(np.arange(1, n - 1), np.round(np.linspace(0, n - 1, 512))),
                    200, replace=False)
    build[at[:100]] = -2**62 - np.arange(100)
    build[at[100:]] = 2**62 + np.arange(100)
    probe = np.concatenate([build, build + 1, [-2**63 + 1, 2**63 - 1, 2**62 + 50]])
    check_join(ctx, stream, build, np.arange(n), probe)


@pytest.mark.parametrize("kind", ["even", "shuffled", "repeated"])
def test_tens_of_millions_of_probes(ctx, stream, kind):
    """Many rounds per warp: every match once, compared on the device."""
    n, m = 1_000_000, 2**25 + 77
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    build = torch.arange(n, device="cuda") * 4 + torch.randint(0, 4, (n,), generator=g, device="cuda")
    at = torch.randint(0, n, (m,), generator=g, device="cuda")
    probe = build[at]
    probe[::5] = -7
    if kind == "repeated":  # each of 1000 keys twice
        build[n - 1000:] = build[:1000]
        probe = torch.where(at >= n - 1000, torch.full_like(probe, -7), probe)
    order = torch.randperm(n, generator=g, device="cuda") if kind != "even" else torch.arange(n, device="cuda")
    copies = torch.where(probe == -7, 0, torch.where(at < 1000, 2 if kind == "repeated" else 1, 1))
    pairs = int(copies.sum())
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ht = pq.pq_join_build(ctx, build[order].contiguous(), order, stream=stream)
        r, w, cnt = pq.pq_join_probe(ctx, ht, probe, pairs, stream=stream)
        ht.free(stream)
        ctx.sync(stream)
    assert int(cnt.item()) == pairs
    assert bool((torch.bincount(r, minlength=m) == copies).all())
    assert bool((build[w] == probe[r]).all())
    # Pairs are distinct: a row's two matches are different build rows.
    assert torch.unique(r * n + w).numel() == pairs
