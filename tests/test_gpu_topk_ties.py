"""The top-k operator on sums that tie: the keys decide, in blocks with and
without a first threshold."""
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
    c = pq.Context(arena_bytes=256 << 20)
    yield c
    c.close()


# Blocks of one pair, at and over 2048 pairs, at and over 16 pairs per thread.
@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 4096, 100_003, 1_300_000, 6_000_007])
@pytest.mark.parametrize("k", [1, 10, 32])
@pytest.mark.parametrize("sums", ["equal", "ten", "top-few", "lowest"])
@pytest.mark.parametrize("keys", ["up", "down", "random", "extreme"])
def test_ties(ctx, n, k, sums, keys):
    rng = np.random.default_rng(n + k)
    s = {"equal": lambda: np.full(n, 7), "ten": lambda: rng.integers(-5, 5, size=n),
         "top-few": lambda: np.where(rng.random(n) < 1e-4, 2**40, rng.integers(0, 1000, size=n)),
         "lowest": lambda: np.full(n, -2**63)}[sums]().astype(np.int64)
    x = {"up": lambda: np.arange(n), "down": lambda: np.arange(n)[::-1] - 5,
         "random": lambda: rng.permutation(n) * 3 - n,
         "extreme": lambda: np.where(np.arange(n) == n // 2, -2**62,
                                     2**63 - 1 - rng.permutation(n))}[keys]().astype(np.int64)
    stream = torch.cuda.Stream()
    dk, ds = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, s))
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        gk, gs, cnt = pq.pq_topk(ctx, dk, ds, k, stream=stream)
        ctx.sync(stream)
    m = min(k, n)
    at = np.lexsort((x, -(s.astype(np.float64))))[:m] if n < 10**6 else None
    if at is None:  # the pairs of the best sums, then by key
        cut = np.partition(s, n - m)[n - m]
        pool = np.flatnonzero(s >= cut)
        at = pool[np.lexsort((x[pool], -(s[pool].astype(np.float64))))][:m]
    assert int(cnt.item()) == m
    assert np.array_equal(gk[:m].cpu().numpy(), x[at])
    assert np.array_equal(gs[:m].cpu().numpy(), s[at])
