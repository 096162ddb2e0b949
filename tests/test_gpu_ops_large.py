"""Operators on more rows than 32 bits count."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402


def bucket(key, log2P):
    return ((key * 0x9E3779B97F4A7C15) % 2**64) >> (64 - log2P)


@pytest.mark.parametrize("log2P", [10, 12])
def test_partition_bucket_of_more_than_2_32_rows(log2P):
    """One key holds 2^32 rows and a few more (52 GB in all): every offset
    after its bucket lies beyond 2^32."""
    n, hot, rare = 2**32 + 4099, 5, (7, -100, 31, 90)
    key = torch.full((n,), hot, dtype=torch.int32, device="cuda")
    at = {k: 1000 * (j + 1) for j, k in enumerate(rare)}
    for k, j in at.items():
        key[j * 10:j * 10 + j] = k
    count = {**at, hot: n - sum(at.values())}
    assert len({bucket(k, log2P) for k in count}) == len(count)
    ctx, s = pq.Context(arena_bytes=17 << 30), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        out, _, off = pq.pq_partition(ctx, key, log2P=log2P, stream=s)
        ctx.sync(s)
    want, got = [0] * ((1 << log2P) + 1), off.tolist()
    for k, c in count.items():
        want[bucket(k, log2P) + 1] = c
    for b in range(1 << log2P):
        want[b + 1] += want[b]
    assert got == want
    for k in count:
        b = bucket(k, log2P)
        assert bool((out[want[b]:want[b + 1]] == k).all())
    ctx.close()
