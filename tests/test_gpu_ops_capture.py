"""Operators under stream capture: what the graph writes on every replay, and
how much scratch a captured call keeps."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402


@pytest.mark.parametrize("dt", [np.int8, np.int32, np.int64])
@pytest.mark.parametrize("n", [16_385, 1_000_003, 20_000_001])
@pytest.mark.parametrize("sel,off", [(False, 0), (False, 1), (True, 0)])
def test_filter_captured(dt, n, sel, off):
    """Scratch of a capture is held for the replays: it does not grow with the
    column (one bit a row would be 2.5 MB at 20M rows)."""
    ctx, s = pq.Context(arena_bytes=64 << 20), torch.cuda.Stream()
    rng = np.random.default_rng(n)
    a = rng.integers(-50, 50, size=n + off).astype(dt)
    rows = np.flatnonzero(rng.random(n) < 0.6).astype(np.int64) if sel else None
    x = torch.from_numpy(a).cuda()[off:]
    y = torch.from_numpy(rows).cuda() if sel else None
    torch.cuda.synchronize()
    before = ctx.stats()["arena_in_use"]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        out, cnt = pq.pq_filter(ctx, x, "<", 20, sel_in=y, stream=s)
    kept = ctx.stats()["arena_in_use"] - before
    for shift in (0, 17):  # other values in the same column on the second replay
        b = np.roll(a[off:], shift)
        x.copy_(torch.from_numpy(b))
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            g.replay()
        ctx.sync(s)
        want = oracle.filter(b, "<", 20, rows)
        assert int(cnt.item()) == len(want)
        assert np.array_equal(out[:len(want)].cpu().numpy(), want)
    assert kept <= 64 << 10
    del g, out, cnt
    ctx.close()
