"""The radix partition over row widths and bucket counts: every sub-tile size
and launch bound of its scatter kernel, more sub-tiles than resident blocks."""
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
    c = pq.Context(arena_bytes=1 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("log2P", [0, 6, 7, 8, 9])
@pytest.mark.parametrize("kt,pay", [("i4", ""), ("i4", "i4"), ("i4", "i1,i4"), ("i8", "i8"),
                                    ("i8", "i8,i1,i4"), ("i8", "i8,i8,i8")])
@pytest.mark.parametrize("off", [0, 1])
def test_row_widths(ctx, log2P, kt, pay, off):
    n, s = 2_500_007, torch.cuda.Stream()
    rng = np.random.default_rng(log2P)
    draw = lambda t: rng.integers(np.iinfo(t).min, np.iinfo(t).max, size=n + off).astype(t)[off:]
    key, cols = draw(kt), [draw(t) for t in pay.split(",") if t]
    # off: columns that start off a 16-byte boundary take no bulk copies.
    dev = lambda a: torch.from_numpy(np.concatenate([a[:off], a])).cuda()[off:]
    k, c = dev(key), [dev(a) for a in cols]
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        ok, oc, o = pq.pq_partition(ctx, k, c, log2P=log2P, stream=s)
        ctx.sync(s)
    wk, wc, wo = oracle.partition(key, log2P, cols)
    assert np.array_equal(o.cpu().numpy(), wo)
    assert np.array_equal(ok.cpu().numpy(), wk)
    for a, b in zip(oc, wc):
        assert np.array_equal(a.cpu().numpy(), b)


def test_threads_with_different_shapes():
    """Two threads, each with a context of its own, partition rows of different
    widths and bucket counts with the same kernel."""
    import threading

    n, errors = 300_007, []

    def work(seed, log2P, wide):
        try:
            rng = np.random.default_rng(seed)
            key = rng.integers(-2**40, 2**40, size=n)
            cols = [rng.integers(0, 100, size=n) for _ in range(3 if wide else 1)]
            ctx, s = pq.Context(arena_bytes=256 << 20), torch.cuda.Stream()
            with torch.cuda.stream(s):
                k, c = torch.from_numpy(key).cuda(), [torch.from_numpy(a).cuda() for a in cols]
                for _ in range(200):
                    ok, _, o = pq.pq_partition(ctx, k, c, log2P=log2P, stream=s)
                ctx.sync(s)
            wk, _, wo = oracle.partition(key, log2P, cols)
            assert np.array_equal(o.cpu().numpy(), wo) and np.array_equal(ok.cpu().numpy(), wk)
            ctx.close()
        except Exception as e:  # seen by the test's thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in ((1, 7, True), (2, 3, False))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
