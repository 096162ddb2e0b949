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
