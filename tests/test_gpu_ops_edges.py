"""Operators at the sizes where their kernels change shape: edges of warp
tiles and blocks, the rules that choose between kernels, scratch that does
not fit.  Everything is an integer and compared for equality with the
oracle."""
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
    c = pq.Context(arena_bytes=6 << 30)
    yield c
    c.close()


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check_filter(ctx, stream, a, op, c, off=0, sel=None, d_n=None):
    x = dev(a)[off:]
    y = None if sel is None else dev(sel)
    n_dev = None if d_n is None else torch.tensor([d_n], device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        out, cnt = pq.pq_filter(ctx, x, op, c, sel_in=y, d_n_in=n_dev, stream=stream)
        ctx.sync(stream)
    want = oracle.filter(a[off:], op, c, sel if d_n is None else sel[:d_n])
    assert int(cnt.item()) == len(want)
    assert np.array_equal(out[:len(want)].cpu().numpy(), want)


# One warp tile is 512 rows, one block of the single launch 32 of them.
@pytest.mark.parametrize("dt", [np.int8, np.int32, np.int64])
@pytest.mark.parametrize("n", [511, 512, 513, 16383, 16384, 16385, 24_577, 3_000_011])
@pytest.mark.parametrize("off", [0, 1])
def test_filter_tile_edges(ctx, stream, dt, n, off):
    rng = np.random.default_rng(n + off)
    info = np.iinfo(dt)
    a = rng.integers(-50, 50, size=n + off).astype(dt)
    a[rng.integers(0, n, size=20)] = info.min  # the type's extremes
    a[rng.integers(0, n, size=20)] = info.max
    for op, c in ((">", 0), ("<=", int(info.min)), (">=", int(info.max)), ("!=", 7),
                  ("<", -2**63), (">", 2**40), ("all", 0)):
        check_filter(ctx, stream, a, op, c, off)


@pytest.mark.parametrize("n,held", [(512, 512), (16384, 16383), (16385, 513), (200_001, 0),
                                    (200_001, 131_073), (3_000_011, 2_999_999)])
def test_filter_selection_edges(ctx, stream, n, held):
    rng = np.random.default_rng(n)
    a = rng.integers(0, 100, size=2 * n).astype(np.int8)
    sel = np.sort(rng.choice(2 * n, size=n, replace=False)).astype(np.int64)
    check_filter(ctx, stream, a, "<", 50, sel=sel)
    check_filter(ctx, stream, a, "<", 50, sel=sel, d_n=held)


def test_filter_without_room_for_its_bits(stream):
    """9M rows keep 1.1 MB of predicate bits; the arena is the smallest allowed."""
    small = pq.Context(arena_bytes=1 << 20)
    a = np.random.default_rng(5).integers(0, 100, size=9_000_001).astype(np.int32)
    check_filter(small, stream, a, "<", 37)
    small.close()
