"""Operators whose outputs lie over their inputs (through the C functions):
the results equal those of separate arrays."""
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
    c = pq.Context(arena_bytes=2 << 30)
    yield c
    c.close()


@pytest.fixture(scope="module")
def stream():
    return torch.cuda.Stream()


# In order, in order but for a late part, in no order; groups over the keys and
# sums over the values, the two swapped, or both halfway into the values.
@pytest.mark.parametrize("order", ["sorted", "late", "random"])
@pytest.mark.parametrize("where", ["same", "swapped", "shifted"])
def test_groupby_over_its_inputs(ctx, stream, order, where):
    n, g = 3_000_017, 700_001
    rng = np.random.default_rng(5)
    k = rng.integers(0, g, size=n) * 3 - 1_000_000
    if order != "random":
        k.sort()
    if order == "late":
        k = np.roll(k, -n // 50)
    v = rng.integers(-1000, 1000, size=n)
    buf = torch.empty(2 * n, dtype=torch.int64, device="cuda")
    kt, vt = buf[:n], buf[n:]
    kt.copy_(torch.from_numpy(k))
    vt.copy_(torch.from_numpy(v))
    ok, os = {"same": (kt, vt), "swapped": (vt, kt),
              "shifted": (buf[n // 2:n // 2 + g], buf[n // 2 + g:n // 2 + 2 * g])}[where]
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    ctx.check(pq.library().pq_groupby_sum(ctx.h, pq.col(kt), pq.col(vt), ok.data_ptr(),
                                          os.data_ptr(), g, cnt.data_ptr(), stream.cuda_stream))
    ctx.sync(stream)
    uk, inv = np.unique(k, return_inverse=True)
    sums = np.zeros(len(uk), np.int64)
    np.add.at(sums, inv, v)
    m = int(cnt.item())
    assert m == len(uk)
    gk, gs = ok[:m].cpu().numpy(), os[:m].cpu().numpy()
    at = np.argsort(gk)
    assert np.array_equal(gk[at], uk) and np.array_equal(gs[at], sums)


# One block, the sizes around it, and several tiles per block.
@pytest.mark.parametrize("n", [300, 16_384, 16_385, 200_003, 4_000_001, 12_000_001])
@pytest.mark.parametrize("deferred", [False, True])
def test_filter_refines_a_selection_in_place(ctx, stream, n, deferred):
    rng = np.random.default_rng(n)
    a = rng.integers(0, 100, size=n).astype(np.int32)
    sel = np.flatnonzero(rng.random(n) < 0.9).astype(np.int64)
    buf = torch.from_numpy(np.concatenate([sel, sel[:100]])).cuda()
    x, m = torch.from_numpy(a).cuda(), len(sel)
    n_in = torch.tensor([m], device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):  # later rounds drop nothing more
        ctx.check(pq.library().pq_filter(ctx.h, pq.col(x), pq.CMP["<"], 97, buf.data_ptr(), m,
                                         n_in.data_ptr() if deferred else None, buf.data_ptr(),
                                         cnt.data_ptr(), stream.cuda_stream))
        ctx.sync(stream)
        want = sel[a[sel] < 97]
        assert int(cnt.item()) == len(want)
        assert np.array_equal(buf[:len(want)].cpu().numpy(), want)
        m = len(want)
        n_in.fill_(m)
        torch.cuda.synchronize()
