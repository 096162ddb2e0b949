"""A streamed plan over packed columns in an arena that has room for its tables
but not for the columns' block entries as well."""
import pytest

import datagen
from gpu_util import assert_same, oracle_plan

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02862_gb300 as pq  # noqa: E402

COLS = (("key", "seg"), ("key", "dref", "date"), ("mkey", "price", "disc", "date2"))


@pytest.mark.parametrize("batch", [1, 3])
def test_block_entries_make_room_for_the_tables(batch):
    tabs = datagen.make(50_000, 500_000, 2_000_000, seed=4)
    want = oracle_plan(*tabs, d_op="all", m_op="all", f_op="all")
    s = torch.cuda.Stream()

    def run(arena):
        ctx = pq.Context(arena_bytes=arena, chunk_bytes=1 << 20)
        T = [pq.pq_load_columns(ctx, [pq.pq_pack_column(torch.from_numpy(t[c])) for c in names],
                                mode=pq.PQ_STREAMING, stream=s)
             for t, names in zip(tabs, COLS)]
        plan = pq.make_plan(*T, d_op="all", m_op="all", f_op="all")
        if batch == 1:
            res = [pq.pq_run_plan(ctx, plan, stream=s)]
        else:
            res = pq.pinned_results(batch)
            pq.pq_run_batch(ctx, [plan] * batch, res, stream=s)
        ctx.sync(s)
        for i in range(batch):
            assert_same(res[i].as_dict(), want, arena)
        high = ctx.stats()["arena_high_water"]
        for t in T:
            t.free(s)
        ctx.sync(s)
        ctx.close()
        return high

    # 16 bytes per 4096 rows and column, in pieces of 256.
    entries = sum(len(names) * -(-16 * -(-len(t[names[0]]) // 4096) // 256) * 256
                  for t, names in zip(tabs, COLS))
    high = run(512 << 20)
    run(high - entries)
