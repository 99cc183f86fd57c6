"""A step whose per-session counts disagree with the table rows -- as when a commit on another
stream falls between the two reads -- is refused whole where a row holds fewer blocks than
were counted, and takes the counted ones where it holds more.  The counts are changed by
hand.  Sessions taken by maximum and by the threshold, lists in shared memory and beyond."""
import numpy as np
import pytest

from ._pool_words import pool_words

pytestmark = pytest.mark.gpu

# sessions, blocks of each, victims: one or two sessions, several, by the threshold (compared
# with one another, and sorted), lists past what shared memory holds
SIZES = [(4, 40, 50), (4, 40, 100), (300, 9, 200), (700, 3, 900), (6, 1024, 2500), (40, 60, 1100)]


@pytest.mark.parametrize("call", ["evict", "turn"])
@pytest.mark.parametrize("S,blocks,k", SIZES)
def test_counts_that_disagree(S, blocks, k, call, tmp_path):
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    cap, budget, host = max(k, blocks), (S - 1) * blocks, 2 * k + 8
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, page_tokens=1, max_sessions=S, max_blocks=cap, hbm_pages=budget,
                  hbm_budget_pages=budget, host_pages=host)
    try:
        # session 0 lies on the host, the others fill the HBM pages
        table = np.full((S, cap), -1, np.int32)
        table[0, :k] = -2 - np.arange(k)
        table[1:, :blocks] = np.arange(budget).reshape(S - 1, blocks)
        ctx = np.full(S, blocks, np.int32)
        ctx[0] = k
        st = np.zeros(S, dtype=lv.SESSION_DTYPE)
        st["gen_us"] = 1000 * np.arange(S)
        pool.import_placement(table, ctx)
        pool.set_sessions(st)
        _, _, cnt = pool_words(pool, tmp_path)
        result = np.zeros(1, lv.RESIDENT_DTYPE)

        def step():
            if call == "evict":
                lv.lv_evict(pool.handle, 0, k, 0, pool.victims, pool.slots, result, pool.stream)
            else:
                outs = (pool.victims, pool.slots, pool.blks, pool.pages, pool.app)
                lv.lv_turn(pool.handle, 0, 0, 0, 0, 0, outs, result, None, 0, pool.stream)
            err = pool.sync(raise_on_error=False)
            pool.clear_error()
            return err

        before = pool.tables()
        for nth in range(1, k // blocks + 1):        # the nth session in victim order
            if nth not in (1, 2, k // blocks) or nth * blocks == k:
                continue
            cnt[S - nth, 0] += 3
            assert step() == lv.LV_ERR_STATE
            for x, y in zip(before, pool.tables()):
                assert np.array_equal(x, y)
            cnt[S - nth, 0] -= 3
        # two blocks fewer than the row holds: the others, and then the next sessions'
        cnt[S - 1, 0] -= 2
        assert step() == 0
        order = [(s, b, int(table[s, b])) for s in range(S - 1, 0, -1) for b in range(blocks - 1, -1, -1)
                 if s < S - 1 or b >= 2]
        assert int(result["n_victims"][0]) == k
        assert pool.victims[:k].cpu().numpy().tolist() == [list(v) for v in order[:k]]
        cnt[S - 1, 0] += 2
        t, own_hbm, _ = pool.tables()
        a, d = pool.counts()
        assert np.array_equal(a, (t >= 0).sum(1)) and np.array_equal(d, (t <= -2).sum(1))
        assert np.array_equal(cnt.cpu().numpy(), np.stack([a, d], 1))
        s, b = np.nonzero(t >= 0)
        assert np.array_equal(own_hbm[t[s, b]], s << 16 | b) and (own_hbm != -1).sum() == len(s)
    finally:
        pool.close()
