"""A free (lv_cancel) may run on another stream while a call allocates.  The call's verdict is
then one of the two that the orders of the calls would give, it ends, and the tables agree with
one another; and a count that says there is room where the bitmap has none -- as between the
two writes of a free -- allocates nothing.  Both forms of the decision kernels: bitmaps copied
to shared memory, and (large pools) changed in place."""
import numpy as np
import pytest

from ._pool_words import pool_words

pytestmark = pytest.mark.gpu
LARGE = 760_000        # pages of one tier: past what the kernels copy


def _pool(S, cap, hbm, budget, host):
    from paper_2606_22983_gb300.pool import KVPool
    return KVPool(layers=1, kv_heads=1, head_dim=8, page_tokens=1, max_sessions=S, max_blocks=cap, hbm_pages=hbm,
                  hbm_budget_pages=budget, host_pages=host)


def _states(lv, S):
    st = np.zeros(S, dtype=lv.SESSION_DTYPE)
    st["gen_us"] = 1_000_000 * np.arange(S)
    return st


@pytest.mark.parametrize("pages", [96, LARGE])
def test_full_tiers_whatever_the_counts_say(pages, tmp_path):
    import torch
    from paper_2606_22983_gb300 import lv
    S = 4 if pages < 1000 else 32
    cap = 64 if pages < 1000 else 65536
    pool = _pool(S, cap, pages, pages, pages)
    try:
        per = pages // S                         # blocks of each session in each tier
        table = np.full((S, cap), -1, np.int32)
        table[:, :per] = np.arange(S * per).reshape(S, per)
        table[:, per:2 * per] = -(np.arange(S * per).reshape(S, per) + 2)
        assert S * per == pages and 2 * per <= cap
        pool.import_placement(table, np.full(S, 2 * per, np.int32))
        pool.set_sessions(_states(lv, S))
        hbm, host, _ = pool_words(pool, tmp_path)
        before = pool.tables()
        hbm -= 3
        host -= 3
        v = torch.tensor([[3, per - 1, table[3, per - 1]], [3, per - 2, table[3, per - 2]]], dtype=torch.int32).cuda()
        b = torch.arange(per, per + 5, dtype=torch.int32).cuda()
        result = np.zeros(1, lv.RESIDENT_DTYPE)
        outs = (pool.victims, pool.slots, pool.blks, pool.pages, pool.app)
        calls = [
            (lv.LV_ERR_NO_HBM, lambda: pool.swap_in(0, b, 2)),
            (lv.LV_ERR_NO_HBM, lambda: lv.lv_session_append(pool.handle, 0, 2, pool.app, None, pool.stream)),
            (lv.LV_ERR_NO_HOST, lambda: pool.swap_out(v, 2)),
            (lv.LV_ERR_NO_HOST, lambda: pool.exchange(v, 2, 0, b, 2)),
            (lv.LV_ERR_NO_HBM, lambda: pool.exchange(None, 0, 0, b, 2)),
            (lv.LV_ERR_NO_HOST, lambda: lv.lv_evict(pool.handle, 0, 2, 0, pool.victims, pool.slots, result, pool.stream)),
            (lv.LV_ERR_NO_HOST, lambda: lv.lv_turn(pool.handle, 0, 0, 0, 0, 0, outs, result, None, 0, pool.stream)),
        ]
        for want, call in calls:
            call()
            assert pool.sync(raise_on_error=False) == want
            pool.clear_error()
            for x, y in zip(before, pool.tables()):
                assert np.array_equal(x, y)
        assert int(result["k"][0]) == per        # every block that the turn loads needs a victim
        hbm += 3
        host += 3
        st = pool.stats()
        assert (st["hbm_allocated"], st["host_allocated"]) == (pages, pages)
    finally:
        pool.close()


def _consistent(pool):
    t, own_hbm, own_host = pool.tables()
    s, b = np.nonzero(t >= 0)
    assert np.array_equal(own_hbm[t[s, b]], s << 16 | b) and (own_hbm >= 0).sum() == len(s)
    s, b = np.nonzero(t <= -2)
    assert np.array_equal(own_host[-(t[s, b] + 2)], s << 16 | b) and (own_host >= 0).sum() == len(s)
    st = pool.stats()
    assert st["hbm_allocated"] == (own_hbm != -1).sum() and st["host_allocated"] == (own_host != -1).sum()
    a, d = pool.counts()
    assert np.array_equal(a, (t >= 0).sum(1)) and np.array_equal(d, (t <= -2).sum(1))
    return t, own_hbm, own_host


@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("call", ["turn", "exchange", "swap_in", "append", "swap_out"])
def test_cancel_on_another_stream(call, large):
    import torch
    from paper_2606_22983_gb300 import lv
    S, cap, per, R = 6, 64, 20, 8
    budget = S * per - 12 + R                   # session 0 has 12 blocks on the host, session 1 eight
    host = 12 + R + (R if call == "swap_out" else 40)
    pool = _pool(S, cap, LARGE if large else budget, budget, LARGE if large else host)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        table = np.full((S, cap), -1, np.int32)
        table[:, :per] = np.arange(S * per).reshape(S, per)
        table[0, :12] = -(np.arange(12) + 2)
        table[1, :R] = -(np.arange(12, 12 + R) + 2)
        used = table[table >= 0]
        table[table >= 0] = np.arange(len(used))
        budget_used = len(used)
        ctx = np.full(S, per, np.int32)
        rng = np.random.default_rng(7)
        victims = torch.tensor([[5, per - 1 - i, int(table[5, per - 1 - i])] for i in range(R)], dtype=torch.int32).cuda()
        if call == "swap_out":                  # host slots are reserved and released instead
            spare = torch.tensor([[4, per - 1 - i, int(table[4, per - 1 - i])] for i in range(R)], dtype=torch.int32).cuda()
        blks0, blks1 = torch.arange(12, dtype=torch.int32).cuda(), torch.arange(R, dtype=torch.int32).cuda()
        free = budget - budget_used             # HBM pages: all but R are taken by then
        locs = torch.empty(R, dtype=torch.int32).cuda()
        pages, slots = torch.empty(64, dtype=torch.int32).cuda(), torch.empty(64, dtype=torch.int32).cuda()
        for rnd in range(12 if large else 60):
            pool.import_placement(table, ctx)
            pool.set_sessions(_states(lv, S))
            pool.sync()
            # the reservations that are given back while the call runs
            with torch.cuda.stream(a):
                if call == "swap_out":
                    lv.lv_swap_out(pool.handle, spare, R, slots, None, 0, a)
                    locs.copy_(-(slots[:R] + 2))
                else:
                    lv.lv_swap_in(pool.handle, 1, blks1, R, pages, None, 0, a)
                    locs.copy_(pages[:R])
            torch.cuda.synchronize()
            held = set(locs.tolist())
            result = np.zeros(1, lv.RESIDENT_DTYPE)
            with torch.cuda.stream(a):
                torch.cuda._sleep(20_000 + int(rng.integers(0, 12_000)))
            with torch.cuda.stream(b):
                torch.cuda._sleep(20_000 + int(rng.integers(0, 24_000)))
            lv.lv_cancel(pool.handle, locs, R, b)
            if call == "turn":
                outs = (pool.victims, pool.slots, pool.blks, pool.pages, pool.app)
                lv.lv_turn(pool.handle, 0, 0, 3, 0, 0, outs, result, None, 0, a)
            elif call == "exchange":
                lv.lv_swap_exchange(pool.handle, victims, 2, 0, blks0, 12, slots, pages, 0, a)
            elif call == "swap_in":
                lv.lv_swap_in(pool.handle, 0, blks0, free - R // 2, pages, None, 0, a)
            elif call == "append":
                lv.lv_session_append(pool.handle, 5, free - R // 2, pages, None, a)
            else:
                lv.lv_swap_out(pool.handle, victims, R, slots, None, 0, a)
            torch.cuda.synchronize()
            err = pool.sync(raise_on_error=False)
            pool.clear_error()
            t, own_hbm, own_host = _consistent(pool)
            if call == "turn":
                # either order of the two calls serves the turn: with fewer victims after the cancel
                assert err == 0 and int(result["status"][0]) == 0
                assert 0 <= int(result["k"][0]) <= 15 - (free - R) and (t[0, :per + 3] >= 0).all()
                continue
            assert err in (0, lv.LV_ERR_NO_HOST if call == "swap_out" else lv.LV_ERR_NO_HBM)
            if err:
                assert np.array_equal(t, table) and (own_hbm != -2).all() and (own_host != -2).all()
            elif call == "swap_in":
                got = pages[:free - R // 2].tolist()
                assert len(set(got)) == len(got) and (own_hbm[got] == -2).all()
            elif call == "swap_out" and not large:
                assert set((-(slots[:R] + 2)).tolist()) == held
    finally:
        pool.close()


def test_blocks_while_the_session_grows():
    """The blocks of a session read on one stream while it grows on another, past several times
    the reader's threads: those that it had, and any of the new ones."""
    import torch
    from paper_2606_22983_gb300 import lv
    pool = _pool(1, 4096, 4096, 4096, 1)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        pool.import_placement(np.where(np.arange(4096) < 10, np.arange(4096), -1).astype(np.int32)[None], np.array([10], np.int32))
        pool.sync()
        torch.cuda.synchronize()
        blks, count = torch.empty(4096, dtype=torch.int32).cuda(), torch.zeros(1, dtype=torch.int64).cuda()
        for rnd in range(200):
            lv.lv_session_append(pool.handle, 0, 20, None, None, a)
            lv.lv_session_blocks(pool.handle, 0, 0, blks, count, b)
            torch.cuda.synchronize()
            had, got = 10 + 20 * rnd, blks[:int(count)].cpu().numpy()
            assert np.array_equal(got[:had], np.arange(had))       # and any of the twenty new ones
            assert (np.diff(got) > 0).all() and len(got) <= had + 20 and got[-1] < had + 20
        assert pool.sync() == 0
    finally:
        pool.close()
