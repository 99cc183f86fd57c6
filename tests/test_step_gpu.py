"""The one-CTA decisions at the edges of their lists: sessions taken by repeated maximum and by
the sort, victim and load lists that fit in shared memory and that do not, loads ordered in
the step and by the grid-wide kernel.  The host's model of a turn is plain numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
T = 16


def _order(states, resident, now):
    """Every resident block in victim order: (T_next descending, session, block descending)."""
    t = np.maximum(states["gen_us"] - states["play_us"], 0) + 3_000_000
    out = []
    for s in sorted(range(len(states)), key=lambda s: (-int(t[s]), s)):
        out += [(s, b, resident[s][b]) for b in sorted(resident[s], reverse=True)]
    return out


# sessions, blocks of each, host blocks of the turn's session, scattered order, table capacity
SIZES = [(2, 3, 1, False, 4), (5, 40, 33, True, 64), (9, 64, 64, True, 64), (40, 7, 7, False, 8),
         (70, 2, 2, True, 32), (300, 9, 9, False, 16), (12, 1023, 1023, True, 1024), (12, 1024, 1024, True, 1024),
         (12, 1025, 1025, True, 2048), (12, 1025, 1025, False, 2048), (40, 200, 200, False, 256),
         (1500, 3, 3, False, 4), (4096, 2, 2, True, 2)]


@pytest.mark.parametrize("S,blocks,away,scatter,cap", SIZES)
@pytest.mark.parametrize("grow", [0, 40])
def test_turn_decisions(S, blocks, away, scatter, cap, grow):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    if grow and blocks + 4 > cap:
        grow = 0
    rng = np.random.default_rng(S * 7 + blocks + grow)
    n = np.full(S, blocks)
    sid = int(rng.integers(0, S))
    total = int(n.sum())
    budget = total - away
    host = 2 * away + 64
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=S, max_blocks=cap, hbm_pages=budget,
                  hbm_budget_pages=budget, host_pages=host)
    try:
        table = np.full((S, cap), -1, np.int32)
        pages, slots = rng.permutation(budget), rng.permutation(host)[:away]
        p = 0
        for s in range(S):
            k = blocks - (away if s == sid else 0)
            table[s, :k] = pages[p:p + k]
            p += k
        table[sid, blocks - away:blocks] = -(slots + 2)
        ctx = np.full(S, blocks * T, np.int32)
        st = np.zeros(S, dtype=lv.SESSION_DTYPE)
        st["gen_us"] = rng.integers(0, 30_000_000, S) // (1 if S < 100 else 10_000_000) * 1
        st["flags"] = lv.LV_RESP_OPEN
        pool.import_placement(table, ctx)
        pool.set_sessions(st)
        new = -(-(blocks * T + grow) // T) - blocks
        k = away + new
        cand = rng.permutation(S).astype(np.int32)
        keys = rng.integers(0, 1 + away // 2, cap).astype(np.uint64) if scatter else None
        result = np.zeros(1, lv.RESIDENT_DTYPE)
        lv.lv_turn(pool.handle, -1, 5, grow, 1_000_000, 10, (pool.victims, pool.slots, pool.blks, pool.pages, pool.app),
                   result, cand, S, pool.stream, 0, keys)
        pool.sync()
        # the same turn on the host
        resident = [{b: int(table[s, b]) for b in range(cap) if table[s, b] >= 0} for s in range(S)]
        want = [v for v in _order(st, resident, 5) if v[0] != sid][:k]
        assert len(want) == k
        free_slots = sorted(set(range(host)) - set(slots.tolist()))
        loads = list(range(blocks - away, blocks))
        if scatter:
            loads.sort(key=lambda b: (int(keys[b]), b))
        free = sorted(v[2] for v in want)
        r = result[0]
        assert (int(r["sid"]), int(r["k"]), int(r["n_found"]), int(r["n_victims"]), int(r["n_loaded"]),
                int(r["n_appended"]), int(r["status"])) == (sid, k, k, k, away, new, 0)
        assert pool.victims[:k].cpu().numpy().tolist() == [list(v) for v in want]
        assert pool.slots[:k].cpu().numpy().tolist() == free_slots[:k]
        assert pool.blks[:away].cpu().numpy().tolist() == loads
        assert pool.pages[:away].cpu().numpy().tolist() == free[:away]
        assert pool.app[:new].cpu().numpy().tolist() == free[away:away + new]
        for (s, b, _), h in zip(want, free_slots):
            table[s, b] = -(h + 2)
        table[sid, loads] = free[:away]
        table[sid, blocks:blocks + new] = free[away:away + new]
        got, own_hbm, own_host = pool.tables()
        assert np.array_equal(got, table)
        a, b = pool.counts()
        assert np.array_equal(a, (table >= 0).sum(1)) and np.array_equal(b, (table <= -2).sum(1))
        s_idx, b_idx = np.nonzero(table >= 0)
        assert np.array_equal(own_hbm[table[s_idx, b_idx]], s_idx << 16 | b_idx)
        # a second decision reads the counts that the first one left
        victims, m = pool.select(5, 10, 0)
        after = pool.get_sessions()
        resident = [{b: int(table[s, b]) for b in range(cap) if table[s, b] >= 0} for s in range(S)]
        want = _order(after, resident, 5)[:10]
        assert victims.cpu().numpy().tolist() == [list(v) for v in want]
        lv.lv_evict(pool.handle, 5, 10, 0, pool.victims, pool.slots, result, pool.stream)
        pool.sync()
        assert pool.victims[:len(want)].cpu().numpy().tolist() == [list(v) for v in want]
    finally:
        pool.close()


@pytest.mark.parametrize("where", ["device", "pinned", "pageable", "overlapping", "misaligned"])
@pytest.mark.parametrize("n_blocks", [20, 1500])
def test_step_outputs_wherever_they_lie(where, n_blocks):
    """The lists of a step are the same in device memory, where the kernel writes them itself, as
    in host memory and in device arrays that it may not write: overlapping ones (each list is
    copied in turn, so the last one stands) and one that is not aligned for 32-bit words."""
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    rng = np.random.default_rng(n_blocks)
    S, away = 4, n_blocks - 3
    budget, host = S * n_blocks - away, 2 * away + 8
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=S, max_blocks=n_blocks, hbm_pages=budget,
                  hbm_budget_pages=budget, host_pages=host)
    try:
        table = np.full((S, n_blocks), -1, np.int32)
        pages = rng.permutation(budget)
        slots = rng.permutation(host)[:away]
        table[0, 3:] = -(slots + 2)
        table[0, :3] = pages[:3]
        table[1:] = pages[3:].reshape(S - 1, n_blocks)
        st = np.zeros(S, dtype=lv.SESSION_DTYPE)
        st["gen_us"] = [0, 9_000_000, 8_000_000, 7_000_000]
        pool.import_placement(table, np.full(S, n_blocks * T, np.int32))
        pool.set_sessions(st)
        sizes = [budget * 12, budget * 4, n_blocks * 4, n_blocks * 4]        # victims, slots, blocks, pages
        at = np.concatenate([[0], np.cumsum([s + 16 for s in sizes])])
        kw = dict(dtype=torch.uint8, device=pool.device) if where in ("device", "overlapping", "misaligned") else dict(dtype=torch.uint8)
        buf = torch.zeros(int(at[-1]) + 16, **kw)
        buf = buf.pin_memory() if where == "pinned" else buf
        off = [int(x) for x in at[:4]]
        if where == "misaligned":
            off[1] += 2
        if where == "overlapping":
            off[2] = off[3] = off[0]           # pages lie over blocks and over the first victims
        outs = tuple(buf.data_ptr() + o for o in off) + (None,)
        lv.lv_turn(pool.handle, 0, 0, 0, 1_000_000, 10, outs, None, None, 0, pool.stream)
        pool.sync()
        got = [buf[o:o + s].cpu().numpy() for o, s in zip(off, sizes)]
        want_victims = [(1, b, table[1, b]) for b in range(n_blocks - 1, 2, -1)]
        want_slots = sorted(set(range(host)) - set(slots.tolist()))[:away]
        want_pages = sorted(v[2] for v in want_victims)
        assert got[1][:4 * away].copy().view(np.int32).tolist() == want_slots
        assert got[3][:4 * away].copy().view(np.int32).tolist() == want_pages
        if where != "overlapping":
            assert got[0][:12 * away].copy().view(np.int32).reshape(-1, 3).tolist() == [list(v) for v in want_victims]
            assert got[2][:4 * away].copy().view(np.int32).tolist() == list(range(3, n_blocks))
    finally:
        pool.close()
