"""Pools whose allocation bitmaps do not fit in shared memory decide as smaller ones do: the
same calls -- turns with ordered loads and growth, evictions, exchanges, swaps, commits,
cancels and growth, with short lists and with lists past what shared memory holds -- on a pool
of 760,000 pages and slots and on one of a few thousand, with the same budget, give the same
lists, tables, owners and counts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LARGE = 760_000
S, CAP = 6, 3000


def _pools(tiers, budget, host):
    from paper_2606_22983_gb300.pool import KVPool
    kw = dict(layers=1, kv_heads=1, head_dim=8, page_tokens=2, max_sessions=S, max_blocks=CAP, hbm_budget_pages=budget,
              tiers=tiers)
    # (the host tier is never short in either)
    return [KVPool(hbm_pages=budget + 40, host_pages=host, **kw), KVPool(hbm_pages=LARGE, host_pages=LARGE, **kw)]


@pytest.mark.parametrize("tiers", [0, 1])
@pytest.mark.parametrize("most", [60, 2800])         # blocks of a session at most
def test_same_decisions(tiers, most):
    import torch
    from paper_2606_22983_gb300 import lv
    rng = np.random.default_rng(most + tiers)
    blocks = rng.integers(most // 2, most, S)
    host = int(2 * S * CAP + 16)
    budget = int(blocks.sum() * 3 // 4)
    pools = _pools(tiers, budget, host)
    try:
        table = np.full((S, CAP), -1, np.int32)
        pages, slots, used = rng.permutation(budget + 40).tolist(), rng.permutation(host).tolist(), 0
        for s in range(S):
            for b in range(blocks[s]):
                if used < budget - 8 and rng.random() < 0.72:
                    table[s, b], used = pages.pop(), used + 1
                else:
                    table[s, b] = -(slots.pop() + 2)
        ctx = (2 * blocks - rng.integers(0, 2, S)).astype(np.int32)
        st = np.zeros(S, dtype=lv.SESSION_DTYPE)
        st["gen_us"] = rng.integers(0, 10_000_000, S)
        for p in pools:
            p.import_placement(table, ctx)
            p.set_sessions(st)
            assert p.sync() == 0
        errors = []
        for step in range(40):
            call = ["turn", "evict", "exchange", "out", "in", "append", "resident"][int(rng.integers(0, 7))]
            sid, n = int(rng.integers(0, S)), int(rng.integers(1, most))
            grow, back = int(rng.choice([0, 1, 9])), rng.random() < 0.4
            keys = rng.integers(0, 50, CAP).astype(np.uint64) if rng.random() < 0.5 else None
            got = []
            for p in pools:
                result = np.zeros(1, lv.RESIDENT_DTYPE)
                outs = (p.victims, p.slots, p.blks, p.pages, p.app)
                lists = []
                if call in ("turn", "resident"):
                    if call == "turn":
                        lv.lv_turn(p.handle, sid, step, grow, 1_000_000, 5, outs, result, None, 0, p.stream, 0, keys)
                    else:
                        lv.lv_make_resident(p.handle, sid, step, 0, lv.LV_RESIDENT_PRELOAD, -1, *outs, result, p.stream)
                    p.sync(raise_on_error=False)
                    r = result[0]
                    nv, nl, na = int(r["n_victims"]), int(r["n_loaded"]), int(r["n_appended"])
                    lists = [p.victims[:nv], p.slots[:nv], p.blks[:nl], p.pages[:nl], p.app[:na], torch.from_numpy(result.view(np.int64))]
                elif call == "evict":
                    lv.lv_evict(p.handle, step, n, 0, p.victims, p.slots, result, p.stream)
                    p.sync(raise_on_error=False)
                    nv = int(result["n_victims"][0])
                    lists = [p.victims[:nv], p.slots[:nv], torch.from_numpy(result.view(np.int64))]
                elif call == "append":
                    lists = [p.append(sid, grow)] if p.counts()[0].sum() + grow < budget else []
                else:
                    v, nv = p.select(step, n)
                    v = v.clone()
                    b, nb = p.blocks(sid, 1)
                    b = b[v.new_tensor(np.random.default_rng(step).permutation(nb)).long()].contiguous() if nb else b
                    if call == "exchange":
                        v = v[v[:, 0] != sid].contiguous()
                        free = budget - int(p.stats()["hbm_allocated"])
                        nb = min(nb, len(v) + free)
                        lists = [*p.exchange(v, len(v), sid, b, nb)]
                    elif call == "out" and nv:
                        slots_, commit = p.swap_out(v, nv)
                        lists = [slots_.clone(), commit.clone()]
                        if back:
                            p.cancel((-(lists[0] + 2)).int(), nv)
                        else:
                            p.remap(lists[1], nv)
                    elif call == "in" and nb:
                        nb = min(nb, budget - int(p.stats()["hbm_allocated"]) + 3)   # some are refused
                        if nb > 0:
                            pages_, commit = p.swap_in(sid, b, nb)
                            lists = [pages_.clone(), commit.clone()]
                            if int(lists[0][0]) < 0:
                                lists.pop()             # (a refused call writes no entries)
                            else:
                                (p.cancel(lists[0], nb) if back else p.remap(lists[1], nb))
                err = p.sync(raise_on_error=False)
                p.clear_error()
                t, own_hbm, own_host = p.tables()
                stats = p.stats()
                got.append(([x.cpu().numpy().copy() for x in lists], err, t, own_hbm[:budget + 40], own_host[:host], *p.counts(),
                            {k: stats[k] for k in ("hbm_allocated", "host_allocated", "pages_out", "pages_in", "clean_copies",
                                                   "appended_pages", "cancels")}))
                assert (own_hbm[budget + 40:] == -1).all() and (own_host[host:] == -1).all(), (step, call)
                assert stats["hbm_allocated"] == (own_hbm != -1).sum() and stats["host_allocated"] == (own_host != -1).sum()
            a, b = got
            errors.append(a[1])
            assert len(a[0]) == len(b[0]) and all(np.array_equal(x, y) for x, y in zip(a[0], b[0])), (step, call)
            for x, y in zip(a[1:], b[1:]):
                assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y, (step, call)
        assert errors.count(0) > 20
    finally:
        for p in pools:
            p.close()
