"""lv_remap's forms -- the entries free their old locations themselves, or a release pass does,
with 1, 2 or 4 entries per thread -- leave the same tables, owners, counts and free pages,
with wrong entries among the right ones and under both tier modes; and the default form on both
sides of the line between them, in session order and in any other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
T = 16


def _run(env, tiers, n_sessions, blocks, seed, monkeypatch):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    if env is None:
        monkeypatch.delenv("LV_REMAP_ENTRIES_PER_THREAD", raising=False)
    else:
        monkeypatch.setenv("LV_REMAP_ENTRIES_PER_THREAD", env)
    rng = np.random.default_rng(seed)
    N = n_sessions * blocks
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=n_sessions, max_blocks=blocks, hbm_pages=N + 5,
                  hbm_budget_pages=N + 5, host_pages=N + 7, tiers=tiers)
    try:
        table = rng.permutation(N + 5)[:N].astype(np.int32).reshape(n_sessions, blocks)
        pool.import_placement(table, np.full(n_sessions, blocks * T, np.int32))
        seen = []
        for rnd in range(3):
            tables, _, _ = pool.tables()
            s, b = np.nonzero(tables >= 0)
            pick = rng.permutation(len(s))[:max(1, len(s) // 2)]
            victims = np.stack([s[pick], b[pick], tables[s[pick], b[pick]]], 1).astype(np.int32)
            v = torch.from_numpy(victims).cuda()
            _, commit = pool.swap_out(v, len(v))
            c = commit.cpu().numpy().copy()
            # wrong entries name blocks that no right entry names (which of two entries for a block
            # is taken is open), but for one entry that is there twice
            bad = [[0, blocks, 3], [n_sessions, 0, 3]]
            rest = np.setdiff1d(np.arange(len(s)), pick)
            if len(rest) >= 4:
                o = [(int(s[x]), int(b[x])) for x in rest[:4]]
                bad += [[*o[0], -1], [*o[1], N + 5], [*o[2], -(N + 9)], [*o[3], int(tables[o[3]])]]
            bad = np.array(bad + [c[-1].tolist()], np.int32)
            entries = np.concatenate([bad, c] if rnd == 1 else [c, bad])
            pool.remap(torch.from_numpy(entries).cuda(), len(entries))
            err = pool.sync(raise_on_error=False)
            pool.clear_error()
            seen.append((err != 0, *pool.tables(), *pool.counts()))
            # half of one session's offloaded blocks come back
            sid = int(s[pick[0]])
            blks, n = pool.blocks(sid, 1)
            n = (n + 1) // 2
            pages, commit = pool.swap_in(sid, blks[:n].clone(), n)
            seen.append((pages.cpu().numpy(),))
            pool.remap(commit, n)
            st = pool.stats()
            seen.append((pool.sync(), *pool.tables(), *pool.counts(), {k: st[k] for k in (
                "hbm_allocated", "host_allocated", "remap_entries", "clean_copies", "clean_out")}))
            t, _, _ = pool.tables()
            a, d = pool.counts()
            assert np.array_equal(a, (t >= 0).sum(1)) and np.array_equal(d, (t <= -2).sum(1))
        return seen
    finally:
        pool.close()


@pytest.mark.parametrize("tiers", [0, 1])
@pytest.mark.parametrize("n_sessions,blocks", [(1, 2), (5, 40), (33, 70)])
def test_forms_agree(tiers, n_sessions, blocks, monkeypatch):
    want = _run(None, tiers, n_sessions, blocks, 3, monkeypatch)
    for env in ("1", "2", "4"):
        got = _run(env, tiers, n_sessions, blocks, 3, monkeypatch)
        for w, g in zip(want, got):
            for x, y in zip(w, g):
                assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y


@pytest.mark.parametrize("order", ["sessions", "mixed"])
@pytest.mark.parametrize("n", [2**14 - 1, 2**14, 2**14 + 1, 2**18 + 1, 700_001])
@pytest.mark.parametrize("S", [1, 16, 700, 4096])
def test_default_form(S, n, order, tmp_path):
    """The kernel's per-session counts after a commit of n entries, and the pages it freed."""
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    from ._pool_words import pool_words
    blocks = -(-(n + 3) // S)
    if blocks > 65536:
        return
    N = S * blocks
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, page_tokens=1, max_sessions=S, max_blocks=blocks, hbm_pages=N,
                  hbm_budget_pages=N, host_pages=N)
    try:
        rng = np.random.default_rng(n + S)
        table = rng.permutation(N).astype(np.int32).reshape(S, blocks)
        pool.import_placement(table, np.full(S, blocks, np.int32))
        pick = rng.permutation(N)[:n] if order == "mixed" else np.arange(n)
        s, b = pick // blocks, pick % blocks
        v = torch.from_numpy(np.stack([s, b, table[s, b]], 1).astype(np.int32)).cuda()
        _, commit = pool.swap_out(v, n)
        pool.remap(commit, n)
        assert pool.sync() == 0
        free = np.sort(table[s, b])
        table[s, b] = -(np.arange(n) + 2)
        t, own_hbm, own_host = pool.tables()
        assert np.array_equal(t, table)
        assert np.array_equal(np.nonzero(own_hbm == -1)[0], free) and (own_host[:n] == (s << 16 | b)).all()
        _, _, cnt = pool_words(pool, tmp_path)
        assert np.array_equal(cnt.cpu().numpy(), np.stack([(t >= 0).sum(1), (t <= -2).sum(1)], 1))
        # the freed pages, and no others, are there to be taken
        sid = int(s[0])
        back = np.nonzero(t[sid] <= -2)[0].astype(np.int32)
        pages, commit = pool.swap_in(sid, torch.from_numpy(back).cuda(), len(back))
        assert pool.sync() == 0 and np.array_equal(pages.cpu().numpy(), free[:len(back)])
        pool.remap(commit, len(back))
        assert pool.sync() == 0
        a, d = pool.counts()
        assert np.array_equal(cnt.cpu().numpy(), np.stack([a, d], 1))
        assert pool.stats()["hbm_allocated"] == N - n + len(back)
    finally:
        pool.close()
