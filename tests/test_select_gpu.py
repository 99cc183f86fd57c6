"""lv_select_victims and lv_select_victims_noalloc where their kernels change: sessions at the
edges of a cluster's chunks, one victim to past the largest single-kernel selection, many
sessions of one block, rows on both sides of the census's forms.  The order is a plain sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
T = 16
NOW = 10_000_000


def _want(st, table, within, policy, counters, fallback):
    rank = []
    for s in range(len(st)):
        x = st[s]
        if policy:
            if not x["flags"] & 1:
                rank.append((0, min(max(int(x["last_use_us"]), 0), 0xFFFFFFFF), s))
            continue
        normal = not x["flags"] & 3 and not NOW < x["protect_until_us"]
        if not normal and not (fallback and not x["flags"] & 1):
            continue
        if counters:
            play = int(x["reply_tokens"]) * 80_000 if x["flags"] & 4 and x["reply_tokens"] > 0 else 0
        else:
            play = max(0, int(x["gen_us"]) - int(x["play_us"]))
        reply = max(0, int(x["reply_ema_us"]) if x["reply_n"] > 0 else 3_000_000)
        t = min(min(play, 0xFFFFFFFF) + min(reply, 0xFFFFFFFF), 0xFFFFFFFF)
        rank.append((0 if normal else 1, -t, s))
    out = []
    for _, _, s in sorted(rank):
        b = np.nonzero(table[s] >= 0)[0]
        b = b if within else b[::-1]
        out += [(s, int(x), int(table[s, x])) for x in b]
    return out


CASES = [(1, 5), (31, 40), (512, 3), (513, 3), (1024, 9), (1025, 2), (2048, 1), (4096, 1), (4096, 4), (3, 1024), (5, 1030)]


@pytest.mark.parametrize("S,B", CASES)
@pytest.mark.parametrize("within,policy,counters,fallback", [(0, 0, 0, 0), (1, 0, 1, 1), (0, 1, 0, 0)])
def test_selection(S, B, within, policy, counters, fallback):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    rng = np.random.default_rng(S * 31 + B)
    table = np.full((S, B), -1, np.int32)
    n = rng.integers(0 if S > 1 else 1, B + 1, S)
    where = rng.random((S, B)) < 0.8
    hbm = host = 0
    for s in range(S):
        for b in range(n[s]):
            if where[s, b]:
                table[s, b], hbm = hbm, hbm + 1
            else:
                table[s, b], host = -(host + 2), host + 1
    hbm, host = max(hbm, 1), max(host, 1)
    st = np.zeros(S, dtype=lv.SESSION_DTYPE)
    st["ctx_tokens"] = n * T
    st["flags"] = rng.choice([0, 1, 2, 4, 4, 4, 6], S)
    st["gen_us"] = rng.choice([0, 5_000_000, 2**33, int(1e15)], S) + rng.integers(0, 4, S)
    st["play_us"] = rng.integers(0, 3, S)
    st["reply_tokens"] = rng.choice([0, 50, 2**40], S)
    st["reply_n"] = rng.integers(0, 2, S)
    st["reply_ema_us"] = rng.choice([0, 1_000_000, 2**34], S)
    st["protect_until_us"] = rng.choice([0, NOW, NOW + 1], S)
    st["last_use_us"] = rng.choice([-5, 0, 7, 2**35], S)
    want = _want(st, table, within, policy, counters, fallback)
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=S, max_blocks=B, hbm_pages=hbm, hbm_budget_pages=hbm,
                  host_pages=host, within_order=within, policy=policy, t_play_mode=counters)
    try:
        pool.import_placement(table, n * T)
        pool.set_sessions(st)
        dev = torch.from_numpy(table).cuda()
        sess = torch.from_numpy(st.view(np.uint8).copy()).cuda()
        for k in (0, 1, 33, 2048, 2049, len(want) + 5):
            m = min(k, len(want))
            out = torch.full((max(k, 1), 3), -7, dtype=torch.int32, device="cuda")
            cnt = torch.full((1,), -7, dtype=torch.int64, device="cuda")
            lv.lv_select_victims(pool.handle, NOW, k, fallback, out, k, cnt, pool.stream)
            stats = pool.stats()
            assert (stats["last_select_count"], stats["last_select_total"], int(cnt)) == (m, len(want), m)
            got = out.cpu().numpy()
            assert got[:m].tolist() == [list(v) for v in want[:m]] and (got[m:] == -7).all()
            q = lv.lv_rank_params(num_sessions=S, max_blocks=B, page_tokens=T, within_order=within, t_play_mode=counters,
                                  flags=fallback, reply_prior_us=3_000_000, unit_us=80_000, policy=policy, reserved=0)
            out.fill_(-7)
            lv.lv_select_victims_noalloc(q, sess, dev, NOW, k, out, k, cnt, pool.stream)
            assert int(cnt) == m
            got = out.cpu().numpy()
            assert got[:m].tolist() == [list(v) for v in want[:m]] and (got[m:] == -7).all()
    finally:
        pool.close()
