"""The copy-engine path where its transfers are ordered and cut: runs of consecutive host slots
around the 24 pages of a chunk, many short runs beside a long one, every slot by itself, blocks
listed in any order.  Every byte of both tiers is compared."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B, HOST = 64, 140                     # pages of 1 MiB: a chunk of 24 MiB holds 24


def _slots(pattern):
    if pattern == "one run":
        return np.arange(30, 30 + B)
    if pattern == "every other":
        return np.arange(0, 2 * B, 2)
    out, at = [], 1                   # "mixed": runs of 1, 2, 5, 25 and 31 with holes between
    for n in (1, 25, 2, 5, 31):
        out += range(at, at + n)
        at += n + 3
    return np.array(out)


@pytest.mark.parametrize("pattern", ["one run", "every other", "mixed"])
@pytest.mark.parametrize("n_out,n_in", [(64, 64), (25, 24), (1, 49), (49, 1), (23, 0), (0, 25)])
@pytest.mark.parametrize("how", ["exchange", "async", "swap"])
def test_staged_moves_every_byte(pattern, n_out, n_in, how):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    rng = np.random.default_rng(100 * n_out + n_in)
    hbm = 2 * B
    pool = KVPool(layers=8, kv_heads=4, head_dim=512, page_tokens=16, elem_bytes=2, max_sessions=2,
                  max_blocks=B, hbm_pages=hbm, hbm_budget_pages=hbm, host_pages=HOST)
    try:
        assert pool.J * pool.P == 1 << 20
        table = np.full((2, B), -1, np.int32)
        table[0] = rng.permutation(hbm)[:B]
        table[1] = -(rng.permutation(_slots(pattern)) + 2)
        pool.import_placement(table, np.full(2, B * 16, np.int32))
        pool.kv.view(torch.int64).random_(generator=torch.Generator("cuda").manual_seed(n_out))
        kv = pool.kv.cpu().numpy()
        host = rng.bytes(pool.host.size)
        host = np.frombuffer(host, np.uint8).reshape(pool.host.shape)
        pool.host[:] = host
        torch.cuda.synchronize()
        victims = np.array([(0, b, table[0, b]) for b in rng.permutation(B)[:n_out]], np.int32).reshape(-1, 3)
        loads = rng.permutation(B)[:n_in].astype(np.int32)
        v = torch.from_numpy(victims).cuda() if n_out else None
        b = torch.from_numpy(loads).cuda() if n_in else None
        if how == "swap":
            slot = pool.swap_out(v, n_out, lv.LV_MODE_STAGED)[0] if n_out else None
            page = pool.swap_in(1, b, n_in, lv.LV_MODE_STAGED)[0] if n_in else None
        else:
            mode = lv.LV_MODE_STAGED | (lv.LV_MODE_ASYNC if how == "async" else 0)
            slot, page = pool.exchange(v, n_out, 1, b, n_in, mode)
        pool.sync()
        want_kv, want_host = kv.copy(), host.copy()
        if n_out:
            want_host[slot.cpu().numpy()[:n_out]] = kv[:, victims[:, 2]].transpose(1, 0, 2)
        if n_in:
            want_kv[:, page.cpu().numpy()[:n_in]] = host[-(table[1, loads] + 2)].transpose(1, 0, 2)
        assert np.array_equal(pool.kv.cpu().numpy(), want_kv)
        assert np.array_equal(pool.host, want_host)
    finally:
        pool.close()
