"""Pack, unpack and checksums from a list of page ids, wherever the list lies, with ids outside
the pool in it, on both sides of the shared cursor's limit, by TMA and by plain copies; and
pools of different sub-page sizes side by side (their stage kernels share one limit)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sums(kv, pages, hbm):
    out = np.zeros(len(pages), np.uint64)
    J, _, P = kv.shape
    w = (2 * np.arange(J * P // 8, dtype=np.uint64) + 1).astype(np.uint64)
    with np.errstate(over="ignore"):
        for i, p in enumerate(pages):
            if 0 <= p < hbm:
                out[i] = (np.ascontiguousarray(kv[:, p]).view(np.uint64).reshape(-1) * w).sum(dtype=np.uint64)
    return out


@pytest.mark.parametrize("where", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("shape,n,kernel", [((2, 2, 64), 1, "tma"), ((3, 1, 8), 37, "tma"), ((40, 1, 8), 61, "tma"),
                                            ((40, 1, 8), 64, "lsu"), ((2, 4, 960), 5, "tma")])
def test_page_lists(where, shape, n, kernel, monkeypatch):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    monkeypatch.setenv("LV_STAGE_KERNEL", kernel)
    layers, heads, dim = shape
    hbm = 2 * n + 3
    kw = dict(max_sessions=2, max_blocks=2, host_pages=0)
    pool = KVPool(layers=layers, kv_heads=heads, head_dim=dim, hbm_pages=hbm, hbm_budget_pages=hbm, **kw)
    small = KVPool(layers=1, kv_heads=1, head_dim=8, hbm_pages=4, hbm_budget_pages=4, **kw)
    try:
        rng = np.random.default_rng(n)
        kv = rng.integers(0, 256, (pool.J, hbm, pool.P)).astype(np.uint8)
        pool.kv.copy_(torch.from_numpy(kv))
        order = rng.permutation(hbm).astype(np.int32)
        src, dst = order[:n].copy(), order[n:2 * n].copy()
        if n > 3:
            src[1], dst[2] = hbm, -1
        lists = [torch.from_numpy(a) for a in (src, dst)]
        lists = [a.cuda() if where == "device" else a.pin_memory() if where == "pinned" else a for a in lists]
        run = torch.full((n, pool.J, pool.P), 7, dtype=torch.uint8, device="cuda")
        sums = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        lv.lv_page_checksums(pool.handle, lists[0], n, sums, pool.stream)
        lv.lv_pack_pages(pool.handle, lists[0], n, run, pool.stream)
        lv.lv_unpack_pages(pool.handle, run, lists[1], n, pool.stream)
        err = pool.sync(raise_on_error=False)
        assert err == (lv.LV_ERR_BOUNDS if n > 3 else 0)
        want = np.full((n, pool.J, pool.P), 7, np.uint8)
        for i in range(n):
            if 0 <= src[i] < hbm:
                want[i] = kv[:, src[i]]
        assert np.array_equal(run.cpu().numpy(), want)
        assert np.array_equal(sums.cpu().numpy().view(np.uint64), _sums(kv, src, hbm))
        for i in range(n):
            if 0 <= dst[i] < hbm:
                kv[:, dst[i]] = want[i]
        assert np.array_equal(pool.kv.cpu().numpy(), kv)
    finally:
        small.close()
        pool.close()


@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_checksums_around_the_cursor(extra):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    ctas = torch.cuda.get_device_properties(0).multi_processor_count * 8
    n = ctas * 4 // 2 + extra                     # units of J = 2, four to a batch
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=2, max_blocks=2, hbm_pages=n, hbm_budget_pages=n,
                  host_pages=0)
    try:
        rng = np.random.default_rng(1)
        kv = rng.integers(0, 256, (2, n, pool.P)).astype(np.uint8)
        pool.kv.copy_(torch.from_numpy(kv))
        pages = rng.permutation(n).astype(np.int32)
        sums = torch.zeros(n, dtype=torch.int64, device="cuda")
        for _ in range(2):
            lv.lv_page_checksums(pool.handle, torch.from_numpy(pages).cuda(), n, sums, pool.stream)
            pool.sync()
            assert np.array_equal(sums.cpu().numpy().view(np.uint64), _sums(kv, pages, n))
    finally:
        pool.close()
