"""The scheduling round at the edges of its CTAs' chunks (512 requests) and cluster sizes, with
keys that tie in their upper half or whole, against the oracle's scheduler."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 511, 512, 513, 1024, 1025, 2047, 2049, 3000, 4095])
@pytest.mark.parametrize("kind", ["mixed", "one class", "all equal", "wide"])
def test_round_at_chunk_edges(n, kind):
    from oracle.scheduler import schedule
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    rng = np.random.default_rng(n)
    arr = np.zeros(n, dtype=lv.REQUEST_DTYPE)
    arr["id"] = rng.permutation(n)
    arr["started"] = rng.random(n) < 0.7 if kind in ("mixed", "wide") else 1
    arr["play_buffer_us"] = 0 if kind == "all equal" else rng.integers(0, 1 << 40 if kind == "wide" else 8_000_000, n)
    arr["ready_age_us"] = rng.integers(0, 1 << 62 if kind == "wide" else 20, n)
    arr["kv_pages"] = rng.integers(0, 1 << 24 if kind == "wide" else 2000, n)
    arr["tokens"] = rng.integers(0, 400, n)
    arr["kv_needed"] = rng.integers(0, 50, n)
    wide = kind == "wide"
    args = (1 << 32 if wide else 2_000_000, 1 << 16 if wide else 4, 1 << 16 if wide else 1, 1 << 32 if wide else 30_000,
            1 << 32 if wide else 40_000, 90 * n, 12 * n)
    want_order, want_batch = schedule([{k: int(r[k]) for k in lv.REQUEST_DTYPE.names} for r in arr], *args)
    pool = KVPool(layers=1, kv_heads=1, head_dim=8, max_sessions=4, max_blocks=4, hbm_pages=16,
                  hbm_budget_pages=16, host_pages=16)
    try:
        q = lv.lv_sched_params(p_safe_us=args[0], alpha=args[1], beta=args[2], occupied=args[3],
                               allocatable=args[4], token_budget=args[5], kv_budget=args[6])
        order, batch = np.full(n, -1, np.int32), np.full(1, -1, np.int32)
        lv.lv_schedule(pool.handle, q, arr, n, order, batch, pool.stream)
        pool.sync()
        assert order.tolist() == want_order
        assert order[:int(batch[0])].tolist() == want_batch
    finally:
        pool.close()
