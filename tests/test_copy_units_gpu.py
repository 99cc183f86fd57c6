"""The exchange copy takes a page in 16 KiB units whatever its sub-page size: pages whose
sub-pages are far smaller than a unit, cross its edge, match it, or exceed it, and more
sub-page arrays than a CTA keeps addresses for.  Every byte of both tiers is compared."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (layers, KV heads, head dim, page tokens, element bytes): sub-pages of 16 B, 48 B, 1008 B,
# 16368 B, 16 KiB, 16400 B and 40 KiB; 1200 arrays of 16 B
SHAPES = [(3, 1, 8, 1, 2), (7, 1, 24, 2, 1), (5, 1, 63, 16, 1), (2, 1, 1023, 16, 1), (2, 4, 128, 16, 2),
          (3, 1, 1025, 16, 1), (2, 8, 80, 32, 2), (600, 1, 8, 1, 2)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n_out,n_in", [(6, 9), (9, 6), (5, 0), (0, 4)])
def test_exchange_moves_every_byte(shape, n_out, n_in):
    import torch
    from paper_2606_22983_gb300 import lv
    from paper_2606_22983_gb300.pool import KVPool
    layers, heads, dim, tokens, elem = shape
    S, B, host_pages = 3, 16, 40
    hbm = 2 * B
    rng = np.random.default_rng(n_out * 31 + n_in)
    pool = KVPool(layers=layers, kv_heads=heads, head_dim=dim, page_tokens=tokens, elem_bytes=elem,
                  max_sessions=S, max_blocks=B, hbm_pages=hbm, hbm_budget_pages=hbm, host_pages=host_pages)
    try:
        # sessions 0 and 1 in HBM but for the last 8 blocks of session 1; session 2 in the host tier
        table = np.full((S, B), -1, np.int32)
        pages, slots = rng.permutation(hbm), rng.permutation(host_pages)
        table[0], table[1, :8] = pages[:B], pages[B:B + 8]
        table[1, 8:], table[2] = -(slots[:8] + 2), -(slots[8:8 + B] + 2)
        pool.import_placement(table, np.full(S, B * tokens, np.int32))
        kv = rng.integers(0, 256, (pool.J, hbm, pool.P)).astype(np.uint8)
        host = rng.integers(0, 256, pool.host.shape).astype(np.uint8)
        pool.kv.copy_(torch.from_numpy(kv))
        pool.host_dev.copy_(torch.from_numpy(host))
        torch.cuda.synchronize()
        blocks = rng.permutation(B)[:n_out].astype(np.int32)
        loads = rng.permutation(B)[:n_in].astype(np.int32)
        victims = np.array([(0, b, table[0, b]) for b in blocks], np.int32).reshape(-1, 3)
        v = torch.from_numpy(victims).cuda() if n_out else None
        b = torch.from_numpy(loads).cuda() if n_in else None
        slot, page = pool.exchange(v, n_out, 2, b, n_in)
        pool.sync()
        slot, page = slot.cpu().numpy(), page.cpu().numpy()
        want_kv, want_host = kv.copy(), host.copy()
        want_host[slot] = kv[:, victims[:, 2]].transpose(1, 0, 2)
        want_kv[:, page] = host[-(table[2, loads] + 2)].transpose(1, 0, 2)
        assert np.array_equal(pool.kv.cpu().numpy(), want_kv)
        assert np.array_equal(pool.host, want_host)
    finally:
        pool.close()
