"""The performance cases of the KV swap path: what a serving engine's KV manager has it do.

Each case is one pass of a kind of work, through the calls of ``paper_2606_22983_gb300``
that an engine makes, with the values these meet in service:

  turn      a turn of one session: the clients' playback reports, then ``lv_turn`` picks the
            first speaking session with offloaded KV, evicts what its reload needs and loads it
  grow      a turn of a session whose KV was preloaded: its context grows (``lv_turn`` with
            appended tokens) and idle sessions give up as many pages as it takes
  relieve   memory pressure, then a preload: ``lv_evict`` frees pages (offload only), and a user
            who starts to speak has their session loaded ahead of the turn (reload only)
  handoff   the same exchange of KV by a host-driven manager: rank, then swap out, commit, swap
            in, commit one after the other, or one ``lv_swap_exchange``
  rank      one eviction decision over a large pool's metadata
  schedule  one round of the urgency scheduler over the ready requests
  pages     pages saved aside and put back elsewhere, with their checksums: ``lv_page_checksums``,
            ``lv_pack_pages``, ``lv_unpack_pages``, ``lv_page_checksums``

The outputs are bytes and whole numbers throughout, so they are compared exactly.
"""
import math
import random

import numpy as np
import torch

from paper_2606_22983_gb300 import lv
from paper_2606_22983_gb300.harness import fill_random
from paper_2606_22983_gb300.pool import KVPool

SEC = 1_000_000
STEP_US = SEC // 2                     # between two passes
BASE_US = 100 * SEC                    # the first pass's time
MOST_HBM = 8 << 30                     # bytes of KV that a drawn case holds in HBM
MOST_MOVE = 1 << 30                    # bytes that a drawn case moves each way

# the benchmark's KV shapes (layers, KV heads, head dim): pages of 16 KiB and 1.5 MiB, and a
# small model's pages of 192 KiB between the two
TINY = dict(layers=2, kv_heads=2, head_dim=64, page_tokens=16, elem_bytes=2)
THINKER = dict(layers=48, kv_heads=4, head_dim=128, page_tokens=16, elem_bytes=2)
SMALL = dict(layers=24, kv_heads=2, head_dim=64, page_tokens=16, elem_bytes=2)


def page_bytes(c):
    return 2 * c["layers"] * c["page_tokens"] * c["kv_heads"] * c["head_dim"] * c["elem_bytes"]


def listed():
    turn = dict(kind="turn", scatter=False, inclusive=False, lru=False, overlap=False)
    hand = dict(kind="handoff", inclusive=False)
    rank = dict(kind="rank", lru=False, ascending=False, counters=False, fallback=False, bare=False)
    return [
        # the smallest pool: eight sessions of a two-layer model, a few hundred KB a turn
        dict(turn, name="turn_tiny", sessions=8, max_blocks=128, blocks=60, move=24, **TINY),
        # a turn of the benchmark's model, 300 MB each way, with the copies on the copy stream
        dict(turn, name="turn_thinker", sessions=16, max_blocks=1024, blocks=210, move=203, overlap=True,
             **THINKER),
        # many short sessions of a small model, reloaded in scattered order
        dict(turn, name="turn_many", sessions=1000, max_blocks=256, blocks=45, move=45, scatter=True, **SMALL),
        # a long context comes back: the largest turn, over 1 GB each way
        dict(turn, name="turn_long", sessions=6, max_blocks=4096, blocks=720, move=705, **THINKER),
        # turns that find their KV in HBM and only grow, by 16 to 96 tokens each
        dict(kind="grow", name="grow", sessions=24, idle=8, max_blocks=256, blocks=30, least=16, most=96,
             inclusive=False, **THINKER),
        # pages freed under pressure and a preload at speech start, 48 pages (72 MB) each
        dict(kind="relieve", name="relieve", sessions=6, idle=10, max_blocks=256, blocks=60, move=48,
             inclusive=False, **THINKER),
        # the host-driven manager: the four calls one after the other, over the mapped pool
        dict(hand, name="handoff_calls", sessions=6, idle=26, max_blocks=512, blocks=100, move=37, exchange=False,
             staged=False, **SMALL),
        # the host-driven manager with the copy engines
        dict(hand, name="handoff_staged", sessions=5, idle=3, max_blocks=256, blocks=160, move=150, exchange=True,
             staged=True, **THINKER),
        # a decision over a million resident pages
        dict(rank, name="rank_1024", sessions=1024, max_blocks=1024, k=256, **dict(TINY, layers=1, kv_heads=1, head_dim=8)),
        # and over the most sessions a pool takes, in the counters' estimate and with the fallback tier
        dict(rank, name="rank_4096", sessions=4096, max_blocks=256, k=1500, counters=True, fallback=True,
             **dict(TINY, layers=1, kv_heads=1, head_dim=8)),
        # a scheduling round of a busy stage
        dict(kind="schedule", name="schedule", n=3000, **TINY),
        # 500 pages (0.8 GB) saved aside and restored, with checksums of both
        dict(kind="pages", name="pages", n=500, **THINKER),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _shape(rng):
    return dict(layers=rng.choice([2, 5, 12, 24, 28, 48]), kv_heads=rng.choice([1, 2, 4, 8]),
                head_dim=rng.choice([64, 96, 128]), page_tokens=rng.choice([16, 16, 32]),
                elem_bytes=rng.choice([2, 2, 1]))


def draw(rng: random.Random):
    kind = rng.choice(["turn", "turn", "turn", "grow", "relieve", "handoff", "handoff", "rank", "rank",
                       "schedule", "pages"])
    if kind == "schedule":
        return dict(kind=kind, n=_log(rng, 5, 4096), **TINY)
    if kind == "rank":
        sessions = _log(rng, 8, 4096)
        return dict(kind=kind, sessions=sessions, max_blocks=_log(rng, 32, min(4096, (1 << 20) // sessions)),
                    k=_log(rng, 1, 4096), lru=rng.random() < 0.2, ascending=rng.random() < 0.2,
                    counters=rng.random() < 0.3, fallback=rng.random() < 0.4, bare=rng.random() < 0.25,
                    **dict(TINY, layers=1, kv_heads=1, head_dim=8))
    c = dict(kind=kind, **_shape(rng))
    pb = page_bytes(c)
    # a host tier with a slot for every block: pools that a preparation page-locks quickly
    inclusive = rng.random() < 0.25 and pb <= 256 << 10
    if kind == "pages":
        return dict(c, n=_log(rng, 1, min(8192, 2 * MOST_MOVE // (3 * pb))))
    room = (1 << 30 if inclusive else MOST_HBM) // pb     # pages the sessions may hold together
    if kind == "grow":
        idle = rng.randint(6, 12)
        blocks = _log(rng, 16, max(16, min(128, room // 40)))
        return dict(c, sessions=_log(rng, 4, 32), idle=idle, max_blocks=blocks + _log(rng, 224, 1024),
                    blocks=blocks, least=rng.choice([1, 16]), most=rng.choice([24, 96, 96]),
                    inclusive=inclusive)
    most = MOST_MOVE if kind == "turn" else MOST_MOVE // 2   # these move one way at a time
    move = _log(rng, 1, max(1, min(700, most // pb, room // 16)))
    blocks = move + _log(rng, 1, max(1, move // 2))
    if kind == "turn":
        sessions = _log(rng, 3, max(3, min(1024, room // (2 * blocks))))
        return dict(c, sessions=sessions, max_blocks=2 * blocks + _log(rng, 1, 1024), blocks=blocks, move=move,
                    scatter=rng.random() < 0.4, inclusive=inclusive, lru=rng.random() < 0.2,
                    overlap=rng.random() < 0.4)
    c = dict(c, sessions=rng.randint(4, 8), idle=_log(rng, 1, max(1, min(256, room // (2 * blocks) - 8))),
             max_blocks=2 * blocks + _log(rng, 1, 1024), blocks=blocks, move=move, inclusive=inclusive)
    if kind == "relieve":
        return c
    how = rng.choice([(False, False), (True, False), (True, True), (False, True)])
    return dict(c, exchange=how[0], staged=how[1])


# ------------------------------------------------------------------ state
class _Mapped:
    """The pool's host tier as a CUDA array that keeps the pool alive."""

    def __init__(self, pool):
        self.pool = pool
        nbytes = pool.host_pages * pool.J * pool.P
        self.__cuda_array_interface__ = {"shape": (nbytes // 8,), "typestr": "<i8", "version": 3, "strides": None,
                                         "data": (lv.lv_pool_host_device_ptr(pool.handle), False)}


class _State:
    pass


def _pinned(array):
    """A page-locked copy of a numpy array's bytes."""
    return torch.from_numpy(np.ascontiguousarray(array).view(np.uint8).reshape(-1)).pin_memory()


def _rows(rows):
    """Event lists of equal length in page-locked memory, and the address of each."""
    a = np.stack(rows)
    t = _pinned(a)
    return t, [t.data_ptr() + i * a[0].nbytes for i in range(len(a))], len(a[0])


def _event(kind, sid, t, a=0, b=0):
    return (kind, sid, t, a, b)


def _events(items):
    return np.array(items, dtype=lv.EVENT_DTYPE)


def _pool(c, total, budget, host_pages, sessions, max_blocks, **over):
    return KVPool(layers=c["layers"], kv_heads=c["kv_heads"], head_dim=c["head_dim"], page_tokens=c["page_tokens"],
                  elem_bytes=c["elem_bytes"], max_sessions=sessions, max_blocks=max_blocks, hbm_pages=total,
                  hbm_budget_pages=budget, host_pages=host_pages, stream=torch.cuda.current_stream().cuda_stream,
                  **over)


def _placed(rng, n_blocks, max_blocks, host_of, hbm_pages, host_pages):
    """Every block on a random HBM page, but the last host_of[s] blocks of session s on random
    host slots, as in a pool that has been in service for a while."""
    S = len(n_blocks)
    pages, slots = rng.permutation(hbm_pages), rng.permutation(host_pages)
    table = np.full((S, max_blocks), -1, np.int32)
    p = h = 0
    for s in range(S):
        n, away = int(n_blocks[s]), int(host_of.get(s, 0))
        table[s, :n - away] = pages[p:p + n - away]
        table[s, n - away:n] = -(slots[h:h + away] + 2)
        p, h = p + n - away, h + away
    return table


def _sizes(rng, lo, hi, S):
    """The block counts of S sessions: evenly spread over lo..hi, and dealt out in random order."""
    return rng.permutation(np.linspace(lo, hi, S).round().astype(np.int64))


def _contexts(rng, c, n_blocks):
    """Context lengths of so many blocks, the last one filled in part."""
    return (np.asarray(n_blocks) * c["page_tokens"] - rng.integers(0, c["page_tokens"], len(n_blocks))).astype(np.int32)


def _talking(rng, S):
    """Sessions in the middle of a conversation: a reply of 5 to 30 s partly played."""
    st = np.zeros(S, dtype=lv.SESSION_DTYPE)
    st["flags"] = lv.LV_RESP_OPEN
    st["gen_us"] = rng.integers(5 * SEC, 30 * SEC, S)
    st["play_us"] = (rng.random(S) * st["gen_us"]).astype(np.int64)
    st["reply_tokens"] = st["gen_us"] // 80_000
    st["reply_n"] = rng.integers(0, 4, S)
    st["reply_ema_us"] = np.where(st["reply_n"] > 0, rng.integers(SEC // 2, 6 * SEC, S), 0)
    st["last_use_us"] = rng.integers(0, BASE_US, S)
    return st


def _ready(s, c, pool, table, ctx, states, seed, kv=True):
    pool.import_placement(table, ctx)
    pool.set_sessions(states)
    s.pool, s.handle, s.stream, s.i = pool, pool.handle, pool.stream, 0
    if kv:
        fill_random(pool, seed)
        s.kv = pool.kv.view(-1).view(torch.int64)
        s.host = torch.as_tensor(_Mapped(pool), device=pool.device)
    s.result = torch.zeros(lv.RESIDENT_DTYPE.itemsize // 8, dtype=torch.int64, device=pool.device)
    pool.sync()
    return s


def _prepare_turn(c, seed):
    rng, s = np.random.default_rng(seed), _State()
    S, B, D = c["sessions"], c["blocks"], c["move"]
    n = _sizes(rng, B, min(c["max_blocks"], B + B // 8), S)
    total = int(n.sum())
    away = int(rng.integers(0, S))                 # the session whose KV is in the host tier
    budget = total - D
    host = (total if c["inclusive"] else 2 * D) + 64
    pool = _pool(c, budget, budget, host, S, c["max_blocks"],
                 policy=lv.LV_POLICY_LRU if c["lru"] else lv.LV_POLICY_NEXT_USE,
                 tiers=lv.LV_TIERS_INCLUSIVE if c["inclusive"] else lv.LV_TIERS_EXCLUSIVE)
    R, reports = 32, min(S, 64)
    rows = [_events([_event(lv.LV_EV_PLAYBACK, int(x), BASE_US + i * STEP_US, STEP_US)
                     for x in rng.permutation(S)[:reports]]) for i in range(R)]
    s.events, s.event_at, s.n_events = _rows(rows)
    s.perms = torch.from_numpy(np.stack([rng.permutation(S) for _ in range(R)]).astype(np.int32)).cuda()
    s.perm_at = [s.perms[i].data_ptr() for i in range(R)]
    s.audio = [int(x) for x in rng.integers(5 * SEC, 30 * SEC, R)]
    s.keys, s.key_at = None, [None] * R
    if c["scatter"]:
        keys = np.stack([rng.permutation(c["max_blocks"]) for _ in range(R)]).astype(np.int64)
        s.keys = torch.from_numpy(keys).cuda()
        s.key_at = [s.keys[i].data_ptr() for i in range(R)]
    s.flags = lv.LV_RESIDENT_ASYNC_COPY if c["overlap"] else 0
    s.S = S
    _ready(s, c, pool, _placed(rng, n, c["max_blocks"], {away: D}, budget, host), _contexts(rng, c, n),
           _talking(rng, S), seed)
    s.outs = (pool.victims, pool.slots, pool.blks, pool.pages, None)
    s.answer = (pool.victims[:D], pool.slots[:D], pool.blks[:D], pool.pages[:D], s.result, s.kv, s.host)
    return s


def _run_turn(s):
    i, r = s.i, s.i % len(s.event_at)
    s.i += 1
    lv.lv_session_events(s.handle, s.event_at[r], s.n_events, s.stream)
    lv.lv_turn(s.handle, -1, BASE_US + i * STEP_US, 0, s.audio[r], s.audio[r] // 80_000, s.outs, s.result,
               s.perm_at[r], s.S, s.stream, s.flags, s.key_at[r])
    if s.flags:
        lv.lv_join(s.handle, s.stream)             # what follows on the stream reads the session's KV
    return s.answer


def _prepare_grow(c, seed):
    rng, s = np.random.default_rng(seed), _State()
    S, I, B, T = c["sessions"], c["idle"], c["blocks"], c["page_tokens"]
    R = 32                                         # turns before these conversations end
    # the turns grow the contexts alike for every seed (how many pages a pass moves follows from
    # it); which session, where its KV lies and what it holds are the seed's
    fixed = np.random.default_rng(1)
    grow = fixed.permutation(np.linspace(c["least"], c["most"], R).round().astype(np.int64))
    tail = fixed.integers(1, T + 1, S)             # rows in the last block of the i-th to speak
    at, new = tail.astype(np.int64), []
    for i in range(R):
        new.append(int(-(-(at[i % S] + grow[i]) // T) - (-(-at[i % S] // T))))
        at[i % S] += grow[i]
    # the idle sessions hold what these turns take
    n = np.concatenate([_sizes(rng, max(1, B - B // 4), B + B // 4, S), np.full(I, max(B, -(-sum(new) // I) + 1))])
    order = rng.permutation(S)
    ctx = _contexts(rng, c, n)
    ctx[order] = (n[order] - 1) * T + tail
    total = int(n.sum())
    host = (total if c["inclusive"] else 0) + sum(new) + 32
    pool = _pool(c, total, total, host, S + I, c["max_blocks"],
                 tiers=lv.LV_TIERS_INCLUSIVE if c["inclusive"] else lv.LV_TIERS_EXCLUSIVE)
    rows = [_events([_event(lv.LV_EV_PLAYBACK, int(x), BASE_US + i * STEP_US, STEP_US)
                     for x in rng.permutation(S)[:4]]) for i in range(R)]
    s.events, s.event_at, s.n_events = _rows(rows)
    s.sid, s.grow = [int(order[i % S]) for i in range(R)], [int(x) for x in grow]
    s.audio = [int(x) for x in rng.integers(2 * SEC, 6 * SEC, R)]
    st = _talking(rng, S + I)
    st["gen_us"][:S] = rng.integers(2 * SEC, 6 * SEC, S)
    st["play_us"][:S] = 0
    st["gen_us"][S:], st["play_us"][S:] = rng.integers(40 * SEC, 60 * SEC, I), 0   # long replies just begun
    table = _placed(rng, n, c["max_blocks"], {}, total, host)
    s.table, s.ctx = torch.from_numpy(table).cuda(), torch.from_numpy(ctx).cuda()
    s.begin = _pinned(st)
    _ready(s, c, pool, table, ctx, st, seed)
    s.N = S + I
    s.outs = (pool.victims, pool.slots, None, None, pool.app)
    s.answers = [(pool.victims[:m], pool.slots[:m], pool.app[:m], s.result, s.kv, s.host) for m in new]
    return s


def _run_grow(s):
    i, r = s.i, s.i % len(s.event_at)
    s.i += 1
    if r == 0 and i > 0:                           # these conversations are over: new ones begin
        lv.lv_pool_import(s.handle, s.table, s.ctx, s.stream)
        lv.lv_session_set(s.handle, s.begin, 0, s.N, s.stream)
    lv.lv_session_events(s.handle, s.event_at[r], s.n_events, s.stream)
    lv.lv_turn(s.handle, s.sid[r], BASE_US + r * STEP_US, s.grow[r], s.audio[r], s.audio[r] // 80_000, s.outs,
               s.result, None, 0, s.stream)
    return s.answers[r]


def _prepare_cycle(c, seed):
    """Sessions that take turns: one has just begun a long reply (it is evicted next), the one
    before it is offloaded and starts to speak, the one before that begins its turn."""
    rng, s = np.random.default_rng(seed), _State()
    C, I, B, D = c["sessions"], c["idle"], c["blocks"], c["move"]
    n = _sizes(rng, B, min(c["max_blocks"], B + B // 8), C + I)
    total = int(n.sum())
    order = [int(x) for x in rng.permutation(C)]
    budget = total - D
    host = (total if c["inclusive"] else 2 * D) + 64
    pool = _pool(c, budget, budget, host, C + I, c["max_blocks"],
                 tiers=lv.LV_TIERS_INCLUSIVE if c["inclusive"] else lv.LV_TIERS_EXCLUSIVE)
    rows = []
    for i in range(C):
        t = BASE_US + i * STEP_US
        y, z, w = order[i], order[i - 1], order[i - 2]
        ev = [_event(lv.LV_EV_TURN_END, y, t, int(rng.integers(40 * SEC, 60 * SEC)), 600),
              _event(lv.LV_EV_SPEECH_START, z, t), _event(lv.LV_EV_SPEECH_STOP, w, t),
              _event(lv.LV_EV_TURN_BEGIN, w, t)]
        idle = C + rng.permutation(I)[:min(I, 8)]
        rows.append(_events(ev + [_event(lv.LV_EV_PLAYBACK, int(x), t, STEP_US) for x in idle]))
    s.events, s.event_at, s.n_events = _rows(rows)
    st = _talking(rng, C + I)
    st["flags"][:C], st["gen_us"][:C], st["play_us"][:C] = lv.LV_RUNNING, 0, 0
    st["flags"][order[-1]] = lv.LV_RESP_OPEN
    st["gen_us"][order[-1]] = 50 * SEC
    st["flags"][order[-2]] = lv.LV_IMMEDIATE
    st["gen_us"][C:] = np.minimum(st["gen_us"][C:], 25 * SEC)
    _ready(s, c, pool, _placed(rng, n, c["max_blocks"], {order[-1]: D}, budget, host), _contexts(rng, c, n), st, seed)
    s.loads = [order[i - 1] for i in range(C)]
    s.D, s.cap = D, pool.cap
    dev = pool.device
    s.count = torch.zeros(2, dtype=torch.int64, device=dev)
    s.count_at = (s.count.data_ptr(), s.count.data_ptr() + 8)
    return s


def _prepare_relieve(c, seed):
    s = _prepare_cycle(c, seed)
    p = s.pool
    s.result2 = torch.zeros_like(s.result)
    s.answer = (p.victims[:s.D], p.slots[:s.D], s.result, p.blks[:s.D], p.pages[:s.D], s.result2, s.kv, s.host)
    return s


def _run_relieve(s):
    i, r = s.i, s.i % len(s.event_at)
    s.i += 1
    now, p = BASE_US + i * STEP_US, s.pool
    lv.lv_session_events(s.handle, s.event_at[r], s.n_events, s.stream)
    lv.lv_evict(s.handle, now, s.D, 0, p.victims, p.slots, s.result, s.stream)
    lv.lv_make_resident(s.handle, s.loads[r], now, 0, lv.LV_RESIDENT_PRELOAD, -1, None, None, p.blks, p.pages, None,
                        s.result2, s.stream)
    return s.answer


def _prepare_handoff(c, seed):
    s = _prepare_cycle(c, seed)
    p, D = s.pool, s.D
    s.exchange, s.mode = c["exchange"], lv.LV_MODE_STAGED if c["staged"] else lv.LV_MODE_AUTO
    s.commit_in = torch.empty((D, 3), dtype=torch.int32, device=p.device)
    s.answer = (p.victims[:D], s.count, p.slots[:D], p.blks[:D], p.pages[:D], s.kv, s.host)
    if not s.exchange:
        s.answer += (p.commit[:D], s.commit_in)
    return s


def _run_handoff(s):
    i, r = s.i, s.i % len(s.event_at)
    s.i += 1
    p, D, sid = s.pool, s.D, s.loads[r]
    lv.lv_session_events(s.handle, s.event_at[r], s.n_events, s.stream)
    lv.lv_select_victims(s.handle, BASE_US + i * STEP_US, D, 0, p.victims, D, s.count_at[0], s.stream)
    if s.exchange:
        lv.lv_session_blocks(s.handle, sid, 1, p.blks, s.count_at[1], s.stream)
        lv.lv_swap_exchange(s.handle, p.victims, D, sid, p.blks, D, p.slots, p.pages, s.mode, s.stream)
    else:
        lv.lv_swap_out(s.handle, p.victims, D, p.slots, p.commit, s.mode, s.stream)
        lv.lv_remap(s.handle, p.commit, D, s.stream)
        lv.lv_session_blocks(s.handle, sid, 1, p.blks, s.count_at[1], s.stream)
        lv.lv_swap_in(s.handle, sid, p.blks, D, p.pages, s.commit_in, s.mode, s.stream)
        lv.lv_remap(s.handle, s.commit_in, D, s.stream)
    return s.answer


def _prepare_rank(c, seed):
    rng, s = np.random.default_rng(seed), _State()
    S, B = c["sessions"], c["max_blocks"]
    n = _sizes(rng, B - B // 4, B, S)
    # one session in sixteen has a part of its KV in the host tier
    host_of = {int(x): B // 3 for x in rng.permutation(S)[:max(1, S // 16)]}
    away = sum(host_of.values())
    total = int(n.sum()) - away
    pool = _pool(c, total, total, max(1, away), S, B,
                 policy=lv.LV_POLICY_LRU if c["lru"] else lv.LV_POLICY_NEXT_USE,
                 within_order=lv.LV_ASCENDING if c["ascending"] else lv.LV_SUFFIX_FIRST,
                 t_play_mode=lv.LV_PLAY_COUNTERS if c["counters"] else lv.LV_PLAY_PLAYBACK)
    st = _talking(rng, S)
    u = rng.random(S)
    st["flags"] = np.where(u < 0.1, lv.LV_RUNNING, np.where(u < 0.2, lv.LV_IMMEDIATE, st["flags"]))
    st["protect_until_us"] = np.where(u > 0.95, BASE_US + 2 * SEC, 0)
    # half of them are always there to be evicted, so that k are found for certain
    st["flags"][:S // 2], st["protect_until_us"][:S // 2] = lv.LV_RESP_OPEN, 0
    s = _ready(s, c, pool, _placed(rng, n, B, host_of, total, max(1, away)), _contexts(rng, c, n), st, seed, kv=False)
    s.flags = lv.LV_SELECT_FALLBACK if c["fallback"] else 0
    s.k = min(c["k"], (S // 2) * (B - B // 4 - B // 3))
    s.out = torch.empty((s.k, 3), dtype=torch.int32, device=pool.device)
    s.count = torch.zeros(1, dtype=torch.int64, device=pool.device)
    s.params = None
    if c["bare"]:                                  # the caller's own tables, no pool
        s.tables = torch.empty((S, B), dtype=torch.int32, device=pool.device)
        s.sessions = torch.empty(S * lv.SESSION_DTYPE.itemsize, dtype=torch.uint8, device=pool.device)
        lv.lv_read_tables(pool.handle, s.tables, None, None, s.stream)
        lv.lv_session_get(pool.handle, s.sessions, 0, S, s.stream)
        s.params = lv.lv_rank_params(num_sessions=S, max_blocks=B, page_tokens=c["page_tokens"],
                                     within_order=int(c["ascending"]), t_play_mode=int(c["counters"]),
                                     flags=s.flags, reply_prior_us=3 * SEC, unit_us=80_000, policy=int(c["lru"]),
                                     reserved=0)
    return s


def _run_rank(s):
    now = BASE_US + (s.i % 16) * STEP_US           # the protections run out on the way
    s.i += 1
    if s.params is not None:
        lv.lv_select_victims_noalloc(s.params, s.sessions, s.tables, now, s.k, s.out, s.k, s.count, s.stream)
    else:
        lv.lv_select_victims(s.handle, now, s.k, s.flags, s.out, s.k, s.count, s.stream)
    return s.out, s.count


def _prepare_schedule(c, seed):
    rng, s = np.random.default_rng(seed), _State()
    n = c["n"]
    reqs = np.zeros(n, dtype=lv.REQUEST_DTYPE)
    reqs["id"] = rng.permutation(n)
    reqs["started"] = rng.random(n) < 0.7
    reqs["play_buffer_us"] = rng.integers(0, 8, n) * 700_000 + rng.integers(0, 50, n) * 1000
    reqs["ready_age_us"] = rng.integers(0, 10_000_000, n)
    reqs["kv_pages"] = rng.integers(0, 2048, n)
    reqs["tokens"] = rng.integers(1, 512, n)
    reqs["kv_needed"] = rng.integers(0, 64, n)
    pool = _pool(c, 64, 64, 64, 8, 16)
    _ready(s, c, pool, np.full((8, 16), -1, np.int32), np.zeros(8, np.int32), np.zeros(8, lv.SESSION_DTYPE), seed, kv=False)
    s.reqs, s.n = _pinned(reqs), n                 # the engine's ready set, in host memory
    s.params = lv.lv_sched_params(p_safe_us=2 * SEC, alpha=4, beta=1, occupied=30_000, allocatable=40_000,
                                  token_budget=8192, kv_budget=4096)
    s.order = torch.empty(n, dtype=torch.int32, device=pool.device)
    s.batch = torch.empty(1, dtype=torch.int32, device=pool.device)
    return s


def _run_schedule(s):
    lv.lv_schedule(s.handle, s.params, s.reqs, s.n, s.order, s.batch, s.stream)
    return s.order, s.batch


def _prepare_pages(c, seed):
    rng, s = np.random.default_rng(seed), _State()
    n = c["n"]
    total = 2 * n + 1 + n // 8
    pool = _pool(c, total, total, 0, 4, 4)
    pool.import_placement(np.full((4, 4), -1, np.int32), np.zeros(4, np.int32))
    s.pool, s.handle, s.stream, s.i, s.n = pool, pool.handle, pool.stream, 0, n
    fill_random(pool, seed)
    s.kv = pool.kv.view(-1).view(torch.int64)
    pages = torch.from_numpy(rng.permutation(total)[:2 * n].astype(np.int32)).to(pool.device)
    s.old, s.new = pages[:n].clone(), pages[n:].clone()
    s.saved = torch.empty(n * page_bytes(c) // 8, dtype=torch.int64, device=pool.device)
    s.sums = torch.zeros((2, n), dtype=torch.int64, device=pool.device)
    s.sums_at = (s.sums.data_ptr(), s.sums.data_ptr() + 8 * n)
    pool.sync()
    return s


def _run_pages(s):
    lv.lv_page_checksums(s.handle, s.old, s.n, s.sums_at[0], s.stream)
    lv.lv_pack_pages(s.handle, s.old, s.n, s.saved, s.stream)
    lv.lv_unpack_pages(s.handle, s.saved, s.new, s.n, s.stream)
    lv.lv_page_checksums(s.handle, s.new, s.n, s.sums_at[1], s.stream)
    return s.sums, s.saved, s.kv


_KINDS = {"turn": (_prepare_turn, _run_turn), "grow": (_prepare_grow, _run_grow),
          "relieve": (_prepare_relieve, _run_relieve), "handoff": (_prepare_handoff, _run_handoff),
          "rank": (_prepare_rank, _run_rank), "schedule": (_prepare_schedule, _run_schedule),
          "pages": (_prepare_pages, _run_pages)}


def prepare(case, seed):
    make, run_kind = _KINDS[case["kind"]]
    s = make(case, seed)
    s.run = run_kind
    return s


def run(state):
    return state.run(state)


def work(case):
    """Bytes that a pass has to read or write once: KV pages in both tiers, block tables,
    requests and their order."""
    c, kind = case, case["kind"]
    pb = page_bytes(c)
    if kind == "rank":
        return {"bytes": c["sessions"] * (c["max_blocks"] * 7 / 8 * 4 + 72) + 12 * c["k"], "flops": 0}
    if kind == "schedule":
        return {"bytes": 52 * c["n"], "flops": 0}
    if kind == "pages":
        return {"bytes": 6 * c["n"] * pb, "flops": 0}     # two reads for the sums, two copies
    if kind == "grow":
        return {"bytes": 2 * pb * (c["least"] + c["most"]) / 2 / c["page_tokens"], "flops": 0}
    return {"bytes": 4 * c["move"] * pb, "flops": 0}      # read and written once on the way out, and in


def tolerance(case):
    return "exact"


def exact(case, seed):
    return None                                    # whole numbers and bytes: there is nothing to round
