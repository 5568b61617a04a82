"""The calls a user of kvtier makes, as measurable cases.

A serving engine runs one epoch at a time: score every resident block and choose the
victims, move them to the host ring, bring prefetched ones back, admit new blocks.  The
cases cover that loop as a whole and each of its calls alone, from a pool of 4,096
head-blocks to one of 18.8 million, for GQA, MHA, MQA and MLA models, the three eviction
policies, the confidence blend, the head-importance matrix, block-granular and
allocation-free selection, the position-ordered prefetch, and content hashing with
deduplication.

The pools are those of `workloads.config` and of the tests: their layers, heads, eviction
and promotion shares, and their traces.  Calls that never touch block bytes (everything up
to the choice of victims, and the prefetch list) run on pools with 64- to 256-byte blocks
(`tiny_entries` there), which leaves entry counts, state arrays and traces as they are.

A trace is the touches of one epoch: every (layer, head) of the blocks that this epoch's
requests use, plus one touch with a miss flag for every slot that the epoch before has
freed and filled again.  Those slots are the victims of the pass before, so `run` lets each
selection write its victims straight into the tail of the next trace.  Six traces are used
in turn, and a pool has lived through a few epochs before it is handed over.
"""
import math

import numpy as np
import torch

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

TRACES = 6          # traces a pool goes through in turn
WARM_EPOCHS = 12    # epochs a pool has behind it when it is handed over
DECAY = 0.9
KAPPA, WINDOW = 100.0, 16     # confidence blend


# ---- the cases -----------------------------------------------------------------------

def _case(kind, arch, layers, heads, blocks, **more):
    c = {"kind": kind, "arch": arch, "layers": layers, "heads": heads, "blocks": blocks, "style": "chat",
         "evict": 0.10, "policy": 0, "blend": False, "weights": False}
    c.update(more)
    return c


def listed():
    return [
        # the test pool (2 layers x 512 blocks x 4 heads): a call is launches and latency
        _case("epoch", "gqa", 2, 4, 512, name="epoch-tiny", style="entry", evict=0.05),
        # a 61-layer MLA model's pool, one entry per block, agentic sessions, confidence blend on
        _case("epoch", "mla", 61, 1, 14912, name="epoch-mla-blend", style="agentic", blend=True),
        # a 32-layer GQA model's pool of 24 GiB under shared-prefix chat: the ordinary call
        _case("epoch", "gqa", 32, 8, 12288, name="epoch-chat"),
        # four models in one 150 GiB pool: the largest call, and the benchmark's
        _case("epoch", "fleet", 0, 0, 10720, name="epoch-fleet", style="mixed"),
        # events, update and selection as three calls (what a pool sharded over GPUs does), the
        # EMA-only policy, the head-importance matrix updated every epoch; an odd number of blocks
        _case("split", "gqa", 80, 8, 5003, name="split-heads", style="long", evict=0.15, policy=1, weights=True),
        # eviction of whole paged blocks by their aggregate over the heads
        _case("blocks", "gqa", 32, 8, 12288, name="blocks-chat"),
        # selection for an engine that has no memory to spare: a ragged number of entries
        {"kind": "static", "name": "static-ragged", "n": 1_000_003, "evict": 0.10},
        # the whole epoch of the test pool, LRU policy: the host's part and the launches count
        _case("step", "gqa", 2, 4, 512, name="step-tiny-lru", style="entry", evict=0.05, policy=2, q_heads=16,
              head_dim=64, block_tokens=16, promote=0.02, order="recent", deferred=False, batch_mb=1),
        # the whole epoch of the chat pool at 1/16: victims leave and prefetched runs return
        _case("step", "gqa", 32, 8, 768, name="step-chat", q_heads=32, head_dim=128, block_tokens=16,
              promote=0.03, order="runs", deferred=True, batch_mb=64),
        # the same for the 80-layer long-context pool at 1/64, whose prefetch is ordered by
        # position: runs of eight slots all over the ring
        _case("step", "gqa", 80, 8, 288, name="step-longctx", style="long", evict=0.15, q_heads=64, head_dim=128,
              block_tokens=16, promote=0.10, order="position", deferred=True, batch_mb=64),
        # the blocks that one epoch admits to the chat pool at 1/4 are hashed and deduplicated
        {"kind": "hash", "name": "hash-chat", "arch": "gqa", "layers": 32, "heads": 8, "q_heads": 32, "head_dim": 128,
         "block_tokens": 16, "blocks": 3072, "hashed": 78_643},
        # eight long sequences ask for the blocks of their next positions
        {"kind": "prefetch", "name": "prefetch-longctx", "layers": 80, "heads": 8, "blocks": 2304, "n_pos": 256,
         "sequences": 8, "away": 0.4},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, lo, hi):
    """An architecture and a pool of roughly lo .. hi entries of it."""
    n = _log_uniform(rng, lo, hi)
    arch = rng.choice(["gqa", "gqa", "mha", "mqa", "mla"])
    layers = rng.choice([2, 16, 28, 32, 61, 80] if n > 40_000 else [2, 4, 6])
    heads = {"gqa": rng.choice([2, 4, 8]), "mha": rng.choice([12, 32]), "mqa": 1, "mla": 1}[arch]
    return arch, layers, heads, max(8, n // (layers * heads))


def draw(rng):
    kind = rng.choice(["epoch", "epoch", "epoch", "split", "blocks", "static", "step", "step", "hash", "prefetch"])
    if kind in ("epoch", "split", "blocks"):
        if kind == "epoch" and rng.random() < 0.25:
            return _case(kind, "fleet", 0, 0, _log_uniform(rng, 40, 10_700), style="mixed",
                         evict=rng.uniform(0.02, 0.15), policy=rng.choice([0, 0, 1, 2]), blend=rng.random() < 0.3,
                         weights=rng.random() < 0.3)
        arch, layers, heads, blocks = _draw_shape(rng, 4_000, 12_000_000)
        return _case(kind, arch, layers, heads, blocks, style=rng.choice(["chat", "long", "agentic"]),
                     evict=rng.uniform(0.02, 0.25), policy=rng.choice([0, 0, 1, 2]), blend=rng.random() < 0.3,
                     weights=rng.random() < 0.3)
    if kind == "static":
        return {"kind": "static", "n": _log_uniform(rng, 4_000, 4_194_304), "evict": rng.uniform(0.02, 0.25)}
    if kind == "step":
        arch, layers, heads, blocks = _draw_shape(rng, 4_000, 150_000)
        mla = arch == "mla"
        if mla:   # (a block of an MLA model holds nine times the bytes of a head of the others)
            blocks = max(8, blocks // 9)
        return _case("step", arch, layers, heads, blocks, style=rng.choice(["chat", "long", "agentic"]),
                     evict=rng.uniform(0.05, 0.15), policy=rng.choice([0, 0, 1, 2]),
                     q_heads={"gqa": 4 * heads, "mha": heads, "mqa": 32, "mla": 128}[arch],
                     head_dim=rng.choice([64, 128]), block_tokens=64 if mla else 16,
                     promote=rng.uniform(0.01, 0.04), order=rng.choice(["recent", "runs", "position"]),
                     deferred=rng.random() < 0.5, batch_mb=rng.choice([8, 64]))
    if kind == "hash":
        if rng.random() < 0.3:   # MLA: few and long messages
            blocks = _log_uniform(rng, 8, 300)
            n = 61 * blocks
            return {"kind": "hash", "arch": "mla", "layers": 61, "heads": 1, "q_heads": 128, "head_dim": 128,
                    "block_tokens": 64, "blocks": blocks, "hashed": max(1, int(n * rng.uniform(0.1, 0.9)))}
        blocks = _log_uniform(rng, 16, 1500)
        n = 32 * 8 * blocks
        return {"kind": "hash", "arch": "gqa", "layers": 32, "heads": 8, "q_heads": 32, "head_dim": rng.choice([64, 128]),
                "block_tokens": 16, "blocks": blocks, "hashed": max(1, int(n * rng.uniform(0.05, 0.3)))}
    n_pos = _log_uniform(rng, 33, 1000)
    layers, heads = rng.choice([32, 80]), rng.choice([1, 8])
    sequences = rng.randint(1, max(1, min(16, 2304 // n_pos)))
    return {"kind": "prefetch", "layers": layers, "heads": heads, "blocks": max(n_pos * sequences, 512) + rng.randint(0, 99),
            "n_pos": n_pos, "sequences": sequences, "away": rng.uniform(0.1, 0.8)}


# ---- pools and traces ----------------------------------------------------------------

def _ok(rc, what):
    if rc != B.KV_OK:
        raise B.KVError(rc, what)


_STREAM = []


def _compute():
    """The engine's compute stream: epochs follow one another on it, whichever pool they belong to."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _partition(arch, layers, heads, blocks, q_heads=None, head_dim=1, block_tokens=16, ring=16):
    if arch == "gqa":
        return W.gqa(layers, q_heads or 4 * heads, heads, head_dim, block_tokens, blocks, ring)
    if arch == "mha":
        return W.mha(layers, heads, head_dim, block_tokens, blocks, ring)
    if arch == "mqa":
        return W.mqa(layers, q_heads or 32, head_dim, block_tokens, blocks, ring)
    return W.mla(layers, 8 if head_dim == 1 else 512, 0 if head_dim == 1 else 64, block_tokens, blocks, ring)


def _partitions(case):
    if case["arch"] == "fleet":
        nb = case["blocks"]
        return [_partition("mha", 32, 32, nb), _partition("gqa", 80, 8, nb), _partition("mqa", 32, 1, nb),
                _partition("mla", 61, 1, nb)]
    ring = 16
    if case["kind"] == "step":   # room for the victims of three epochs
        ring = 3 * _victims(case) + 16
    return [_partition(case["arch"], case["layers"], case["heads"], case["blocks"], case.get("q_heads"),
                       case.get("head_dim", 1), case.get("block_tokens", 16), ring)]


def _entries(case):
    if case["kind"] == "static":
        return case["n"]
    if case["arch"] == "fleet":
        return case["blocks"] * (32 * 32 + 80 * 8 + 32 + 61)
    return case["layers"] * case["heads"] * case["blocks"]


def _victims(case):
    if case["kind"] == "blocks":
        return int(case["evict"] * case["layers"] * case["blocks"]) * case["heads"]
    return max(4, int(case["evict"] * _entries(case)))


def _touched_blocks(style, p, r):
    """Block numbers that one epoch's requests touch in a partition (repeats are repeated touches)."""
    nb, tok = p.blocks_per_layer, p.block_tokens
    if style == "mixed":
        style = "chat" if r.random() < 0.5 else "agentic"
    if style == "long":      # 64 sequences: the last 4K tokens of each, and 5 % of the older blocks
        win = max(1, min(4096 // tok, (nb * 8 // 9) // 64))
        perm = np.random.default_rng(nb).permutation(nb)
        n_win = min(nb, 64 * win)
        old = r.choice(nb - n_win, size=int(0.05 * (nb - n_win)), replace=False) if nb > n_win else []
        return np.concatenate([perm[:n_win], perm[n_win + np.asarray(old, np.int64)]])
    runs = []
    if style == "chat":      # Zipf(1.1) over 500 shared prefixes, and a fresh prompt for each request
        lens = np.maximum(1, W.lognormal_tokens(np.random.default_rng(nb), 600, 1.0, 8192, 500) // tok)
        region = max(1, int(0.6 * nb))
        starts = (np.cumsum(lens) - lens) % region
        n_req = max(1, int(round(40 * min(1.0, nb / 12288))))
        for q in W.zipf_bounded(r, 1.1, 500, n_req):
            runs.append((starts[q] + np.arange(min(lens[q], region))) % region)
            fresh = max(1, nb - region)
            n = min(fresh, max(1, int(W.lognormal_tokens(r, 600, 1.0, 8192, 1)[0]) // tok))
            runs.append((region + (r.integers(0, fresh) + np.arange(n)) % fresh) % nb)
    else:                    # agentic: 30 sessions append a turn, most of them re-read what they have
        n_act = max(1, int(round(30 * min(1.0, nb / 4096))))
        for _ in range(n_act):
            start, old = int(r.integers(0, nb)), int(min(nb // 8, r.integers(1, 9) * 800 // tok))
            add = min(max(1, nb // 8), max(1, int(W.lognormal_tokens(r, 800, 1.0, 1 << 16, 1)[0]) // tok))
            if r.random() < 0.7:
                runs.append((start + np.arange(old)) % nb)
            runs.append((start + old + np.arange(add)) % nb)
    return np.concatenate(runs)


def _touches(style, parts, bases, r):
    """Entry ids of one epoch's touches, on the GPU."""
    out = []
    for p, base in zip(parts, bases):
        if style == "entry":   # independent touches: block ~ Zipf(1.1), layer and head uniform
            n = int(0.2 * p.n_entries)
            block = np.random.default_rng(7).permutation(p.blocks_per_layer)[W.zipf_bounded(r, 1.1, p.blocks_per_layer, n)]
            ids = (r.integers(0, p.n_layers, n) * p.blocks_per_layer + block) * p.heads + r.integers(0, p.heads, n)
            out.append(torch.from_numpy(base + ids).cuda())
            continue
        blocks = torch.from_numpy(_touched_blocks(style, p, r)).cuda()
        layer = torch.arange(p.n_layers, device="cuda") * (p.blocks_per_layer * p.heads)
        head = torch.arange(p.heads, device="cuda")
        out.append((base + (blocks[:, None] * p.heads)[:, None, :] + layer[None, :, None]
                    + head[None, None, :]).reshape(-1))
    return torch.cat(out)


class _Engine:
    """A pool with its traces: what a serving engine holds between two epochs."""

    def __init__(self, case, seed):
        self.case = case
        r = np.random.default_rng(seed)
        g = torch.Generator(device="cuda").manual_seed(seed)
        step = case["kind"] == "step"
        self.parts = parts = _partitions(case)
        self.n = n = sum(p.n_entries for p in parts)
        self.k = k = _victims(case)
        self.k_blocks = k // parts[0].heads if case["kind"] == "blocks" else 0
        entry = max(p.entry_bytes for p in parts)
        staging = max(case.get("batch_mb", 0) << 20, 2 * entry) + (case.get("batch_mb", 0) << 20) // entry * 24 + 4096
        self.batch = case.get("batch_mb", 0) << 20
        self.m = min(int(case.get("promote", 0) * n), k // 2) if step else 0
        # handles for as many epochs as a long-running measurement makes (they are never reused)
        tags = n + 64 + (k * min(60_000, (1 << 27) // k) if step else 0)
        self.pool = p = B.Pool(parts, tags, staging_bytes=staging, max_promote=max(4096, self.m + 16),
                               host_meta=step, stream=_compute())
        for ring in p.rings:
            ring.zero_()
        bases = np.concatenate([[0], np.cumsum([q.n_entries for q in parts])])[:-1].tolist()
        if case["arch"] == "fleet":
            weights = torch.from_numpy(np.random.default_rng(seed + 1).dirichlet(np.full(16, 0.5))).cuda()
            pairs = torch.multinomial(weights, n + 16, replacement=True, generator=g).to(torch.uint8)
        else:
            pairs = torch.randint(0, 16, (n + 16,), dtype=torch.uint8, device="cuda", generator=g)
        self.pairs = pairs
        torch.cuda.synchronize()
        _ok(p.kv_admit(0, DECAY, pairs, True)[0], "kv_admit")
        _ok(p.kv_set_policy(case["policy"]), "kv_set_policy")
        if case["blend"]:
            _ok(p.kv_set_confidence_blend(KAPPA, WINDOW), "kv_set_confidence_blend")
        if case.get("deferred"):
            _ok(p.kv_set_deferred_packing(True), "kv_set_deferred_packing")
        # each trace: the touches, then the slots that the epoch before has freed (its victims)
        self.traces = []
        for _ in range(TRACES):
            ids = _touches(case["style"], parts, bases, r)
            head = ids.numel() // 4 * 4
            trace = torch.empty(head + k, dtype=torch.int32, device="cuda")
            trace[:head] = ids[:head].to(torch.int32)
            hit = torch.zeros(head + k, dtype=torch.uint8, device="cuda")
            chance = (pairs[ids[:head]].float() + 0.5) / 16.0
            hit[:head] = (torch.rand(head, device="cuda", generator=g) < chance).to(torch.uint8)
            trace[head:] = torch.randperm(n, device="cuda", generator=g)[:k].to(torch.int32)
            self.traces.append((trace, hit, trace[head:]))
            del ids, chance
        self.observed = []
        if case["weights"]:
            for _ in range(TRACES):
                self.observed.append([torch.exp(torch.randn(q.n_layers, 1 if q.variant == W.MLA else q.n_q_heads,
                                                            device="cuda", generator=g)) for q in parts])
        self.promote_at = self._promote_order(r) if step else None
        self.epoch, self.cursor = 0, 0
        torch.cuda.synchronize()
        for _ in range(WARM_EPOCHS):
            self.one_pass()
        torch.cuda.synchronize()

    def _promote_order(self, r):
        """Places, among the k slots that one demotion fills, of the blocks to bring back."""
        k, m, order = self.k, self.m, self.case["order"]
        if order == "recent":      # what has just left
            return np.arange(k - m, k, dtype=np.uint64)
        if order == "runs":        # runs of up to 2,048 slots at random places
            run = max(1, min(2048, m // 4))
            rows = r.permutation(k // run)[: -(-m // run)]
            return (rows[:, None] * run + np.arange(run)[None, :]).reshape(-1)[:m].astype(np.uint64)
        # position order: a block's heads are neighbours, its layers a stripe apart
        p = self.parts[0]
        stripe = k // p.n_layers // p.heads
        if stripe == 0:
            return r.permutation(k)[:m].astype(np.uint64)
        at = (r.permutation(stripe)[:, None, None] * p.heads + np.arange(p.n_layers)[None, :, None] * (stripe * p.heads)
              + np.arange(p.heads)[None, None, :])
        return at.reshape(-1)[:m].astype(np.uint64)

    def one_pass(self):
        case, p, k = self.case, self.pool, self.k
        trace, hit, _ = self.traces[self.epoch % TRACES]
        self.epoch += 1
        victims = self.traces[self.epoch % TRACES][2]
        if self.observed:
            for q, x in enumerate(self.observed[self.epoch % TRACES]):
                _ok(p.kv_head_importance_update(q, x, DECAY), "kv_head_importance_update")
        kind = case["kind"]
        if kind == "split":
            _ok(p.kv_epoch_events(trace, hit), "kv_epoch_events")
            _ok(p.kv_epoch_update(self.epoch), "kv_epoch_update")
            _ok(p.kv_select_victims(k, victims), "kv_select_victims")
        elif kind == "blocks":
            _ok(p.kv_epoch_score(self.epoch, trace, hit), "kv_epoch_score")
            _ok(p.kv_select_victim_blocks(self.k_blocks, victims)[0], "kv_select_victim_blocks")
        else:
            _ok(p.kv_epoch_score_select(self.epoch, trace, hit, trace.numel(), k, victims), "kv_epoch_score_select")
        if kind == "step":
            ring = self.parts[0].ring_slots
            # what is brought back left one epoch ago, or just now (nothing has left before the first epoch)
            left = self.cursor if case["order"] == "recent" else self.cursor - k
            _ok(p.kv_demote(victims, k, self.batch), "kv_demote")
            if self.m and left >= 0:
                _ok(p.kv_promote(0, (self.promote_at + np.uint64(left)) % np.uint64(ring), self.batch), "kv_promote")
            _ok(p.kv_flush(), "kv_flush")
            self.cursor += k
            _ok(p.kv_admit(self.epoch, DECAY, self.pairs, False)[0], "kv_admit")
        n = self.n
        out = {"victims": victims, "score": p.score[:n], "ema": p.ema[:n], "last_epoch": p.last_epoch[:n],
               "touch": p.touch[:n], "hits": p.hits, "misses": p.misses, "P": p.P}
        if self.observed:
            out["importance"] = [p.kv_head_importance(q) for q in range(len(self.parts))]
        if kind == "step":
            out.update(tag=p.tag[:n], pair=p.pair[:n], state=p.state[:n], slab=p.slabs[0].view(torch.int64),
                       ring=p.rings[0].view(torch.int64), ring_meta=p.metas[0])
        return out


class _Static:
    """Scores and states of somebody else's cache: recency classes times sixteen reuse probabilities."""

    def __init__(self, case, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        self.k = _victims(case)
        self.arrays = []
        for _ in range(TRACES):
            age = torch.randint(0, 16, (n,), device="cuda", generator=g).float()
            pair = torch.randint(0, 16, (n,), device="cuda", generator=g).float()
            noise = torch.rand(n, device="cuda", generator=g)
            own = torch.rand(n, device="cuda", generator=g) < 0.5     # half of the entries share their class's score
            score = DECAY ** age * (pair + 0.5) / 16.0 * torch.where(own, 1.0 + 0.3 * noise, torch.ones_like(noise))
            state = (torch.rand(n, device="cuda", generator=g) > 0.01).to(torch.uint8)
            score = torch.where(state != 0, score, torch.full_like(score, math.inf))
            self.arrays.append((score, state))
        self.victims = torch.empty(self.k, dtype=torch.int32, device="cuda")
        self.status = torch.zeros(4, dtype=torch.int32, device="cuda")
        self.at = 0

    def one_pass(self):
        score, state = self.arrays[self.at % TRACES]
        self.at += 1
        _ok(B.kv_select_victims_static(score, state, score.numel(), self.k, self.victims, self.status,
                                       _compute()), "kv_select_victims_static")
        return {"victims": self.victims, "status": self.status}


class _Hash:
    """New blocks of a pool, two fifths of them with the content of another block (shared prefixes)."""

    def __init__(self, case, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        part = _partition(case["arch"], case["layers"], case["heads"], case["blocks"], case["q_heads"], case["head_dim"],
                          case["block_tokens"])
        self.pool = B.Pool([part], part.n_entries, staging_bytes=part.entry_bytes + 4096, max_promote=64,
                           host_meta=False, stream=_compute())
        blocks = part.n_layers * part.blocks_per_layer
        slab = self.pool.slabs[0].view(torch.int64).view(blocks, -1)
        for lo in range(0, blocks, 1 << 14):
            slab[lo:lo + (1 << 14)].random_(generator=g)
        copies = torch.randperm(blocks, device="cuda", generator=g)[: 2 * blocks // 5]
        slab[copies] = slab[copies[torch.randint(0, max(1, copies.numel() // 2), (copies.numel(),), device="cuda", generator=g)]]
        m = case["hashed"]
        self.m = m
        self.ids = torch.randperm(part.n_entries, device="cuda", generator=g)[:m].sort().values.to(torch.int32)
        self.digests = torch.empty((m, 32), dtype=torch.uint8, device="cuda")
        self.canon = torch.empty(m, dtype=torch.int32, device="cuda")
        self.refs = torch.empty(m, dtype=torch.int32, device="cuda")
        self.table = torch.empty(B.kv_dedup_table_slots(m), dtype=torch.int32, device="cuda")
        self.unique = torch.zeros(4, dtype=torch.int32, device="cuda")
        self.status = torch.zeros(4, dtype=torch.int32, device="cuda")

    def one_pass(self):
        p = self.pool
        _ok(p.kv_hash_entries(self.ids, self.m, self.digests), "kv_hash_entries")
        _ok(B.kv_dedup_digests(self.digests, self.m, self.canon, self.refs, self.table, self.unique, self.status, p.compute),
            "kv_dedup_digests")
        return {"digests": self.digests, "canon": self.canon, "refcount": self.refs, "unique": self.unique[:1]}


class _Prefetch:
    """Long sequences of which a share of the blocks has gone to the host."""

    def __init__(self, case, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        layers, heads, nb, n_pos = case["layers"], case["heads"], case["blocks"], case["n_pos"]
        n = layers * heads * nb
        self.case = case
        part = _partition("gqa" if heads > 1 else "mqa", layers, heads, nb, ring=int(n * case["away"]) + 64)
        self.pool = p = B.Pool([part], n + 64, staging_bytes=8 << 20, max_promote=4096, host_meta=False,
                               stream=_compute())
        pairs = torch.randint(0, 16, (n + 16,), dtype=torch.uint8, device="cuda", generator=g)
        # block handles were given out in (layer, block, head) order; a sequence owns scattered blocks
        perm = torch.randperm(nb, device="cuda", generator=g)
        layer = torch.arange(layers, device="cuda")[None, :, None] * (nb * heads)
        head = torch.arange(heads, device="cuda")[None, None, :]
        self.tables = [(perm[s * n_pos:(s + 1) * n_pos, None, None] * heads + layer + head).to(torch.int32).contiguous()
                       for s in range(case["sequences"])]
        gone = (torch.rand((layers, nb), device="cuda", generator=g) < case["away"] * 0.95).nonzero()
        gone = ((gone[:, 0] * nb + gone[:, 1]) * heads)[:, None] + torch.arange(heads, device="cuda")[None, :]
        gone = gone.reshape(-1)[: part.ring_slots].to(torch.int32)
        # local layers look a few hundred tokens back, global ones thousands
        self.spans = [(128.0 * 2.0 ** (5.0 * torch.arange(layers, device="cuda") / layers)
                       * torch.exp(0.2 * torch.randn(layers, device="cuda", generator=g))).float() for _ in range(TRACES)]
        self.slots = [torch.full((n_pos * layers * heads,), -1, dtype=torch.int64, device="cuda") for _ in self.tables]
        self.counts = torch.zeros((case["sequences"], 2), dtype=torch.int64, device="cuda")
        self.pos = [int(x) for x in np.random.default_rng(seed).integers(0, n_pos, case["sequences"])]
        self.at = 0
        torch.cuda.synchronize()
        _ok(p.kv_admit(0, DECAY, pairs, False)[0], "kv_admit")
        if gone.numel():
            _ok(p.kv_demote(gone, gone.numel(), 4 << 20), "kv_demote")
        p.sync()

    def one_pass(self):
        p = self.pool
        _ok(p.kv_prefetch_window_update(0, self.spans[self.at % TRACES], DECAY), "kv_prefetch_window_update")
        self.at += 1
        n_pos = self.case["n_pos"]
        for s, table in enumerate(self.tables):
            pos = (self.pos[s] + self.at) % n_pos
            _ok(p.kv_prefetch_list(0, table, n_pos, pos, 1 if s % 2 else -1, self.slots[s], self.slots[s].numel(), self.counts[s]),
                "kv_prefetch_list")
        return {"slots": self.slots, "counts": self.counts, "window": p.kv_prefetch_window(0)}


_STATES = {"epoch": _Engine, "split": _Engine, "blocks": _Engine, "step": _Engine, "static": _Static, "hash": _Hash,
           "prefetch": _Prefetch}


def prepare(case, seed):
    # A pool initialises its memory on a stream of its own: nothing may still be reading what the
    # allocator hands it, and its first user may come from any stream.
    torch.cuda.synchronize()
    state = _STATES[case["kind"]](case, seed)
    torch.cuda.synchronize()
    return state


def run(state):
    return state.one_pass()


def _events(case):
    """Events of one trace, averaged over a few of them."""
    if case["style"] == "entry":
        return int(0.2 * _entries(case)) + _victims(case)
    total = 0
    for p in _partitions(case):
        r = np.random.default_rng(5)
        total += sum(len(_touched_blocks(case["style"], p, r)) for _ in range(4)) // 4 * p.n_layers * p.heads
    return total + _victims(case)


def work(case):
    kind = case["kind"]
    if kind == "static":      # score and state in, victims out
        return {"bytes": 5 * case["n"] + 4 * _victims(case), "flops": 0}
    if kind == "hash":        # block bytes and ids in, digest, canonical position and reference count out
        part = _partition(case["arch"], case["layers"], case["heads"], case["blocks"], case["q_heads"], case["head_dim"],
                          case["block_tokens"])
        return {"bytes": case["hashed"] * (part.entry_bytes + 4 + 32 + 8), "flops": 0}
    if kind == "prefetch":    # handle and location of every candidate inside the windows, slots out
        layers = case["layers"]
        blocks = sum(min(case["n_pos"] / 2, 8.0 * 2.0 ** (5.0 * l / layers)) for l in range(layers))
        return {"bytes": case["sequences"] * blocks * case["heads"] * (8 + 8 * case["away"]), "flops": 0}
    n, events, k = _entries(case), _events(case), _victims(case)
    # per entry: EMA in and out, decay, pair and state in, score out (LRU: the last epoch in);
    # per touched entry the last epoch out; per event its id and flag; the victims out
    size = n * (18 + (4 if case["policy"] == 2 else 0)) + 4 * min(n, events) + 5 * events + 4 * k
    if kind == "step":        # the bytes of the moved entries leave one memory and enter the other
        entry = _partitions(case)[0].entry_bytes
        m = min(int(case["promote"] * n), k // 2)
        size += 2 * entry * (k + m) + 60 * (k + m)
    return {"bytes": size, "flops": 5 * n}


def tolerance(case):
    # Every operation of the path is defined down to its rounding, ties are broken by id, and
    # counters are integers: another correct implementation gives the same bits.
    return "exact"
