"""Which slots promotions and admissions fill.  The library knows the free slots of a partition
without looking for them as long as they are what one demotion left of a full partition, and looks
for them otherwise: after a demotion into a partition with holes, and after a selection or a hash
run has used the list's memory.  A model of the pool in numpy follows random sequences of those
calls; tags, block table, ring metadata and payload (a pattern per handle) are compared exactly."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


class Model:
    def __init__(self, parts):
        self.parts = parts
        self.base = np.cumsum([0] + [p.n_entries for p in parts])
        self.tag = np.full(self.base[-1], -1, np.int64)
        self.ring = [np.full(p.ring_slots, -1, np.int64) for p in parts]
        self.cursor = [0] * len(parts)
        self.next_tag = 0

    def free(self, q):
        return self.base[q] + np.flatnonzero(self.tag[self.base[q]:self.base[q + 1]] < 0)

    def admit(self):
        holes = np.flatnonzero(self.tag < 0)
        self.tag[holes] = self.next_tag + np.arange(holes.size)
        self.next_tag += holes.size

    def demote(self, victims):
        for q, p in enumerate(self.parts):
            v = victims[(victims >= self.base[q]) & (victims < self.base[q + 1])]
            slots = (self.cursor[q] + np.arange(v.size)) % p.ring_slots
            self.ring[q][slots] = self.tag[v]
            self.cursor[q] = int((self.cursor[q] + v.size) % p.ring_slots)
            self.tag[v] = -1

    def promote(self, q, slots):
        self.tag[self.free(q)[: slots.size]] = self.ring[q][slots]
        self.ring[q][slots] = -1


@pytest.mark.parametrize("deferred", [False, True])
@pytest.mark.parametrize("host_meta", [False, True])
@pytest.mark.parametrize("seed,batch", [(1, 20 << 10), (2, 20 << 10), (3, 20 << 10), (4, 512 << 10), (5, 512 << 10)])
def test_sequences(seed, batch, deferred, host_meta):
    """batch: several staged chunks per demotion, or (one chunk) stores straight into the ring."""
    import torch
    parts = [W.gqa(2, 8, 4, 16, 4, 331, 1500, "entry"), W.mla(3, 32, 32, 4, 517, 1100, "entry")]
    r = np.random.default_rng(seed)
    n = sum(p.n_entries for p in parts)
    p = B.Pool(parts, 60_000, staging_bytes=2 * batch + (64 << 10), max_promote=2048, host_meta=host_meta)
    pairs = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_set_deferred_packing(deferred) == 0
    m = Model(parts)
    assert p.kv_admit(0, 0.9, pairs, True)[0] == 0
    m.admit()
    scratch = torch.empty(n, dtype=torch.int32, device="cuda")
    keep = []
    for _ in range(40):
        op = r.choice(["demote", "demote", "promote", "promote", "promote", "select", "hash", "admit"])
        if op == "demote":
            live = np.flatnonzero(m.tag >= 0)
            v = np.sort(r.permutation(live)[: int(r.integers(1, 700))])
            d_v = torch.from_numpy(np.concatenate([v, np.zeros(4, np.int64)]).astype(np.int32)).cuda()
            keep.append(d_v)                      # (deferred packing reads it later)
            torch.cuda.synchronize()
            assert p.kv_demote(d_v, v.size, batch) == 0
            m.demote(v)
        elif op == "promote":
            q = int(r.integers(0, 2))
            held = np.flatnonzero(m.ring[q] >= 0)
            count = min(held.size, m.free(q).size, int(r.integers(1, 200)))
            if count == 0:
                continue
            start = int(r.integers(0, held.size - count + 1))
            slots = held[start:start + count] if r.random() < 0.5 else r.permutation(held)[:count]
            assert p.kv_promote(q, slots.astype(np.uint64), batch) == 0
            m.promote(q, slots)
        elif op == "select":
            resident = int((m.tag >= 0).sum())
            if resident:
                assert p.kv_select_victims(max(1, resident // 3), scratch) == 0
        elif op == "hash":
            out = torch.empty((n, 32), dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            assert p.kv_hash_entries(None, n, out) == 0
            p.sync()
        else:
            assert p.kv_admit(1, 0.9, pairs, True)[0] == 0
            m.admit()
    assert p.kv_flush() == 0
    p.sync()
    tag = p.tag[:n].cpu().numpy().astype(np.int64)
    assert np.array_equal(tag, m.tag)
    assert p.kv_device_status() == 0
    loc = p.loc[: m.next_tag].cpu().numpy().view(np.uint32).astype(np.int64)
    want = np.full(m.next_tag, 0xFFFFFFFF, np.int64)
    want[m.tag[m.tag >= 0]] = np.flatnonzero(m.tag >= 0)
    for q, part in enumerate(parts):
        held = np.flatnonzero(m.ring[q] >= 0)
        want[m.ring[q][held]] = held | 0x80000000
        if host_meta:
            assert np.array_equal(p.ring_meta(q)["tag"][held], m.ring[q][held].astype(np.uint32))
        ring = p.rings[q].numpy()[: part.ring_slots * part.entry_bytes].reshape(part.ring_slots, -1)
        assert np.array_equal(ring[held], W.pattern_bytes(m.ring[q][held], part.entry_bytes))
        chunks = 1 if part.variant == W.MLA else 2
        slab = p.slabs[q].cpu().numpy().reshape(-1, chunks, part.heads, part.entry_bytes // chunks)
        slab = np.ascontiguousarray(slab.transpose(0, 2, 1, 3)).reshape(part.n_entries, -1)
        own = m.tag[m.base[q]:m.base[q + 1]]
        assert np.array_equal(slab[own >= 0], W.pattern_bytes(own[own >= 0], part.entry_bytes))
    assert np.array_equal(loc, want)
    p.close()
