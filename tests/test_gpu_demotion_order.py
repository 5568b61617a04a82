"""Demotions small enough to be stored straight into the ring, behind one of 64 MB whose transfer is
still under way: promotions of slots of either, and small demotions that reach the large one's slots
around the ring, find and leave the right bytes (a pattern per handle; exact)."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

LARGE, SMALL, EB = 1000, 8, 65536


@pytest.mark.parametrize("gather", [0, 1 << 20])
@pytest.mark.parametrize("deferred", [False, True])
@pytest.mark.parametrize("smalls,ring", [(1, 1500), (2, 1500), (3, 1010)])
def test_slots_of_both(smalls, ring, deferred, gather):
    import torch
    part = W.gqa(2, 4, 2, 128, 128, 300, ring, "entry")
    assert part.entry_bytes == EB
    batch = LARGE * EB
    p = B.Pool([part], 8192, staging_bytes=batch + LARGE * 24 + 4096, max_promote=4096, host_meta=True)
    p.rings[0].zero_()
    n = part.n_entries
    pairs = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_set_deferred_packing(deferred) == 0
    assert p.kv_set_gather_threshold(gather) == 0
    assert p.kv_admit(0, 0.9, pairs, True)[0] == 0
    lists = [torch.arange(LARGE, dtype=torch.int32, device="cuda")]
    lists += [torch.arange(LARGE + SMALL * i, LARGE + SMALL * (i + 1), dtype=torch.int32, device="cuda") for i in range(smalls)]
    torch.cuda.synchronize()
    held = np.full(ring, -1, np.int64)
    at = 0
    for d_v in lists:   # (tags are the entry ids after the first admission)
        assert p.kv_demote(d_v, d_v.numel(), batch) == 0
        held[(at + np.arange(d_v.numel())) % ring] = np.arange(at, at + d_v.numel())
        at += d_v.numel()
    # the end of the large demotion and the slots of the last small one
    slots = np.concatenate([np.arange(LARGE - 10, LARGE), (at - SMALL + np.arange(SMALL)) % ring]).astype(np.uint64)
    want = held[slots.astype(np.int64)]
    assert p.kv_promote(0, slots, batch) == 0
    assert p.kv_flush() == 0
    p.sync()
    slab = p.slabs[0].cpu().numpy().reshape(-1, 2, part.heads, EB // 2)
    slab = np.ascontiguousarray(slab.transpose(0, 2, 1, 3)).reshape(n, EB)
    tag = p.tag[:slots.size].cpu().numpy()
    assert np.array_equal(tag, want)
    assert np.array_equal(slab[:slots.size], W.pattern_bytes(want, EB))
    held[slots.astype(np.int64)] = -1
    full = np.flatnonzero(held >= 0)
    got = p.rings[0].numpy()[: ring * EB].reshape(ring, EB)
    assert np.array_equal(got[full], W.pattern_bytes(held[full], EB))
    assert np.array_equal(p.ring_meta(0)["tag"][full], held[full].astype(np.uint32))
    assert p.kv_device_status() == 0
    p.close()
