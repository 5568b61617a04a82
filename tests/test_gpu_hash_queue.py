"""Content hashes at the numbers of entries where the kernel starts to pass its chains of messages
from warp to warp (more than two blocks of 128 messages per SM, not a multiple of that), with
messages of one and of several lengths in a chain, against hashlib.  Digests are bytes: exact."""
import hashlib

import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

FULL = 128 * 148


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("m", [2 * FULL, 2 * FULL + 1, 3 * FULL + 77, 5 * FULL + 128 * 9, 7 * FULL - 3])
def test_digests(m, mixed):
    import torch
    # images of 96 and 512 bytes (last blocks of 32 and 0 bytes), and an MLA one of 1,168
    parts = [W.gqa(2, 4, 2, 8, 16, m // (6 if mixed else 4) + 3, 16, "entry")]
    if mixed:
        parts += [W.gqa(3, 4, 2, 4, 6, m // 12 + 2, 16, "entry"), W.mla(1, 32, 41, 8, m // 3, 16, "entry")]
    p = B.Pool(parts, sum(q.n_entries for q in parts) + 16, staging_bytes=1 << 16, max_promote=64, host_meta=False)
    r = np.random.default_rng(m)
    torch.cuda.synchronize()
    images, base = [], 0
    for q, part in enumerate(parts):
        raw = r.integers(0, 256, p.slabs[q].numel(), dtype=np.uint8)
        p.slabs[q].copy_(torch.from_numpy(raw))
        chunks = 1 if part.variant == W.MLA else 2
        x = raw.reshape(-1, chunks, part.heads, part.entry_bytes // chunks)
        images.append((base, np.ascontiguousarray(x.transpose(0, 2, 1, 3)).reshape(part.n_entries, part.entry_bytes)))
        base += part.n_entries
    assert p.N >= m
    ids = r.permutation(p.N)[:m].astype(np.uint32)
    ids[-1] = ids[0]
    d_ids = torch.from_numpy(ids.view(np.int32)).cuda()
    out = torch.zeros((m, 32), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for d in (d_ids, None):
        out.zero_()
        torch.cuda.synchronize()
        assert p.kv_hash_entries(d, m, out) == 0
        p.sync()
        got = out.cpu().numpy()
        which = ids if d is not None else np.arange(m)
        for j in range(m):
            lo, img = next(x for x in reversed(images) if which[j] >= x[0])
            assert got[j].tobytes() == hashlib.sha256(img[which[j] - lo].tobytes()).digest(), j
    assert p.kv_device_status() == 0
    p.close()


def test_lists_of_falling_length_on_one_pool(monkeypatch):
    """The queue's memory is as an earlier, longer call left it, and before the first call as the
    caller handed it over (here: ones in every bit).  Images of 8 KB: chains are queued again so
    often that the places that warps take reach beyond the ring."""
    import torch
    real = torch.empty

    def ones(*a, **k):
        t = real(*a, **k)
        return t.fill_(255) if t.dtype == torch.uint8 else t

    part = W.gqa(2, 8, 2, 128, 16, 30_000, 16, "entry")
    monkeypatch.setattr(torch, "empty", ones)
    p = B.Pool([part], part.n_entries + 16, staging_bytes=1 << 16, max_promote=64, host_meta=False)
    monkeypatch.undo()
    assert part.entry_bytes == 8192 and p.N == 120_000
    g = torch.Generator(device="cuda").manual_seed(5)
    p.slabs[0].copy_(torch.randint(0, 256, (p.slabs[0].numel(),), dtype=torch.uint8, device="cuda", generator=g))
    raw = p.slabs[0].cpu().numpy().reshape(-1, 2, part.heads, part.entry_bytes // 2)
    img = np.ascontiguousarray(raw.transpose(0, 2, 1, 3)).reshape(part.n_entries, part.entry_bytes)
    want = np.frombuffer(b"".join(hashlib.sha256(x).digest() for x in img), np.uint8).reshape(-1, 32)
    out = torch.zeros((p.N, 32), dtype=torch.uint8, device="cuda")
    for m in (120_000, 78_643, 60_000, 37_889, 120_000, 37_889):
        out.zero_()
        torch.cuda.synchronize()
        assert p.kv_hash_entries(None, m, out) == 0
        p.sync()
        assert np.array_equal(out[:m].cpu().numpy(), want[:m]), m
        assert not out[m:].any()
    assert p.kv_device_status() == 0
    p.close()
