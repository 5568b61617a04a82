"""The event reduction against plain counting: touch counts per entry and (pair, hit) counts are
whole numbers and have to be equal.  Trace lengths around a vector of four, a block's share and
one pass of the whole grid; aligned runs, broken runs, isolated and repeated entries, and the last
entry of an odd pool."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

BLOCK = 512 * 4                # events of one block's vectors
GRID = BLOCK * 296             # events of one vector for every thread of the grid


def trace(style, n, n_events, r):
    if style == "single":
        return r.integers(0, n, n_events)
    if style == "hot":           # a few entries take all touches, the pool's last one among them
        return r.choice(np.array([0, 1, n // 2, n - 2, n - 1]), n_events)
    length = 32 if style == "runs" else 7        # "broken": runs that start anywhere and end inside a vector
    starts = r.integers(0, n // length, -(-n_events // length)) * length + (r.integers(0, 4) if style == "broken" else 0)
    return np.minimum((starts[:, None] + np.arange(length)[None, :]).reshape(-1)[:n_events], n - 1)


@pytest.mark.parametrize("style", ["single", "hot", "runs", "broken"])
@pytest.mark.parametrize("n_events", [1, 3, 4, 7, 128, BLOCK - 4, BLOCK, BLOCK + 5, GRID - 1, GRID + 4, 3 * GRID + 1234, 9 * GRID + 6, 21 * GRID - 2])
def test_counts(style, n_events):
    import torch
    parts = [W.gqa(3, 6, 3, 16, 8, 7001, 16, "entry")]      # 63,009 entries
    n = parts[0].n_entries
    r = np.random.default_rng(n_events)
    pairs = r.integers(0, 16, n + 16).astype(np.uint8)
    d_pairs = torch.from_numpy(pairs).cuda()
    torch.cuda.synchronize()
    p = B.Pool(parts, n + 16, staging_bytes=4096, max_promote=64, host_meta=False)
    assert p.kv_admit(0, 0.9, d_pairs, False)[0] == 0
    ids = trace(style, n, n_events, r).astype(np.uint32)
    hit = r.integers(0, 3, n_events).astype(np.uint8)          # any non-zero flag is a hit
    d_ids = torch.zeros(n_events + 4, dtype=torch.int32, device="cuda")
    d_hit = torch.zeros(n_events + 16, dtype=torch.uint8, device="cuda")
    d_ids[:n_events] = torch.from_numpy(ids.view(np.int32))
    d_hit[:n_events] = torch.from_numpy(hit)
    torch.cuda.synchronize()
    assert p.kv_epoch_events(d_ids, d_hit, n_events) == 0
    p.sync()
    assert np.array_equal(p.touch[:n].cpu().numpy(), np.bincount(ids, minlength=n))
    want = np.bincount(2 * pairs[ids].astype(np.int64) + (hit != 0), minlength=32)
    assert np.array_equal(p.kv_epoch_counts().cpu().numpy(), want)
    assert p.kv_device_status() == 0
    p.close()
