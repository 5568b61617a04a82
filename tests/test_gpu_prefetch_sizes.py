"""The one-launch prefetch list where its geometry changes: no candidate, less than one block's
tile of 1,024, table rows that are and are not vectors of four handles, more tiles than blocks
(a block then takes several), one launch right behind another.  The expected list is the
definition evaluated in numpy on the block table and windows; whole numbers, compared exactly."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


def expected(table, win, loc, pos0, direction):
    n_pos, layers, heads = table.shape
    reach = min(int(win.max()), n_pos - pos0 if direction > 0 else pos0 + 1)
    rows = pos0 + np.arange(reach) * (1 if direction > 0 else -1)
    t = table[rows].astype(np.int64)                                      # [distance][layer][head]
    inside = np.arange(reach)[:, None, None] < win[None, :, None]
    where = np.where(t < loc.size, loc[np.minimum(t, loc.size - 1)], 0xFFFFFFFF).astype(np.int64)
    hit = inside & (where != 0xFFFFFFFF) & ((where & 0x80000000) != 0)
    return (where[hit] & 0x7FFFFFFF).astype(np.uint64)


@pytest.mark.parametrize("layers,heads,n_pos,tokens", [(1, 1, 1, 16.0), (2, 4, 33, 400.0), (3, 3, 150, 900.0), (5, 1, 700, 3000.0),
                                                       (80, 8, 64, 600.0), (8, 8, 6100, 90000.0), (7, 7, 8000, 120000.0)])
def test_list_sizes(layers, heads, n_pos, tokens):
    import torch
    nb = n_pos + 5
    part = W.gqa(layers, 4 * heads, heads, 1, 16, nb, layers * heads * nb // 2 + 8)
    n = part.n_entries
    p = B.Pool([part], n + 64, staging_bytes=1 << 20, max_promote=64, host_meta=False)
    r = np.random.default_rng(n)
    pairs = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_admit(0, 0.9, pairs, False)[0] == 0
    gone = np.sort(r.permutation(n)[: n // 2]).astype(np.int32)
    d_gone = torch.from_numpy(np.concatenate([gone, np.zeros(4, np.int32)])).cuda()
    torch.cuda.synchronize()
    if gone.size:
        assert p.kv_demote(d_gone, gone.size, 1 << 19) == 0
    span = (r.random(layers) * tokens).astype(np.float32)
    assert p.kv_prefetch_window_update(0, torch.from_numpy(span).cuda(), 0.0) == 0
    table = np.ascontiguousarray(r.permutation(n)[: n_pos * layers * heads].reshape(n_pos, layers, heads).astype(np.uint32))
    table.reshape(-1)[r.integers(0, table.size, 3)] = np.array([0xFFFFFFFF, n + 64, n + 70], np.uint32)
    d_table = torch.from_numpy(table.view(np.int32)).cuda()
    calls = [(pos, d) for pos in sorted({0, n_pos // 2, n_pos - 1}) for d in (1, -1)]
    outs = [torch.full((table.size + 1,), -1, dtype=torch.int64, device="cuda") for _ in calls]
    counts = torch.full((len(calls) + 1,), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for i, (pos, d) in enumerate(calls):            # nothing waits between them
        assert p.kv_prefetch_list(0, d_table, n_pos, pos, d, outs[i], table.size, counts[i:]) == 0
    assert p.kv_prefetch_list(0, None, 0, 0, 1, None, 0, counts[len(calls):]) == 0
    p.sync()
    win = p.kv_prefetch_window(0).cpu().numpy().view(np.uint32).astype(np.int64)
    loc = p.loc[: n + 64].cpu().numpy().view(np.uint32)
    got_n = counts.cpu().numpy()
    for i, (pos, d) in enumerate(calls):
        want = expected(table, win, loc, pos, d)
        got = outs[i].cpu().numpy().view(np.uint64)
        assert got_n[i] == want.size, (pos, d)
        assert np.array_equal(got[: want.size], want), (pos, d)
        assert (got[want.size:] == np.uint64(0xFFFFFFFFFFFFFFFF)).all()
    assert got_n[-1] == 0 and p.kv_device_status() == 0
    p.close()
