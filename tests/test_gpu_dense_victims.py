"""Victims of a warp's 1,024 entries leave through shared memory where they are more than 128 and fit: just
at these limits, up to all entries, on pools of one and of several rows, without and with a hint, against
a sort on the host (exact)."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_group", [1, 127, 128, 129, 130, 500, 1023, 1024])
@pytest.mark.parametrize("blocks", [9001, 21_000, 110_003])
def test_victims_per_group(blocks, per_group):
    import torch
    parts = [W.gqa(2, 4, 4, 16, 8, blocks, 16, "entry")]
    n = parts[0].n_entries
    r = np.random.default_rng(blocks + per_group)
    p = B.Pool(parts, n + 16, staging_bytes=4096, max_promote=64, host_meta=False)
    assert p.kv_admit(0, 0.9, torch.zeros(n + 16, dtype=torch.uint8, device="cuda"), False)[0] == 0
    p.sync()
    for again in range(2):
        order = np.argsort(np.concatenate([r.random(1024) for _ in range(-(-n // 1024))]).reshape(-1, 1024), axis=1)
        low = np.zeros(order.shape, bool)
        np.put_along_axis(low, order[:, :per_group], True, axis=1)
        low = low.reshape(-1)[:n]
        score = np.where(low, r.random(n) * 0.5, 1.0 + r.random(n)).astype(np.float32)
        k = int(low.sum()) - again          # (the second time one of the low ones stays)
        victims = torch.full((n + 4,), -1, dtype=torch.int32, device="cuda")
        p.score[:n] = torch.from_numpy(score).cuda()
        torch.cuda.synchronize()
        assert p.kv_select_victims(k, victims) == 0
        p.sync()
        got = victims.cpu().numpy()
        assert np.array_equal(got[:k], np.sort(np.argsort(score, kind="stable")[:k]))
        assert (got[k:] == -1).all()
    assert p.kv_device_status() == 0
    p.close()
