"""The allocation-free selection where the keys that are left fit the list (up to 1,024 of them, after one
or two digits) and where they just do not: a planted band of scores, ties among them, spread over all
chunks of arrays of one to seven rows, against a sort on the host (exact)."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [1, 40, 900, 1 << 20])     # distinct keys of the band: one, few, a last bin's, a first digit's
@pytest.mark.parametrize("m", [1, 1023, 1024, 1025, 5000])
@pytest.mark.parametrize("n", [8193, 20_001, 700_003, 4_194_304])
def test_band(n, m, width):
    import torch
    r = np.random.default_rng(n + m + width)
    score = r.random(n, dtype=np.float32) * np.float32(0.2)                 # below the band ...
    score[r.random(n) < 0.6] += np.float32(4.0)                             # ... and above it
    at = r.choice(n, m, replace=False)
    score[at] = (np.uint32(0x3F800000) + r.integers(0, width, m).astype(np.uint32)).view(np.float32)
    state = (r.random(n) < 0.95).astype(np.uint8)
    state[at[: max(1, m // 2)]] = 1
    resident = np.flatnonzero(state)
    below = int((score[resident] < 0.5).sum())
    band = int(((score[resident] >= 1.0) & (score[resident] < 2.0)).sum())
    d_score, d_state = torch.from_numpy(score).cuda(), torch.from_numpy(state).cuda()
    order = resident[np.argsort(score[resident], kind="stable")]
    for k in sorted({below + 1, below + (band + 1) // 2, below + band}):
        victims = torch.full((k + 4,), -1, dtype=torch.int32, device="cuda")
        status = torch.zeros(4, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert B.kv_select_victims_static(d_score, d_state, n, k, victims, status) == 0
        torch.cuda.synchronize()
        assert int(status[0].item()) == 0
        got = victims.cpu().numpy()
        assert np.array_equal(got[:k], np.sort(order[:k])), k
        assert (got[k:] == -1).all()
