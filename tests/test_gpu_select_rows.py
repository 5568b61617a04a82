"""The persistent selection at the edges of its geometry: rows of one 4,096-entry chunk per SM and
a last, shorter row of equal pieces (multiples of 128 entries), from one entry to more rows than a
warp has lanes, with and without a hint, and replayed from a captured graph.

The expected victims come from a stable sort of (key, id), i.e. the definition of the selection;
they are whole numbers, so the comparison is exact."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

CHUNK, SMS = 4096, 148
ROW = CHUNK * SMS


def expected(score, state, k):
    ids = np.flatnonzero(state != 0)
    order = np.argsort(score[ids] + np.float32(0.0), kind="stable")   # (-0 and +0 tie)
    return np.sort(ids[order[:k]]).astype(np.uint32)


def draw(n, seed, scale=1.0):
    r = np.random.default_rng(seed)
    score = r.uniform(0.5, 2.0, n).astype(np.float32)
    tied = r.random(n) < 0.4
    score[tied] = np.float32(0.75)                       # a heavy tie near the tenth percentile
    score[r.random(n) < 0.01] *= np.float32(-1.0)
    return (score * np.float32(scale)).astype(np.float32)


@pytest.mark.parametrize("n", [1, 3, 5, 127, 128, 129, 1024, 1025, CHUNK - 1, CHUNK + 1, 37 * 1024 + 11, ROW - 1, ROW,
                               ROW + 1, ROW + 128 * SMS, ROW + 128 * SMS + 1, 2 * ROW + 77, 1 << 22])
def test_static_selection_sizes(n):
    import torch
    state = (np.random.default_rng(n).random(n) > 0.02).astype(np.uint8)
    resident = int(state.sum())
    d_state = torch.from_numpy(state).cuda()
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    for call, k in enumerate(sorted({1, max(1, resident // 10), max(1, resident // 2), resident})):
        if k > resident:
            continue
        score = draw(n, 17 * call + n)
        score[state == 0] = np.inf
        out = torch.full((k + 4,), -1, dtype=torch.int32, device="cuda")
        d_score = torch.from_numpy(score).cuda()
        torch.cuda.synchronize()
        assert B.kv_select_victims_static(d_score, d_state, n, k, out, status, torch.cuda.current_stream()) == 0
        torch.cuda.synchronize()
        assert np.array_equal(out[:k].cpu().numpy().view(np.uint32), expected(score, state, k)), (n, k)
        assert (out[k:] == -1).all()
    assert int(status[0]) == 0


@pytest.mark.parametrize("n_rows,rest", [(0, 4096 * 3 + 256), (1, 0), (3, 5000), (5, ROW - 3200), (32, 0), (33, 640)])
def test_hinted_selection_rows(n_rows, rest):
    """Drifting scores keep the threshold inside the hint's bracket; a jump leaves it."""
    import torch
    blocks = (n_rows * ROW + rest) // 2
    w = W.Workload("rows", [W.gqa(1, 4, 2, 4, 2, blocks, 16, "entry")], 0.1, 0.0, seed=3)
    p = B.Pool(w.parts, w.N + 16, staging_bytes=4096, max_promote=64, host_meta=False)
    n = w.N
    p.sync()
    pairs = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_admit(0, 0.9, pairs, False)[0] == 0
    p.sync()
    state = np.ones(n, np.uint8)
    base = draw(n, n)
    scales = [1.0, 1.01, 1.02, 1.03, 30.0, 30.1] if n_rows < 32 else [1.0, 1.01, 1.02]
    for i, scale in enumerate(scales):
        k = n // 10 + i
        score = (base * np.float32(scale)).astype(np.float32)
        out = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        p.score[:n].copy_(torch.from_numpy(score))
        torch.cuda.synchronize()
        assert p.kv_select_victims(k, out) == 0
        p.sync()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), expected(score, state, k)), (n_rows, rest, i)
        assert p.kv_device_status() == 0
    st = p.kv_selection_stats()
    assert st["selections"] == len(scales) and st["hint_hits"] >= 2
    p.close()


def expected_by_bits(score, state, k):
    """Scores ordered by their bits: NaNs with the sign bit lie below -inf, the others above +inf."""
    b = (score + np.float32(0.0)).view(np.uint32).astype(np.int64)
    b = np.where(np.isnan(score), score.view(np.uint32), b)
    key = np.where(b >> 31, 0xFFFFFFFF - b, b + 0x80000000)
    ids = np.flatnonzero(state != 0)
    return np.sort(ids[np.argsort(key[ids], kind="stable")[:k]]).astype(np.uint32)


def with_nans(n, seed):
    r = np.random.default_rng(seed)
    score = draw(n, seed)
    at = r.permutation(n)
    bits = score.view(np.uint32)
    few = max(1, n // 50)
    for i, special in enumerate((0x7FC00000, 0xFFC00000, 0x7FFFFFFF, 0xFFFFFFFF, 0x7F800000, 0xFF800000, 0x80000000, 0)):
        bits[at[i * few:(i + 1) * few]] = special
    return score


@pytest.mark.parametrize("n", [1000, 8192, 37 * 1024 + 11, ROW + 999])
def test_scores_that_are_not_numbers(n):
    """A caller's array may hold them; they have their places in the order like all others."""
    import torch
    state = (np.random.default_rng(n).random(n) > 0.02).astype(np.uint8)
    score = with_nans(n, 5)
    resident = int(state.sum())
    d_score, d_state = torch.from_numpy(score).cuda(), torch.from_numpy(state).cuda()
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    for k in (1, n // 100, n // 10, n // 2, resident - 3, resident):
        out = torch.full((k + 4,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert B.kv_select_victims_static(d_score, d_state, n, k, out, status, torch.cuda.current_stream()) == 0
        torch.cuda.synchronize()
        assert np.array_equal(out[:k].cpu().numpy().view(np.uint32), expected_by_bits(score, state, k)), k
    assert int(status[0]) == 0


@pytest.mark.parametrize("variant", [0, 1])
def test_scores_that_are_not_numbers_in_a_pool(variant):
    """The same with thresholds taken from the selection before (variant 1)."""
    import torch
    w = W.Workload("rows", [W.gqa(1, 4, 2, 4, 2, 50_003, 16, "entry")], 0.1, 0.0, seed=3)
    p = B.Pool(w.parts, w.N + 16, staging_bytes=4096, max_promote=64, host_meta=False)
    pairs = torch.zeros(w.N + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_set_select_variant(variant) == 0
    assert p.kv_admit(0, 0.9, pairs, False)[0] == 0
    p.sync()
    state = np.ones(w.N, np.uint8)
    for i, k in enumerate((w.N // 5, w.N // 5 + 7, w.N // 5 + 9, w.N // 100, w.N - 5, w.N)):
        score = with_nans(w.N, 9 + i // 4)
        out = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        p.score[:w.N].copy_(torch.from_numpy(score))
        torch.cuda.synchronize()
        assert p.kv_select_victims(k, out) == 0
        p.sync()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), expected_by_bits(score, state, k)), (i, k)
        assert p.kv_device_status() == 0
    assert variant == 0 or p.kv_selection_stats()["hint_hits"] >= 1
    p.close()


def test_captured_selection_can_be_replayed():
    import torch
    n, k = ROW + 999, 20_000
    state = np.ones(n, np.uint8)
    d_score, d_state = torch.empty(n, device="cuda"), torch.from_numpy(state).cuda()
    out = torch.empty(k, dtype=torch.int32, device="cuda")
    d_score.copy_(torch.from_numpy(draw(n, 1)))
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    assert B.kv_select_victims_static(d_score, d_state, n, k, out, None, s) == 0   # first call outside the capture
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert B.kv_select_victims_static(d_score, d_state, n, k, out, None, s) == 0
    for seed in (2, 3, 4):
        score = draw(n, seed, scale=seed)
        d_score.copy_(torch.from_numpy(score))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), expected(score, state, k)), seed
