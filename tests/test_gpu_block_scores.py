"""Block-granular selection over head counts that are and are not whole vectors of four entries,
pools whose blocks straddle partitions inside a vector, ragged ends, blocks with FREE heads and
heavy ties, with and without a hint.  The expected blocks come from the definition: heads added in
order in binary32, weight multiplied in, the k lowest by (score, index); ids compared exactly."""
import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


def expected(parts, score, state, k):
    key, heads, first = [], [], []
    base = 0
    for p in parts:
        H, n = p.heads, p.n_entries
        s = score[base:base + n].reshape(-1, H)
        total = np.zeros(s.shape[0], np.float32)
        for h in range(H):
            total = (total + s[:, h]).astype(np.float32)
        total = (total * np.float32((p.n_q_heads // H) if p.variant != W.MLA else p.n_q_heads)).astype(np.float32)
        total[(state[base:base + n].reshape(-1, H) == 0).any(axis=1)] = np.nan      # no candidate
        key.append(total)
        heads.append(np.full(total.size, H))
        first.append(base + np.arange(total.size) * H)
        base += n
    key, heads, first = np.concatenate(key), np.concatenate(heads), np.concatenate(first)
    order = np.argsort(key, kind="stable")                  # (NaN last)
    chosen = np.sort(order[:k])
    return np.concatenate([first[b] + np.arange(heads[b]) for b in chosen]).astype(np.uint32)


def pools():
    for H in (1, 2, 3, 4, 6, 8, 12):
        yield "gqa%d" % H, [W.gqa(2, 2 * H, H, 8, 4, 2713, 40000, "entry")]
    yield "mla", [W.mla(3, 16, 16, 8, 4099, 40000, "entry")]
    yield "mixed", [W.gqa(1, 6, 3, 8, 4, 1001, 9000, "entry"), W.mha(1, 4, 8, 4, 1002, 9000, "entry"),
                    W.mqa(3, 8, 8, 4, 333, 9000, "entry"), W.gqa(2, 16, 8, 8, 4, 501, 9000, "entry")]


@pytest.mark.parametrize("name,parts", list(pools()))
def test_block_scores(name, parts):
    import torch
    n = sum(p.n_entries for p in parts)
    p = B.Pool(parts, n + 64, staging_bytes=1 << 20, max_promote=64, host_meta=False)
    r = np.random.default_rng(n)
    pairs = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert p.kv_admit(0, 0.9, pairs, False)[0] == 0
    gone = np.sort(r.permutation(n)[: n // 40]).astype(np.int32)
    d_gone = torch.from_numpy(np.concatenate([gone, np.zeros(4, np.int32)])).cuda()
    torch.cuda.synchronize()
    assert p.kv_demote(d_gone, gone.size, 1 << 19) == 0
    p.sync()
    state = p.state[:n].cpu().numpy()
    blocks = sum(q.n_layers * q.blocks_per_layer for q in parts)
    base = r.choice(np.array([0.25, 0.5, 1.0, 1.5, 3.0], np.float32), n) * r.choice(np.array([1.0, 1.0, 1.1], np.float32), n)
    out = torch.empty(n + 16, dtype=torch.int32, device="cuda")
    for i, scale in enumerate([1.0, 1.001, 1.002, 7.0]):
        k = blocks // 9 + i
        score = (base * np.float32(scale)).astype(np.float32)
        p.score[:n].copy_(torch.from_numpy(score))
        out.fill_(-1)
        torch.cuda.synchronize()
        want = expected(parts, score, state, k)
        rc, got_n = p.kv_select_victim_blocks(k, out, wait=True)
        assert rc == 0
        p.sync()
        assert got_n == want.size and sum(p.kv_victim_counts()) == want.size
        assert np.array_equal(out[:got_n].cpu().numpy().view(np.uint32), want), (name, i)
        assert p.kv_device_status() == 0
    p.close()
