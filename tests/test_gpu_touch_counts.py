"""Touch counts packed nine bits to an entry between the event reduction and the fused scoring pass:
counts that overflow, once and many times, on one entry, on neighbours and across words, and on the last
entries of an odd pool, against the oracle, bit for bit.  Counts that kv_epoch_events left in the
caller's array before such a call are added to it, and a pool whose touches have cooled down goes on.
"""
import numpy as np
import pytest

from oracle import kv_oracle as O
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


def trace(style, n, r):
    if style == "edges":       # counts around multiples of 512, a different one on each entry of a few words
        counts = np.zeros(n, np.int64)
        counts[:20] = [255, 256, 257, 0, 511, 512, 513, 255, 512, 512, 512, 512, 0, 511, 0, 65536 + 511, 511, 511, 511, 511]
        counts[n - 3:] = [512, 511, 513]
        return r.permutation(np.repeat(np.arange(n), counts))
    if style == "runs":        # blocks that report all their heads, some of them 600 times
        starts = np.repeat(np.arange(0, 64, 4), r.integers(400, 700, 16))
        return (r.permutation(starts)[:, None] + np.arange(4)[None, :]).reshape(-1)
    if style == "in order":    # one entry after the other: every addition of a warp on one word
        return np.repeat(np.arange(n - 8, n), r.integers(500, 2400, 8))
    return r.integers(0, 5, 200_000)      # "hot": 40,000 touches each of five neighbours


@pytest.mark.parametrize("call", ["score", "score_select", "events first"])
@pytest.mark.parametrize("style", ["edges", "runs", "in order", "hot"])
def test_counts_beyond_nine_bits(style, call):
    from lockstep import Lockstep
    w = W.Workload("counts", [W.gqa(3, 6, 3, 16, 8, 1237, 2000, "entry")], 0.05, 0.0, seed=7)   # 11,133 entries
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(len(style))
    for e in range(6):                                # (hot, hot, hot, cool, cool, hot)
        ev = (trace(style, w.N, r) if e not in (3, 4) else r.integers(0, w.N, 3001)).astype(np.uint32)
        hit = r.integers(0, 2, ev.size).astype(np.uint8)
        if call == "events first":                    # half of the trace through the caller's array
            h = ev.size // 2
            d_e, d_h, n = g.stage_events(ev[:h], hit[:h])
            g.check(g.pool.kv_epoch_events(d_e, d_h, n), "kv_epoch_events")
            g.pool.sync()
            assert np.array_equal(g.host_array("touch"), np.bincount(ev[:h], minlength=w.N))
        else:
            h = 0
        d_e, d_h, n = g.stage_events(ev[h:], hit[h:])
        if call == "score":
            g.check(g.pool.kv_epoch_score(e, d_e, d_h, n), "kv_epoch_score")
        else:
            g.check(g.pool.kv_epoch_score_select(e, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
        assert o.epoch_score(e, ev, hit) == O.OK
        ls.compare_state((style, call, e))
        if call != "score":
            rc, v = o.select_victims(w.k)
            assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v)
    ls.close()
