"""Touch counts that stand in the caller's array when a scoring pass begins -- put there by the caller's own
kernel or back from a copy, not by kv_epoch_events -- are that epoch's touches like any others: every call
that scores takes them up, adds its trace's to them and clears them, against the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import kv_oracle as O
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [0, 1, 2])
@pytest.mark.parametrize("blocks", [5, 1237, 60_001])        # one CTA, one row, several rows; odd sizes
@pytest.mark.parametrize("call", ["score", "score_select", "no trace", "overflow"])
def test_counts_of_the_caller(call, blocks, policy):
    from lockstep import Lockstep
    w = W.Workload("array", [W.gqa(3, 6, 3, 16, 8, blocks, max(64, blocks), "entry")], 0.05, 0.0, seed=7)
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20, policy=policy)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(blocks + policy)
    for e in range(4):
        mine = np.where(r.random(w.N) < 0.1, r.integers(0, 1 << r.integers(1, 20), w.N), 0).astype(np.uint32)
        mine[-1] = e                                          # the pool's ragged end
        g.pool.touch[:w.N] = g.torch.from_numpy(mine.view(np.int32)).cuda()
        o.touch[:] = mine
        ev = r.integers(0, w.N, 0 if call == "no trace" else 2501).astype(np.uint32)
        if call == "overflow":
            ev = r.permutation(np.concatenate([ev, np.full(700, r.integers(0, w.N), np.uint32)]))
        hit = r.integers(0, 2, ev.size).astype(np.uint8)
        g.torch.cuda.synchronize()
        d_e, d_h, n = g.stage_events(ev, hit) if ev.size else (None, None, 0)
        if call == "score":
            g.check(g.pool.kv_epoch_score(e, d_e, d_h, n), "kv_epoch_score")
        else:
            g.check(g.pool.kv_epoch_score_select(e, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
        assert o.epoch_score(e, ev, hit) == O.OK
        ls.compare_state((call, blocks, e))
        if call != "score":
            rc, v = o.select_victims(w.k)
            assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v)
    ls.close()
