"""Traces of several rounds of the grid whose vectors are runs, broken runs, single entries and entries out of
range, with flags of any value, mixed in one trace, around a round of the whole grid, against the oracle,
bit for bit, with the status bits."""
import numpy as np
import pytest

from oracle import kv_oracle as O
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

ROUND = 512 * 296 * 8          # events of one round of the grid


@pytest.mark.parametrize("n_events", [ROUND - 5, ROUND + 4, ROUND + 128 * 7 + 3, 2 * ROUND + 131])
def test_mixed_trace(n_events):
    from lockstep import Lockstep
    w = W.Workload("deal", [W.gqa(3, 6, 3, 16, 8, 7001, 9000, "entry")], 0.05, 0.0, seed=7)      # 63,009 entries
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(n_events)
    starts = r.integers(0, w.N // 4 - 9, -(-n_events // 32)) * 4
    ev = (starts[:, None] + np.arange(32)[None, :]).reshape(-1)[:n_events]                       # aligned runs ...
    half = n_events // 2
    ev[half:] = np.sort(r.integers(0, w.N, n_events - half))                                     # ... and freed slots in order
    some = r.integers(0, n_events, 3000)
    ev[some] = r.integers(0, w.N, 3000)
    hit = r.integers(0, 3, n_events).astype(np.uint8) * 85                                       # any non-zero flag is a hit
    ev = ev.astype(np.uint32)
    d_e, d_h, n = g.stage_events(ev, hit)
    g.check(g.pool.kv_epoch_score_select(0, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
    assert o.epoch_score(0, ev, hit) == O.OK
    ls.compare_state(n_events)
    rc, v = o.select_victims(w.k)
    assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v)
    ev[:: n_events // 50] = w.N + 3                                                              # refused, and flagged
    d_e, d_h, n = g.stage_events(ev, hit)
    g.check(g.pool.kv_epoch_score_select(1, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
    assert o.epoch_score(1, ev[ev < w.N], hit[ev < w.N]) == O.OK
    assert g.pool.kv_device_status() == 1          # KV_DEV_EVENT_BAD_ID
    ls.compare_state((n_events, "refused"))
    ls.close()


@pytest.mark.parametrize("blocks", [7001, 7002, 7003])                     # pools of every remainder modulo 4
@pytest.mark.parametrize("n_events", [128, 4096 + 37, ROUND + 128 * 7 + 3])
def test_ids_that_wrap(n_events, blocks):
    """"No entry" (2^32 - 1) and the ids before it, ahead of the pool's first entries: they are refused and
    flagged, and the events beside them count, in warps of runs and in broken ones."""
    from lockstep import Lockstep
    w = W.Workload("wrap", [W.gqa(3, 6, 3, 16, 8, blocks, 9000, "entry")], 0.05, 0.0, seed=7)
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(n_events + blocks)
    starts = r.integers(0, w.N // 4 - 1, -(-n_events // 4)) * 4 + r.integers(0, 4)
    ev = starts[:, None] + np.arange(4)[None, :]
    ev[0] = np.arange(-1, 3)                                               # the first warp: one wrapped run among runs
    some = r.random(len(ev)) < 0.01
    ev[some] = np.arange(4)[None, :] - r.integers(1, 4, int(some.sum()))[:, None]
    ev = ev.reshape(-1)[:n_events].astype(np.int64).astype(np.uint32)      # (-1 is 2^32 - 1)
    hit = r.integers(0, 2, n_events).astype(np.uint8)
    for e, call in enumerate(["fused", "score", "fused"]):
        d_e, d_h, n = g.stage_events(ev, hit)
        if call == "fused":
            g.check(g.pool.kv_epoch_score_select(e, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
        else:
            g.check(g.pool.kv_epoch_score(e, d_e, d_h, n), "kv_epoch_score")
        assert o.epoch_score(e, ev[ev < w.N], hit[ev < w.N]) == O.OK
        assert g.pool.kv_device_status() == 1          # KV_DEV_EVENT_BAD_ID
        ls.compare_state((n_events, blocks, e))
        if call == "fused":
            rc, v = o.select_victims(w.k)
            assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v)
    ls.close()
