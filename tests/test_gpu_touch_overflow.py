"""Epochs in which an entry has more touches than the fused pass's packed counts hold: the pass that finds it
out (without a hint and with one), the epochs behind it, which count in 32 bits, and packed counts again when
those have gone by; pools of one CTA, of one row and of several, of every policy, with and without head
weights, FREE entries among the hot ones' neighbours; and the same in a captured call that is replayed.
Against the oracle, bit for bit."""
import numpy as np
import pytest

from oracle import kv_oracle as O
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

COOL_DOWN = 64       # epochs in 32 bits


def trace(n, hot, r, length=3001):
    ev = r.integers(0, n, length)
    if hot:          # counts around 512 on neighbours, and on the pool's last entries
        at = r.integers(0, n - 8)
        ids = np.concatenate([np.repeat(at + np.arange(8), r.integers(505, 520, 8)), np.repeat([n - 2, n - 1], [512, 700])])
        ev = r.permutation(np.concatenate([ev, ids]))
    return ev.astype(np.uint32), r.integers(0, 2, ev.size).astype(np.uint8)


def score_select(ls, e, ev, hit, check):
    g, o, w = ls.gpu, ls.ora, ls.w
    d_e, d_h, n = g.stage_events(ev, hit)
    g.check(g.pool.kv_epoch_score_select(e, d_e, d_h, n, w.k, g.victims), "kv_epoch_score_select")
    resident = o.state[ev] == O.RESIDENT
    assert o.epoch_score(e, ev[resident], hit[resident]) == O.OK
    if check:
        status = g.pool.kv_device_status()
        assert (status == 0) == bool(resident.all())
        ls.compare_state(e)
        rc, v = o.select_victims(w.k)
        assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v), e


@pytest.mark.parametrize("heads", [None, (0.8, 4)])
@pytest.mark.parametrize("policy", [0, 1, 2])
@pytest.mark.parametrize("blocks", [455, 1237, 110_003])        # 4,095 entries, 11,133, 990,027
def test_hot_now_and_then(blocks, policy, heads):
    from lockstep import Lockstep
    w = W.Workload("hot", [W.gqa(3, 6, 3, 16, 8, blocks, 9 * blocks, "entry")], 0.05, 0.0, seed=7)
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20, policy=policy, heads=heads)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(blocks + policy)
    hot = {0, 4, 5, 5 + COOL_DOWN + 3}                          # the first pass has no hint
    for e in range(max(hot) + 3):
        if heads is not None:
            ls.head_step(e)
        ev, hit = trace(w.N, e in hot, r)
        score_select(ls, e, ev, hit, e < 8 or e > COOL_DOWN)
        if e == 1:                                              # from here on some slots are FREE
            rc, v = o.select_victims(w.k)
            assert rc == O.OK and o.demote(v) == O.OK
            g.check(g.pool.kv_demote(g.victims, w.k, g.batch_bytes), "kv_demote")
            ls.compare_state("demoted", scores=False)
    ls.close()


def test_captured_call_meets_hot_traces():
    import torch
    from lockstep import Lockstep
    w = W.Workload("hot", [W.gqa(3, 6, 3, 16, 8, 7001, 9000, "entry")], 0.05, 0.0, seed=7)
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20)
    g, o = ls.gpu, ls.ora
    r = np.random.default_rng(3)
    score_select(ls, 0, *trace(w.N, False, r), True)            # first call outside the capture
    size = 5000
    d_e = torch.zeros(size, dtype=torch.int32, device="cuda")
    d_h = torch.zeros(size, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=g.pool.compute):
        g.check(g.pool.kv_epoch_score_select(1, d_e, d_h, size, w.k, g.victims), "kv_epoch_score_select")
    for i, hot in enumerate([False, True, True, False, True, False]):
        ev, hit = trace(w.N, False, r, size)
        if hot:
            ev[r.permutation(size)[:1200]] = np.repeat(r.integers(0, w.N, 2).astype(np.uint32), 600)
        d_e.copy_(torch.from_numpy(ev.view(np.int32)))
        d_h.copy_(torch.from_numpy(hit))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert o.epoch_score(1, ev, hit) == O.OK
        ls.compare_state((i, hot))
        rc, v = o.select_victims(w.k)
        assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v), i
    del graph
    ls.close()


def test_no_room_for_packed_counts():
    """Under the LRU policy 25.1 M entries (42 rows) leave no room for packed counts in the stages: the call
    counts in 32 bits, whatever the counts, and stays at two launches."""
    from lockstep import Lockstep
    w = W.Workload("wide", [W.gqa(3, 8, 8, 2, 4, 1_045_834, 64, "entry")], 0.02, 0.0, seed=7)
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20, policy=2)
    g = ls.gpu
    r = np.random.default_rng(5)
    for e, hot in enumerate([False, True, False]):
        before = g.pool.kv_get_stats()["kernel_launches"]
        score_select(ls, e, *trace(w.N, hot, r, 400_001), True)
        assert g.pool.kv_get_stats()["kernel_launches"] - before == 2
    ls.close()
