"""A fused call whose second launch is refused: it reports the error, its events stay counted (pairs and
touches alike, beside those of kv_epoch_events), and kv_epoch_update scores the epoch as if they had come
through kv_epoch_events; the epochs after it are as always.  Against the oracle, bit for bit."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from oracle import kv_oracle as O
from paper_2604_26968_b200 import binding as B
from paper_2604_26968_b200 import build as kv_build
from paper_2604_26968_b200 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def copy(tmp_path_factory):
    # (-Bsymbolic: other tests load the library itself for everybody, and its functions would be taken)
    so = str(tmp_path_factory.mktemp("refused") / "libkvtier_refused.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *kv_build.NVCC_FLAGS, "--threads", "8",
                    "-Xlinker", "--wrap=cudaLaunchKernelExC", "-Xlinker", "-Bsymbolic", *[os.path.join(kv_build.CSRC, s) for s in kv_build.SOURCES],
                    os.path.join(ROOT, "tests", "refused_launch.cu"), "-o", so], check=True)
    return so


@pytest.mark.parametrize("hot", [False, True])      # the touches are in 32 bits already, a while after a hot trace
@pytest.mark.parametrize("before", [0, 1500])       # events that kv_epoch_events has counted
def test_events_stay_counted(copy, monkeypatch, before, hot):
    from lockstep import Lockstep
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B._build, "build", lambda *a, **k: copy)
    w = W.Workload("refused", [W.gqa(3, 6, 3, 16, 8, 1237, 9000, "entry")], 0.05, 0.0, seed=7)     # 11,133 entries
    ls = Lockstep(w, payload=False, batch_bytes=1 << 20)
    g, o = ls.gpu, ls.ora
    switch = C.c_int.in_dll(g.pool.lib, "refuse_cooperative")
    r = np.random.default_rng(before)
    for e in range(5):
        ev = r.integers(0, w.N, 3001).astype(np.uint32)
        if (hot and e == 0) or e == 2:                       # the refused one overflows packed counts, too
            ev = np.concatenate([ev, np.repeat(r.integers(0, w.N, 3).astype(np.uint32), [511, 512, 700])])
        hit = r.integers(0, 2, ev.size).astype(np.uint8)
        first = before if e == 2 else 0
        if first:
            d_e, d_h, n = g.stage_events(ev[:first], hit[:first])
            g.check(g.pool.kv_epoch_events(d_e, d_h, n), "kv_epoch_events")
        d_e, d_h, n = g.stage_events(ev[first:], hit[first:])
        switch.value = int(e == 2)
        rc = g.pool.kv_epoch_score_select(e, d_e, d_h, n, w.k, g.victims)
        switch.value = 0
        if e == 2:
            assert rc == -7                                  # KV_ERR_CUDA
            g.pool.sync()
            assert np.array_equal(g.host_array("touch"), np.bincount(ev, minlength=w.N))
            g.check(g.pool.kv_epoch_update(e), "kv_epoch_update")
        else:
            g.check(rc, "kv_epoch_score_select")
        assert o.epoch_score(e, ev, hit) == O.OK
        ls.compare_state(e)
        if e != 2:
            rc, v = o.select_victims(w.k)
            assert rc == O.OK and np.array_equal(g.victims[:w.k].cpu().numpy().view(np.uint32), v)
    ls.close()
