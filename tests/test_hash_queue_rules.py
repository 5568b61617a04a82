"""The rules by which the hash kernel's warps pass chains of messages on, played through on the CPU:
no place behind the cleared part of the queue's memory is looked at or written, whatever an earlier
call left there, every chain is finished, block after block, and no warp waits for a thread block
that has not started.  Sizes just above a multiple of the
warps are the ones whose warps take the most places that nothing comes to."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2604_26968_b200", "csrc")


@pytest.fixture(scope="module")
def sim(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("sim") / "hash_queue_sim")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "hash_queue_sim.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("seed", [1, 2])
@pytest.mark.parametrize("blocks", [2, 9, 129, 1153])
@pytest.mark.parametrize("resident", [148, 147, 60, 1])
@pytest.mark.parametrize("messages,depth", [(37_889, 2), (60_000, 3), (78_643, 4), (120_000, 5)])
def test_played_through(sim, messages, depth, resident, blocks, seed):
    """depth: groups of four warps per SM; resident: thread blocks of the 148 that run at a time (other
    work may hold SMs)."""
    a = [messages, blocks, 148, 4 * depth, resident, seed]
    r = subprocess.run([sim, *map(str, a)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    most, ring, requeued = map(int, r.stdout.split())
    assert most < ring and requeued <= ring
