"""The order of what demotions and promotions enqueue, without a GPU: kvtier_host.cu is built against
stand-ins for the CUDA runtime and the kernels (enqueued_order.cu), which check that every access to a
ring slot, staging buffer, slab entry, ring record or list word is ordered behind the last write of it,
whatever the streams do in between.  Demotions below and above the size that is stored straight into
the ring follow one another on rings that wrap."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("order") / "enqueued_order")
    csrc = os.path.join(ROOT, "paper_2604_26968_b200", "csrc")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-O1", "-gencode",
                    "arch=compute_100a,code=sm_100a", "-diag-suppress", "186", "--cudart", "none",
                    "-I", os.path.join(ROOT, "include"), "-I", csrc, os.path.join(csrc, "kvtier_host.cu"),
                    os.path.join(ROOT, "tests", "enqueued_order.cu"), "-o", exe], check=True)
    return exe


def play(program, *args):
    r = subprocess.run([program, *map(str, args)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (args, r.stdout)


@pytest.mark.parametrize("gather", [0, 1 << 20])
@pytest.mark.parametrize("deferred", [0, 1])
@pytest.mark.parametrize("scenario", ["both", "behind", "wrap"])
def test_small_demotions_after_a_large_one(program, scenario, deferred, gather):
    play(program, 1, deferred, 400, gather, scenario)


@pytest.mark.parametrize("ring", [100, 250, 400])
@pytest.mark.parametrize("gather", [0, 1 << 20])
@pytest.mark.parametrize("deferred", [0, 1])
def test_random_sequences(program, deferred, gather, ring):
    for seed in range(25):
        play(program, seed, deferred, ring, gather)
