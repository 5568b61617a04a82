"""The allocation-free selection starts clean whatever the calls before it have left in the library's
scratch (one that gave up on a wait, two that ran at the same time): scratch full of noise, where only
the words that number the calls are what calls can have left, against a sort on the host (exact)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2604_26968_b200 import binding as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    torch.cuda.init()
    B.load()
    C.CDLL(os.path.join(ROOT, "paper_2604_26968_b200", "libkvtier.so"), mode=C.RTLD_GLOBAL)
    so = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a",
                    "-diag-suppress", "186", "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2604_26968_b200", "csrc"), os.path.join(ROOT, "tests", "static_scratch.cu"),
                    "-o", so], check=True)
    lib = C.CDLL(so)
    for name in ("scratch_bytes", "scratch_words_at", "scratch_words"):
        getattr(lib, name).restype = C.c_uint64
    lib.select_on.argtypes = [C.c_void_p, C.c_void_p, C.c_uint64, C.c_uint64, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]
    return lib


@pytest.mark.parametrize("variant", [1, 0])
@pytest.mark.parametrize("n", [8192, 8193, 40_001, 1_000_003, 4_194_304])
def test_scratch_in_any_state(probe, n, variant):
    import torch
    r = np.random.default_rng(n)
    score = r.random(n, dtype=np.float32).round(4)   # (ties)
    state = (r.random(n) < 0.9).astype(np.uint8)
    k = n // 10
    resident = np.flatnonzero(state)
    want = np.sort(resident[np.argsort(score[resident], kind="stable")[:k]])
    d_score, d_state = torch.from_numpy(score).cuda(), torch.from_numpy(state).cuda()
    victims = torch.zeros(k + 4, dtype=torch.int32, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    at, words = probe.scratch_words_at(), probe.scratch_words()
    scratch = torch.empty(probe.scratch_bytes(), dtype=torch.uint8, device="cuda")
    for fill in range(3):
        noise = r.integers(0, 256, scratch.numel(), dtype=np.uint8) if fill else np.full(scratch.numel(), 255, np.uint8)
        last = int(r.integers(1, 1 << 40))
        numbers = r.integers(0, last + 1, words)
        numbers[0] = last
        noise[at:at + 8 * words] = numbers.astype(np.uint64).view(np.uint8)
        scratch.copy_(torch.from_numpy(noise))
        for again in range(2):   # (and once more on what that call left)
            victims.zero_()
            torch.cuda.synchronize()
            assert probe.select_on(d_score.data_ptr(), d_state.data_ptr(), n, k, victims.data_ptr(), scratch.data_ptr(),
                                   status.data_ptr(), torch.cuda.current_stream().cuda_stream, variant) == 0
            torch.cuda.synchronize()
            assert int(status[0]) == 0
            assert np.array_equal(victims[:k].cpu().numpy(), want), (fill, again)
