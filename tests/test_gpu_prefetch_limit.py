"""A prefetch list whose last block's wait for the counts before it runs out: the status says so, and
the count, which the caller's word may hold from an earlier call, says that nothing is listed.  The
kernel is built with a limit of one look; its last block has nothing of its own to do and looks while
the first is still reading its part of the table, tile after tile."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_26968_b200", "csrc")


@pytest.mark.gpu
def test_count_of_a_list_that_gave_up(tmp_path):
    import torch
    torch.cuda.init()
    C.CDLL(os.path.join(ROOT, "paper_2604_26968_b200", "libkvtier.so"), mode=C.RTLD_GLOBAL)
    text = open(os.path.join(CSRC, "kv_prefetch.cu")).read()
    limit = "constexpr uint32_t kPfSpins = 1u << 22;"
    assert text.count(limit) == 1
    (tmp_path / "list.cu").write_text(text.replace(limit, "constexpr uint32_t kPfSpins = 1u;"))
    so = str(tmp_path / "probe.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a",
                    "-diag-suppress", "186", "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    '-DLIST_SOURCE="%s"' % (tmp_path / "list.cu"), os.path.join(ROOT, "tests", "prefetch_probe.cu"), "-o", so], check=True)
    lib = C.CDLL(so)
    u64, u32, ptr = C.c_uint64, C.c_uint32, C.c_void_p
    lib.prefetch_list.argtypes = [ptr, ptr, ptr, ptr, u32, u32, u32, ptr, u64, ptr, u64, ptr, u64, ptr, ptr]
    layers, heads, n_pos = 32, 8, 18_944   # 296 blocks of 16 x 1,024 candidates; the windows hold the first one's

    def ints(n, value, dtype=torch.int32):
        return torch.full((n,), value, dtype=dtype, device="cuda")

    win, words, serial, status = ints(layers, 64), ints(1024, 0, torch.int64), ints(4, 0), ints(4, 0)
    table, n_tags = torch.arange(n_pos * layers * heads, dtype=torch.int32, device="cuda"), n_pos * layers * heads
    loc = (torch.arange(n_tags, device="cuda") + (1 << 31)).to(torch.uint32).view(torch.int32)   # all in the host tier
    out, count = ints(4096, -1, torch.int64), ints(2, 77, torch.int64)
    torch.cuda.synchronize()
    assert lib.prefetch_list(win.data_ptr(), words.data_ptr(), serial.data_ptr(), status.data_ptr(), layers, heads, 65535,
                             table.data_ptr(), n_pos, loc.data_ptr(), n_tags, out.data_ptr(), 4096, count.data_ptr(),
                             torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(status[0]) == 32      # KV_DEV_WAIT_EXPIRED
    assert int(count[0]) == 0 and int(count[1]) == 77
    assert int(serial[0]) == 1       # (the next call has its own number)
