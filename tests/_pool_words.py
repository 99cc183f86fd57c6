"""A pool's device words that no call hands out -- the control words and the per-session
counts -- as CUDA tensors, for tests that make them disagree with the tables.  Their places
come from the library's own header, compiled here with the host compiler."""
import ctypes
import os
import subprocess

import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
#include <cstddef>
#include <cstdio>
#include "lv_internal.cuh"
int main() {
  printf("%zu %zu %d %d\\n", offsetof(lv::DevPool, ctl), offsetof(lv::DevPool, cnt), (int)lv::C_HBM_ALLOC,
         (int)lv::C_HOST_ALLOC);
}
"""


def pool_words(pool, tmp_path):
    """(HBM allocation count [1], host allocation count [1], per-session counts [S, 2])."""
    src, exe = tmp_path / "offsets.cpp", tmp_path / "offsets"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2606_22983_gb300", "csrc"), "-I", "/usr/local/cuda/include", str(src), "-o",
                    str(exe)], check=True)
    ctl, cnt, hbm, host = map(int, subprocess.run([str(exe)], check=True, capture_output=True).stdout.split())
    from paper_2606_22983_gb300.pool import _CudaArray
    handle = pool.handle if isinstance(pool.handle, int) else pool.handle.value

    def view(offset, nbytes):           # DevPool is the pool's first member
        p = ctypes.c_void_p.from_address(handle + offset).value
        return torch.as_tensor(_CudaArray(p, nbytes), device=pool.device)

    words = view(ctl, 256).view(torch.int64)
    return words[hbm:hbm + 1], words[host:host + 1], view(cnt, 8 * pool.S).view(torch.int32).view(pool.S, 2)
