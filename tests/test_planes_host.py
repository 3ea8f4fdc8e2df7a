"""Which planes of a caller the solver's kernels take directly (the rest go through a copy)."""
import os
import subprocess

from conftest import ROOT


def test_only_aligned_memory_of_the_solvers_device_while_it_is_current(tmp_path):
    src = tmp_path / "p.cpp"
    src.write_text('''
#include <cuda_runtime.h>
#include <stdio.h>
#include "cgks_internal.h"
int main()
{
    char* p = (char*)4096;
    for (int mem = -1; mem < 2; ++mem)
        for (int dev = 0; dev < 2; ++dev)
            for (int cur = 0; cur < 2; ++cur)
                for (int off = 0; off < 9; off += 4) printf("%d %d %d %d %d\\n", mem, dev, cur, off, (int)cgks::planes_direct(mem, dev, cur, p + off));
    return 0;
}
''')
    exe = str(tmp_path / "p")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-w", "-I", cuda, "-I", os.path.join(ROOT, "paper_2001_01570_gb300", "csrc"), "-o", exe,
                    str(src)], check=True)
    for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        mem, dev, cur, off, direct = map(int, ln.split())
        assert direct == (mem == dev == cur and off % 8 == 0), ln
