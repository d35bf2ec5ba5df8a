"""Who moves a caller's array (csrc/kf_route.h): the rule's host code compiled
by itself, for arrays on another GPU, which no test machine here has, and on
odd bytes (which tests/test_gpu_array_layouts.py runs)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_11744_gb300", "csrc")


def test_arrays_a_kernel_takes(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    prog = tmp_path / "route.cpp"
    prog.write_text('#include <cstdio>\n#include "kf_route.h"\nint main() {\n'
                    "  for (int on = kfg::NO_DEVICE; on < 3; ++on)\n"
                    "    for (int dev = 0; dev < 3; ++dev)\n"
                    "      for (int at = 0; at < 5; ++at)\n"
                    '        std::printf("%d %d %d %d %d\\n", on, dev, at, kfg::kernel_reads((char*)0x1000 + at, on, dev),\n'
                    "                    kfg::kernel_writes(on, dev));\n"
                    "}\n")
    exe = tmp_path / "route"
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(prog), "-o", str(exe)], check=True)
    rows = [tuple(map(int, r.split())) for r in
            subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 4 * 3 * 5
    for on, dev, at, reads, writes in rows:
        here = on in (-1, dev)  # host and managed memory, or the kernel's own GPU
        assert writes == here
        assert reads == (here and at % 4 == 0)
