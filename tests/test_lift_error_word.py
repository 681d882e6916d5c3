"""The lifted call's error word: every bounded wait has a bit of its own, and the message names the pass that
stalled (a host program compiled from the header that both sides share)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1711_05075_gb300", "csrc")


def test_every_wait_has_its_own_bit_and_message(tmp_path):
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "word.cpp"
    src.write_text('#include <cstdio>\n#include "bc_lift4.h"\n'
                   "int main() { using namespace bc;\n"
                   "for (int b : {(int)LIFT_ERR_COPY, (int)LIFT_ERR_ACCUMULATOR, (int)LIFT_ERR_STAGE, (int)LIFT_ERR_DRAIN, (int)LIFT_ERR_LINE})\n"
                   '  std::printf("%d %s\\n", b, lift_stall_message(b).c_str()); }\n')
    exe = tmp_path / "word"
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    rows = [l.split(" ", 1) for l in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    bits = [int(b) for b, _ in rows]
    assert len(set(bits)) == 5 and all(b & (b - 1) == 0 for b in bits)
    assert all("contraction" in m and "NUFFT" not in m for _, m in rows[:4])
    assert "NUFFT" in rows[4][1] and "contraction" not in rows[4][1]
