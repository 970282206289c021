"""The fixed-point reciprocal behind the panel's pivots, on the CPU.

r = R 2^(1 - 32 (L + 1)) lies below 1 / f with 0 < 1 - f r < 2^-(32 L + 28): what is
left out of its last step is under eight units of the word below the result, so that
rounding it to L words is right unless 1 / f lies as close to a boundary.  (The
last Newton step is of third order at L = 7: of second order it leaves 2^-234,
ten bits below the result only.)
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "mpf_host", "recip_host.cpp")
INC = os.path.join(ROOT, "paper_2609_29554_gb300", "csrc")


def test_recip_words_error(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "recip_host")
    subprocess.run([cxx, "-O1", "-w", "-std=c++17", "-I", INC, "-o", exe, SRC], check=True, capture_output=True)
    out = subprocess.run([exe, "4000"], check=True, capture_output=True, text=True).stdout
    worst = {4: 0, 6: 0, 7: 0}
    for line in out.splitlines():
        L, F, R = line.split()
        L, F, R = int(L), int(F, 16), int(R, 16)
        # 1 - f r = (2^(64 L + 31) - F R) / 2^(64 L + 31)
        d = (1 << (64 * L + 31)) - F * R
        assert d > 0
        worst[L] = max(worst[L], d)
    for L, d in worst.items():
        assert d < 1 << (64 * L + 31 - (32 * L + 28)), (L, d.bit_length() - (64 * L + 31))
