"""The LU's panel kernel on the CPU, its warps held back in many orders.

`tests/panel_host/panel_host.cpp` runs the kernel of csrc/panel.cuh with every CUDA
thread as a coroutine and the order of the warps chosen by a seed: a warp goes on
only when the order says so or when nothing else can.  Whatever the kernel's own
barriers and exchanged words leave open is thereby taken to its extremes; the
interchanges and every word of the factored panel must not depend on it, nor on how
the rows are spread over blocks.
"""
import hashlib
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "panel_host", "panel_host.cpp")
INC = os.path.join(ROOT, "paper_2609_29554_gb300", "csrc")


@pytest.fixture(scope="module")
def panel(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("panel") / "panel_host")
    subprocess.run([cxx, "-O2", "-w", "-std=c++17", "-pthread", "-fno-extern-tls-init", "-I", INC, "-o", exe, SRC],
                   check=True, capture_output=True, text=True)

    def run(nc, n, b, rows, order, seed):
        r = subprocess.run([exe, str(nc), str(n), str(b), str(rows), order, str(seed)], check=True,
                           capture_output=True, text=True, timeout=120)
        head, pivots, words = r.stdout.splitlines()
        return head, pivots, hashlib.sha256(words.encode()).hexdigest()
    return run


@pytest.mark.parametrize("nc,n,b,rows", [
    (2, 128, 128, 128),  # one block that owns both rows of every interchange, more than two rows a lane
    (2, 128, 128, 64),   # two blocks, two rows a lane
    (4, 128, 128, 16),   # eight blocks
    (3, 70, 69, 70),     # odd width
])
def test_result_does_not_depend_on_the_order_of_the_warps(panel, nc, n, b, rows):
    want = panel(nc, n, b, rows, "even", 0)
    assert want[0] == "error 0 info 0"
    for seed in range(1, 9):
        for order in ("late", "mixed"):
            assert panel(nc, n, b, rows, order, seed) == want, (order, seed)


def test_result_does_not_depend_on_the_rows_a_block(panel):
    want = panel(2, 128, 128, 128, "even", 0)
    for rows in (8, 24, 64):
        assert panel(2, 128, 128, rows, "late", rows) == want, rows


@pytest.mark.parametrize("nc,n,b,rows", [(2, 100, 100, 50), (3, 65, 65, 33), (4, 90, 77, 30), (4, 64, 64, 64)])
def test_the_panel_is_the_plain_factorisation(panel, nc, n, b, rows):
    # every element one rounding of y - l u with the multiplier that is stored
    assert panel(nc, n, b, rows, "mixed", 3) == panel(nc, n, b, rows, "plain", 0)
