"""The rows a thread of the streamed kernel walks, against the lattice (CPU).

Every row lies in the half-plane and its +-y offsets lead to its periodic
neighbours, also those of a row that stands in for one outside the lattice: its
spins are read, not used.  Each row of the lattice is acted on exactly once.
"""
import os
import shutil
import subprocess
from collections import defaultdict

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rows_stay_in_the_half_plane(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is needed to compile the host form")
    exe = str(tmp_path / "rows_dump")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                        "-I" + os.path.join(ROOT, "paper_1305_6758_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "rows_dump.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    acted = defaultdict(list)
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines():
        L, RS, y0, k, off, yp, ym, act = map(int, line.split())
        HL = L // 2
        y, rest = divmod(y0 * HL + off, HL)
        assert rest == 0 and 0 <= y < L, line
        assert y * HL + yp == (y + 1) % L * HL, line
        assert y * HL + ym == (y - 1) % L * HL, line
        assert y == (y0 + k * RS if act else y0), line
        if act:
            acted[L, RS].append(y)
    assert any(L == 4 * RS for L, RS in acted) and any(3 * RS + 1 == L for L, RS in acted)
    assert (30, 8) in acted and (28, 9) in acted and (60, 16) in acted  # default layouts
    for (L, _), rows in acted.items():
        assert sorted(rows) == list(range(L))
