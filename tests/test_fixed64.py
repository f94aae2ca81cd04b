"""The FP64 form's fixed-point trial direction against 40-digit arithmetic (CPU).

A component is an integer in units of 2^-53: half a unit of rounding plus at
most 2^-55.5 from the evaluation (63-bit products, the truncated Taylor terms
and the FP32-seeded Newton steps), so it is within 0.68 units.
"""
import os
import random
import shutil
import subprocess

import pytest

mpmath = pytest.importorskip("mpmath")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EDGES = [0, 1, 0x3FFFFF, 0x400000, 0x3FFFFFFF, 0x40000000, 0x7FFFFFFE, 0x7FFFFFFF, 0x80000000, 0xBFFFFFFF,
         0xC0000000, 0xFFFFFFFE, 0xFFFFFFFF]


@pytest.mark.parametrize("seed", [1, 2])
def test_trial_direction_is_within_its_rounding(tmp_path, seed):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is needed to compile the host form")
    exe = str(tmp_path / "fixed64_dump")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "paper_1305_6758_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "fixed64_dump.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rng = random.Random(seed)
    pairs = [(a, b) for a in EDGES for b in EDGES]
    for k in range(2000):  # the poles (|z| near 1) and small angles too
        r0, r1 = rng.getrandbits(32), rng.getrandbits(32)
        pairs.append((r0 >> (k % 31) if k % 2 else 0xFFFFFFFF - (r0 >> (k % 31)), r1 >> (k % 7)))
    out = subprocess.run([exe], input="\n".join("%d %d" % p for p in pairs), capture_output=True, text=True, check=True)
    got = [tuple(int(v) for v in line.split()) for line in out.stdout.splitlines()]
    assert len(got) == len(pairs)
    mpmath.mp.dps = 40
    for (r0, r1), t in zip(pairs, got):
        z = mpmath.mpf(2 * r0 + 1) / 2**32 - 1
        rad, phi = mpmath.sqrt((1 - z) * (1 + z)), 2 * mpmath.pi * (2 * r1 + 1) / 2**33
        assert t[2] == z * 2**53
        assert abs(t[0] - rad * mpmath.cos(phi) * 2**53) < 0.68, (r0, r1)
        assert abs(t[1] - rad * mpmath.sin(phi) * 2**53) < 0.68, (r0, r1)
