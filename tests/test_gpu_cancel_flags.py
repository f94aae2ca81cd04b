"""The handles' cancel flags, which come from a pool.

More handles alive than the pool has flags, each with a flag of its own; a flag
that a destroyed handle left set does not stop the next one; and a device reset,
which takes the pool's memory away and lets its address go to someone else, does
not leave a handle writing there.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _small():
    return mp.Simulation([mp.System(2, 1.5, n_paths=2)], 1, 2, graph=False)


def test_more_handles_than_flags():
    sims = [_small() for _ in range(300)]
    sims[0].run()
    want = sims[0].estimates()["e"]
    long = [mp.Simulation([mp.System(16, 1.0, n_paths=4096)], 5000, 5000, graph=False) for _ in range(2)]
    long[0].run()
    for s in sims:  # everyone else's flag
        s.cancel()
    long[0].cancel()
    with pytest.raises(mp.MPError) as ei:
        long[0].estimates()
    assert ei.value.status == mp.MP_ECANCELED
    for s in sims:
        s.run()  # clears its own
    for k in range(0, 300, 7):
        sims[k].cancel()
        sims[k].close()
    for s in sims:
        if s.handle.value:
            assert s.estimates()["e"] == want
    again = [_small() for _ in range(60)]  # flags left set by the closed ones
    for s in again:
        s.run()
        assert s.estimates()["e"] == want
    for s in sims + again + long:
        s.close()


SCRIPT = """
import ctypes, sys
sys.path.insert(0, {root!r})
import paper_1305_6758_gb300 as mp
lib = mp.load_library()
rt = None
for name in ("libcudart.so", "libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
    try:
        rt = ctypes.CDLL(name)
        break
    except OSError:
        pass
if rt is None:
    print("SKIP")
    sys.exit(0)

def once():
    h = ctypes.c_void_p()
    st = lib.mp_create(4, 1.5, 1.0, 0.0, 64, 5, 5, 1, ctypes.byref(h))
    if st != 0:
        return ("create", st)
    out = mp.MPEstimates()
    st = lib.mp_run(h) or lib.mp_estimates(h, 0, ctypes.byref(out))
    lib.mp_destroy(h)
    return ("e", out.e) if st == 0 else ("run", st)

first = once()
assert first == once() and first[0] == "e", first
assert rt.cudaDeviceReset() == 0
held = []
for _ in range(8):  # pinned memory of the caller's, perhaps where the pool was
    p = ctypes.c_void_p()
    assert rt.cudaHostAlloc(ctypes.byref(p), ctypes.c_size_t(16384), ctypes.c_uint(2)) == 0
    ctypes.memset(p, 0x5A, 16384)
    held.append(p)
got = once()
print("after", got)
for p in held:
    assert ctypes.string_at(p, 16384) == b"Z" * 16384
print("OK")
"""


def test_a_device_reset_takes_the_pool_along():
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], capture_output=True, text=True, timeout=120)
    if "SKIP" in r.stdout:
        pytest.skip("no libcudart to reset the device with")
    print(r.stdout, r.stderr)
    assert r.returncode == 0 and "OK" in r.stdout, r.stderr
