"""Host memory of a handle that uses no sweep tables (no GPU)."""
import subprocess
import sys

CODE = """
import ctypes, resource
from paper_2208_09132_gb300 import cdugks, workloads as wl
lib = cdugks.load()
cfg, _ = wl.random_smooth(dim=3, n=(4, 4, 4), nv=(101, 101, 101), seed=1)
g, v, p = cdugks.describe(cfg, cdugks.FP64)
h = ctypes.c_void_p()
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
assert lib.cdugks_create(ctypes.byref(g), ctypes.byref(v), ctypes.byref(p), ctypes.byref(h)) == 0
grown = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before
lib.cdugks_destroy(h)
print(grown * 1024 / 101 ** 3)
"""


def test_creation_keeps_the_velocity_and_reflection_tables_only():
    """Per velocity 64 bytes of the table in FP64, 32 in FP32 and 32 of the mirror
    images, 128 in all, and a quarter of that for the allocator; the records of
    sweep A and B (some 200 more) are formed when a workspace is bound."""
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert float(r.stdout) <= 160
