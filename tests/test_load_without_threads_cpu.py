"""Loading a mechanism where the system gives no further thread (a stack limit that no thread can
have): kernel units are then compiled, or fetched from the cache, by the calling thread."""
import os
import resource
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import sys
sys.path.insert(0, %r)
import threading
try:
    threading.Thread(target=int).start()
    print("threads")
except RuntimeError:
    pass
from paper_2503_24286_gb300 import binding as B
m = B.Mechanism(sys.argv[1], "device=0")
m.prepare("jvp,vjp")
print("loaded", int(m.stat("tile")))
"""


def test_load_and_prepare(mech_files, tmp_path):
    env = dict(os.environ, PYRO_CACHE_DIR=str(tmp_path), OPENBLAS_NUM_THREADS="1", OMP_NUM_THREADS="1")
    run = lambda limit: subprocess.run(  # noqa: E731
        [sys.executable, "-c", PROGRAM % ROOT, mech_files[0][0]], env=env, capture_output=True, text=True, timeout=300,
        preexec_fn=(lambda: resource.setrlimit(resource.RLIMIT_STACK, (1 << 46, resource.RLIM_INFINITY))) if limit else None)
    if resource.getrlimit(resource.RLIMIT_STACK)[1] != resource.RLIM_INFINITY:
        pytest.skip("a hard stack limit")
    first = run(False)                           # fills the cache (the compiler may use threads itself)
    assert first.returncode == 0, first.stderr[-2000:]
    r = run(True)
    if "threads" in r.stdout:
        pytest.skip("the limit did not keep threads from starting")
    assert r.returncode == 0 and r.stdout.split()[-2:] == ["loaded", "1"], r.stderr[-2000:]
