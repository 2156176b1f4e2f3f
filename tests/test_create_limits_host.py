"""ba_problem_create where the process can start no thread: the check of the observations runs in the
calling thread, and a failure comes back as a status.  In a child process, whose limits it lowers."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, resource, sys
import numpy as np
from paper_2605_30583_gb300 import binding
binding.lib()
n_cams, n_pts = 50, 150_000
ci = np.random.default_rng(0).integers(0, n_cams, 4 * n_pts).astype(np.uint32)
pi = np.tile(np.arange(n_pts, dtype=np.uint32), 4)
px = np.zeros((len(ci), 2))
if sys.argv[1] == "bad":
    pi[-1] = n_pts
# room for the problem (24 bytes an observation and the bitmaps), none for another thread's stack
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + 24 * len(ci) + int(sys.argv[2]),) * 2)
h = ctypes.c_void_p()
rc = binding.lib().ba_problem_create(n_cams, n_pts, len(ci), ci.ctypes.data, pi.ctypes.data, px.ctypes.data, 0,
                                     ctypes.byref(h))
print("status", rc, bool(h.value))
"""


def _run(kind, room):
    r = subprocess.run([sys.executable, "-c", CHILD, kind, str(room)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    return r.stdout.split()


def test_create_without_threads():
    """4 MiB above the problem's arrays: less than a thread's stack."""
    assert _run("good", 4 << 20) == ["status", "0", "True"]
    out = _run("bad", 4 << 20)
    assert out[0] == "status" and out[1] != "0" and out[2] == "False"
