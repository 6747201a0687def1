"""mmd_build_opts.threads bounds the host threads of the whole build, the upload to the device included.

In a process of its own: OpenMP keeps the threads that a build has started, so a build with four adds three to the
process's after builds with one, none after a build that had taken more."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import os
import workloads as W
import paper_1804_03415_gb300 as G
A = W.torus_knn(6000, seed=1)
def build(threads, **o):
    G.MMD(A.rowptr, A.col, A.val, threads=threads, **o).close()
    return len(os.listdir("/proc/self/task"))
build(1)
one = build(1, k_max=0)
print("added", build(4, k_max=0) - one, build(4) - one)
"""


def test_build_keeps_to_its_threads():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env={**os.environ, "OMP_NUM_THREADS": "8"},
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["added", "3", "3"]
