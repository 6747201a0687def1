"""The order of the rows on the device (host code): no data race between the pieces of one depth, the same order with one
thread and with several, every row once."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1804_03415_gb300", "csrc")


def sanitized(src, exe, *more):
    return subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fopenmp", "-fsanitize=thread", "-I", CSRC, "-c", src, "-o",
                           exe + ".o"], capture_output=True, text=True).returncode or \
        subprocess.run(["g++", "-fsanitize=thread", exe + ".o", *more, "-o", exe, "-pthread"]).returncode


def test_order_has_no_race(tmp_path):
    probe = tmp_path / "probe.cpp"
    probe.write_text("int main() { return 0; }\n")
    exe = str(tmp_path / "probe")
    if sanitized(str(probe), exe) or subprocess.run([exe]).returncode:
        pytest.skip("the thread sanitizer does not run here")
    obj = str(tmp_path / "order")
    assert subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fopenmp", "-fsanitize=thread", "-I", CSRC, "-c",
                           os.path.join(CSRC, "order.cpp"), "-o", obj + ".o"]).returncode == 0
    exe = str(tmp_path / "harness")
    assert sanitized(os.path.join(ROOT, "tests", "order_harness.cpp"), exe, obj + ".o") == 0
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same order" in r.stdout, r.stderr[:4000]
