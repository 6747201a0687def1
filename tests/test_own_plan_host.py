"""Shares and shared-memory plans of the one-column CG launches (host functions, no GPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1804_03415_gb300")


def test_own_plans(tmp_path):
    from paper_1804_03415_gb300 import build as B

    B.build()
    exe = str(tmp_path / "plans")
    subprocess.run([B.NVCC, "-std=c++17", B.ARCH, "-x", "cu", "-I", os.path.join(PKG, "csrc"),
                    os.path.join(ROOT, "tests", "own_plan_harness.cpp"), "-Xlinker", f"-rpath={PKG}", "-Xlinker", B.OUT,
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and "plans hold" in r.stdout, r.stdout
