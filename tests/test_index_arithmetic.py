"""The kernels' index arithmetic, evaluated on the host by a small program that
includes the kernel sources (tests/index_arithmetic.cu)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_index_arithmetic(tmp_path):
    from paper_1202_6081_gb300.build import ARCH, CSRC, INCLUDE, nvcc
    exe = str(tmp_path / "index_arithmetic")
    subprocess.run([nvcc(), "-std=c++17", "-I", INCLUDE, "-I", CSRC, *ARCH,
                    os.path.join(ROOT, "tests", "index_arithmetic.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
