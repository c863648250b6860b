"""CPU test of the march's texture reads (tests/native/texels_test.cpp against
csrc/texels.h), compiled with g++ and run."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reads_stay_inside_the_texture(tmp_path):
    exe = tmp_path / "texels_test"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2603_02048_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "texels_test.cpp"), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "texels ok" in r.stdout
