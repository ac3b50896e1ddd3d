"""The four-wide form of the BVH on the CPU: structure and walk against the hit/miss links, under
AddressSanitizer and UndefinedBehaviorSanitizer where they are installed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_wide_walk_equals_the_walk_of_the_links(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("g++ or the CUDA headers not available")
    exe = str(tmp_path / "wide_tree")
    csrc = os.path.join(ROOT, "paper_1505_06022_gb300", "csrc")
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I",
           "/usr/local/cuda/include", os.path.join(ROOT, "tests", "wide_tree_main.cpp"),
           os.path.join(csrc, "bvh_build.cpp"), "-o", exe, "-ldl", "-pthread"]
    b = subprocess.run(cmd + ["-fsanitize=address,undefined", "-fno-sanitize-recover=undefined"], capture_output=True, text=True)
    if b.returncode != 0:
        b = subprocess.run(cmd, capture_output=True, text=True)
    assert b.returncode == 0, b.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout + r.stderr)[-3000:]
