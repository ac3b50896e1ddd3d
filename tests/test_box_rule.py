"""The box and stack rules of the four-wide walk and of the walk of the hit/miss links on the CPU against
every triangle in turn (tests/box_rule_main.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("g++ or the CUDA headers not available")
    path = str(tmp_path_factory.mktemp("box_rule") / "box_rule")
    csrc = os.path.join(ROOT, "paper_1505_06022_gb300", "csrc")
    b = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                        "-I", "/usr/local/cuda/include", os.path.join(ROOT, "tests", "box_rule_main.cpp"),
                        os.path.join(csrc, "bvh_build.cpp"), "-o", path, "-ldl", "-pthread"], capture_output=True, text=True)
    assert b.returncode == 0, b.stderr[-3000:]
    return path


def run(exe, *group):
    r = subprocess.run([exe, *group], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout + r.stderr)[-3000:]


def test_negative_tmin(exe):
    """tmin behind the origin, down to -inf, with unit, long and short directions."""
    run(exe, "tmin")


def test_coincident_surfaces(exe):
    """Ties in t between triangles of different leaves: the smallest index wins in any order of the walk."""
    run(exe, "ties")


@pytest.mark.parametrize("group", ["tmin", "ties"])
def test_links(exe, group):
    """The same of the walk of the hit/miss links: boxes without extent behind the origin among them."""
    run(exe, group, "links")
