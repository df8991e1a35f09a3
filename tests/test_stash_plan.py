"""The work list of the one-launch two-pass step (plan_stash, planner.cpp),
built with sanitizers and driven by tests/stash_plan.cpp over random layouts,
grids and ring sizes: the list follows its rule, and a model of the kernel's
CTAs working through it in random turns always comes to an end."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1904_00962_gb300", "csrc")


def test_work_list_under_sanitizers(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "stash_plan"
    cmd = [gxx, "-std=c++17", "-O1", "-g", "-fno-omit-frame-pointer",
           "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
           "-Wall", "-Wextra", "-Werror",
           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
           "-I", CSRC, os.path.join(CSRC, "planner.cpp"),
           os.path.join(ROOT, "tests", "stash_plan.cpp"), "-o", str(exe)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode and "sanitize" in res.stderr and "cannot find" in \
            res.stderr:
        pytest.skip("sanitizer runtime not available")
    assert res.returncode == 0, res.stderr
    run = subprocess.run([str(exe), "1500"], capture_output=True, text=True,
                         timeout=600,
                         env=dict(os.environ, ASAN_OPTIONS="detect_leaks=1"))
    assert run.returncode == 0, run.stderr[-4000:]
    assert run.stdout.strip() == "1500 layouts"
