"""The one-launch step's warps when a launch gives up: the device code of its
workers, drawer and closer, cut from lamb_stash.cu and built for the host by
tests/stash_warps.cpp with a thread for each lane.  Whatever moment a half of a
warp learns of it at, the lanes of the warp leave together, and none leaves a
store to tensor memory in flight."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1904_00962_gb300", "csrc")
UNIFORM = ["drawer_record", "drawer_issued", "drawer_kept_tensor",
           "drawer_kept_record", "closer_record", "closer_done", "worker_wait"]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    tmp = tmp_path_factory.mktemp("stash_warps")
    with open(os.path.join(CSRC, "lamb_stash.cu")) as f:
        text = f.read()
    # the warps' code: up to the kernel itself
    head, marker, _ = text.partition("// The kernel\n")
    assert marker
    lines = [x for x in head.splitlines() if not x.startswith("#include")]
    (tmp / "stash_cut.inc").write_text("\n".join(lines) + "\n}\n}\n")
    exe = tmp / "stash_warps"
    cmd = [gxx, "-std=c++17", "-O1", "-pthread", "-w",
           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
           "-I", CSRC, "-I", str(tmp),
           os.path.join(ROOT, "tests", "stash_warps.cpp"), "-o", str(exe)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    return str(exe)


def _run(harness, scenario):
    res = subprocess.run([harness, scenario], capture_output=True, text=True,
                         timeout=60)
    assert res.returncode == 0, res.stderr


@pytest.mark.parametrize("scenario", UNIFORM)
def test_lanes_of_a_warp_leave_together(harness, scenario):
    _run(harness, scenario)


def test_no_store_to_tensor_memory_outlives_its_worker(harness):
    _run(harness, "worker_stores")
