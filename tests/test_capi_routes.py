"""What a step launches, for any layout and option: the C entry points' host
code, built by tests/capi_routes.cpp on a stand-in for the CUDA runtime, with
launchers that write down their calls."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1904_00962_gb300", "csrc")
AUTO, TWO_PASS, ON_CHIP = 0, 1, 3
GRAD_NORM, SKIP = 0x8, 0x10
TOO_LARGE = 720          # cudaErrorCooperativeLaunchTooLarge
LAUNCH_FAILURE = 719     # cudaErrorLaunchFailure


@pytest.fixture(scope="module")
def routes(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path_factory.mktemp("capi_routes") / "capi_routes"
    cmd = [gxx, "-std=c++17", "-O1", "-w",
           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
           "-I", CSRC, "-x", "c++", os.path.join(CSRC, "lamb_capi.cu"),
           os.path.join(CSRC, "planner.cpp"),
           os.path.join(ROOT, "tests", "capi_routes.cpp"), "-o", str(exe)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]

    def run(sizes, algorithm=AUTO, opt="lamb", flags=0, **options):
        res = subprocess.run(
            [str(exe), str(algorithm), opt, str(flags), sizes] +
            [f"{k}={v}" for k, v in options.items()],
            capture_output=True, text=True, timeout=60)
        assert res.returncode == 0, res.stderr
        return res.stdout.strip()
    return run


BIG = "1000000x200"      # AUTO: a two-pass plan that steps in one launch


@pytest.mark.parametrize("opt", ["lamb", "nlamb", "nnlamb", "lars"])
def test_a_refused_cooperative_launch_takes_the_two_kernels(routes, opt):
    """Fewer SMs free to this process than the device has: the two launches need
    no residency, the step succeeds and no error is left behind."""
    line = routes(BIG, opt=opt, refuse=TOO_LARGE)
    assert line == (f"algo 1 status 0: refused_{opt} {opt}1 {opt}2 timed 2 "
                    "left 0")
    line = routes(BIG, opt=opt)
    assert line == f"algo 1 status 0: stash_{opt} timed 1 left 0"


@pytest.mark.parametrize("flag", [GRAD_NORM, SKIP])
def test_a_refused_launch_behind_the_gradient_check(routes, flag):
    """The check has been launched by then; the two kernels form it again."""
    line = routes(BIG, flags=flag, refuse=TOO_LARGE)
    assert line == ("algo 1 status 0: check refused_lamb lamb1+gn lamb2+gn "
                    "timed 2 left 0")
    assert routes(BIG, flags=flag) == (
        "algo 1 status 0: check stash_lamb timed 2 left 0")


def test_another_launch_error_is_reported(routes):
    line = routes(BIG, refuse=LAUNCH_FAILURE)
    assert line.startswith("algo 1 status 3: refused_lamb timed 0")


@pytest.mark.parametrize("option", [
    {"chunk_elems": 4096}, {"blocks_per_sm": 1}, {"tail_elems": 65536}],
    ids=lambda o: next(iter(o)))
@pytest.mark.parametrize("opt", ["lamb", "lars", "nnlamb"])
def test_options_of_the_two_kernels_keep_them(routes, opt, option):
    """A caller who shapes the two-pass kernels gets them from AUTO, with the
    chunks, the grid or the tail asked for."""
    assert routes(BIG, opt=opt, **option) == (
        f"algo 1 status 0: {opt}1 {opt}2 timed 2 left 0")


def test_options_of_the_on_chip_kernel_keep_it(routes):
    several = "100000x150"       # an on-chip plan of several rounds
    assert routes(several) == "algo 3 status 0: stash_lamb timed 1 left 0"
    for option in ({"onchip_rows": 200}, {"chunk_elems": 4096}):
        assert routes(several, **option) == (
            "algo 3 status 0: onchip_lamb timed 1 left 0")
    # a limit on the CTAs is one of the one launch too
    assert routes(several, onchip_max_ctas=100) == (
        "algo 3 status 0: stash_lamb timed 1 left 0")


# What a step launches where one launch was measured to pay and where not (a
# GB300, us; see one_launch_pays).
@pytest.mark.parametrize("opt,sizes,one", [
    ("lars", "1000000x200", True),                  # 827 / 694
    ("lars", "1000000x300,30000000", True),         # 1287 / 1192
    ("lars", "1000000x50,9400000", True),           # 244 / 228
    ("lars", "4000x20000,6000000", True),           # 447 / 413
    ("lars", "6500000x10", False),                  # 267 / 355
    ("lars", "8000000", False),                     # 49 / 54
    ("lars", "1000000x100,30000000", False),        # 517 / 537
    ("lars", "5600000x10", False),                  # 230 / 244
    ("lars", "500x100000", False),                  # 1229 / 1338
    ("lars", "2000x2000,6000000", False),           # 63 / 66
    ("lamb", "500x100000", True),                   # 1768 / 1370
    ("lamb", "8000000", True),                      # 77 / 61
    ("lamb", "1000000x100,30000000", True),         # 753 / 626
    ("lamb", "10000000x10", False),                 # 587 / 635
    ("lamb", "6500000x10", False),                  # 387 / 402
    ("lamb", "14000000", False),                    # 97 / 105
    ("nlamb", "9000000x10", True),                  # 575 / 548
    ("nlamb", "30000000", False),                   # 212 / 229
])
def test_one_launch_where_it_pays(routes, opt, sizes, one):
    want = f"stash_{opt} timed 1" if one else f"{opt}1 {opt}2 timed 2"
    assert routes(sizes, opt=opt) == f"algo 1 status 0: {want} left 0"


@pytest.mark.parametrize("flag,sizes,one", [
    (GRAD_NORM, "1000000x20,10000000,1000000x20", True),
    (GRAD_NORM, "500x20000,10000000", True),        # 801 / 477
    (GRAD_NORM, "6000000", False),                  # 61 / 73
    (GRAD_NORM, "10000000", False),                 # 86 / 109
    (SKIP, "6000000", False),                       # 65 / 73
    (SKIP, "1000000x20,10000000", True),            # 225 / 192
])
def test_one_launch_behind_the_check_where_it_pays(routes, flag, sizes, one):
    want = "check stash_lamb" if one else "lamb1+gn lamb2+gn"
    assert routes(sizes, flags=flag) == (
        f"algo 1 status 0: {want} timed 2 left 0")
