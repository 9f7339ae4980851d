"""What the host code asks of the device, checked without one: api.cpp, plan.cpp and
tune.cpp linked against a stand-in CUDA runtime (tests/host_calls_check.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_17530_gb300", "csrc")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = tmp_path_factory.mktemp("host_calls") / "host_calls_check"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                           "/usr/local/cuda/include", os.path.join(ROOT, "tests", "host_calls_check.cpp")] +
                          [os.path.join(CSRC, f) for f in ("api.cpp", "plan.cpp", "tune.cpp")] + ["-o", str(exe), "-lpthread"])

    def run(mode):
        out = subprocess.run([str(exe), mode], capture_output=True, text=True, timeout=120)
        assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
    return run


def test_pruned_fill_takes_the_flags_of_its_own_grid(check):
    check("pruned")


def test_device_work_is_ordered_after_the_copies_it_reads(check):
    check("ordering")


def test_tuning_decides_for_the_shapes_it_could_time(check):
    check("tuning")


def test_pruned_call_takes_the_faster_fill(check):
    check("choice")
