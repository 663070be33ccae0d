"""Host-side paths of the library that need a failing call (a capture that
breaks off, an allocation that fails): capi.cu compiled for the host with fakes
of the CUDA runtime and of the kernel launchers (host_paths.cpp), no GPU."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2511_13109_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2511_13109_gb300 import build

    exe = str(tmp_path_factory.mktemp("host_paths") / "host_paths")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    # launchers that no scenario reaches have no fake
    cmd = ["g++", "-std=c++17", "-O1", "-w", "-x", "c++", os.path.join(SRC, "capi.cu"),
           os.path.join(HERE, "host_paths.cpp"), "-I", inc, "-o", exe, "-Wl,--unresolved-symbols=ignore-all"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("scenario", ["second_captured_iteration_fails", "legacy_stream_handle",
                                      "records_leave_with_fgmres", "inner_tolerance_of_the_caller"])
def test_host_path(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
