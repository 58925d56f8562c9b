"""Host code of the engine and the autotuners on a fake CUDA runtime (host_engine.cpp)."""
import os
import subprocess

import pytest

from paper_1705_00103_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("host") / "host_engine")
    src = [os.path.join(build.CSRC, f) for f in ("batch.cpp", "solve.cpp", "plan.cpp")]
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I", build.INCLUDE, "-I", build.CSRC, "-I",
                           build._cuda_include(), os.path.join(HERE, "host_engine.cpp"), *src, "-o", exe,
                           "-Wl,--unresolved-symbols=ignore-all"])
    return exe


@pytest.mark.parametrize("scenario", ["batch_while_tuned", "engine_tuned_depth", "plan_tuned_depth",
                                      "steps_follow_requests", "graph_kept_in_first_burst"])
def test_scenario(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
