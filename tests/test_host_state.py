"""Host logic of the CUDA library's headers (buffers after a failed allocation,
use of a caller's arrays, joining of two streams, settings of a device), compiled with the host
compiler against a fake CUDA runtime: no GPU, and no fault on one, is needed to
see it."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("host") / "host_state")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-g", "-pthread",
                        "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_1902_00095_gb300", "csrc"),
                        os.path.join(HERE, "host_state.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("name", ["mlp_growth", "coupling_planes", "in_place", "fork_join",
                                  "per_device"])
def test_host_state(checks, name):
    r = subprocess.run([checks, name], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_no_setting_of_a_device_is_made_once_per_process():
    """A function-local static that asks for or sets something of the current
    device would hold for the first device only."""
    csrc = os.path.join(ROOT, "paper_1902_00095_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        src = open(os.path.join(csrc, name)).read()
        for m in re.finditer(r"static const [\w: ]+ \w+ = (?:\[[^;]*?\]\s*(?:\(\))?\s*\{.*?\n\s*\}"
                             r"(?:\(\))?;|[^;\[]*;)", src, re.S):
            assert not re.search(r"cudaFuncSetAttribute|cudaGetDevice\b|probe_\w+\(", m.group(0)), \
                (name, m.group(0))
