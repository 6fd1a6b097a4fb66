"""The host runtime (csrc/*.cpp) over a stand-in for the CUDA runtime and the kernels'
launchers (tests/cpp/host_runtime_test.cpp): failing calls, captures and replays."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2204_01287_gb300", "csrc")
SOURCE = os.path.join(ROOT, "tests", "cpp", "host_runtime_test.cpp")
with open(SOURCE) as f:
    SCENARIOS = re.findall(r'\{"(\w+)", \w+\},', f.read())


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("g++ and the CUDA headers are needed")
    out = tmp_path_factory.mktemp("runtime")
    files = [SOURCE] + [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith(".cpp")]
    procs = [subprocess.Popen([gxx, "-O1", "-std=c++17", "-pthread", "-ffp-contract=off", "-I", CSRC,
                               "-I", os.path.join(ROOT, "include"), "-I", cuda, "-c", f,
                               "-o", str(out / f"{i}.o")], stderr=subprocess.PIPE, text=True)
             for i, f in enumerate(files)]
    for p in procs:
        err = p.communicate()[1]
        assert p.returncode == 0, err
    exe = str(out / "runtime")
    subprocess.run([gxx, "-pthread", "-o", exe] + [str(out / f"{i}.o") for i in range(len(files))], check=True)
    return exe


@pytest.mark.parametrize("scenario", SCENARIOS)
def test_host_runtime(runtime, scenario):
    r = subprocess.run([runtime, scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert f"{scenario} ok" in r.stdout
