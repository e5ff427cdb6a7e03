"""The host side of the library against fakes of the kernel launchers and of
the CUDA runtime (api_harness.cu): what it launches, where results go and what
it returns when a call is refused, without a GPU."""
import os
import subprocess

import pytest

from paper_2206_11524_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("api")
    nvcc = build._nvcc()
    include = ["-I", build.INCLUDE, "-I", build.CSRC,
               "-I", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")]
    tests = os.path.join(ROOT, "tests")
    objs = []
    for src in (os.path.join(build.CSRC, "lbm_api.cu"), os.path.join(tests, "api_harness.cu"),
                os.path.join(tests, "api_fakes.cpp")):
        objs.append(str(d / (os.path.basename(src) + ".o")))
        compiler = [nvcc, *build.ARCH] if src.endswith(".cu") else ["g++"]
        subprocess.run([*compiler, "-std=c++17", "-O1", *include, "-c", src, "-o", objs[-1]],
                       check=True)
    exe = str(d / "api_harness")
    subprocess.run(["g++", *objs, "-lpthread", "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("check", ["misaligned_destination", "device_destination", "refused_choice",
                                   "undefined_state", "step_choice"])
def test_host_side(harness, check):
    out = subprocess.run([harness, check], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
