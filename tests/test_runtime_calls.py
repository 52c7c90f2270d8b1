"""What the library asks of the CUDA runtime, without a GPU: its objects linked with a stand-in for the runtime
(tests/fake_runtime.cpp) that launches nothing and checks what it is given."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2412_00802_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    exe = tmp_path_factory.mktemp("runtime") / "fake_runtime"
    cuda = os.path.dirname(os.path.dirname(build.NVCC))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", build.CSRC,
                           os.path.join(ROOT, "tests", "fake_runtime.cpp"), *objs, "-o", str(exe), "-lpthread"])
    return str(exe)


@pytest.mark.parametrize("scenario", ["examples_plan", "examples_one_shot", "second_device", "split_products", "role_block",
                                      "autotune_workspace"])
def test_scenario(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
