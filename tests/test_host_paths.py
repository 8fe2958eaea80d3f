"""The library's host code on a CUDA runtime without a GPU (fake_cuda.cpp): what it does when a call of the
runtime refuses, and what it owes to a second device or stream."""

import os
import subprocess

import pytest

from paper_2111_12493_gb300 import build

TESTS = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    try:
        nvcc = build._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    build.build()
    objects = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    if not all(map(os.path.exists, objects)):
        build.build(force=True)
    out = tmp_path_factory.mktemp("host_paths")
    flags = [f if f != "-O3" else "-O1" for f in build.FLAGS] + ["-I", TESTS]
    made = []
    for src in ("host_paths.cu", "fake_cuda.cpp"):
        made.append(str(out / (src + ".o")))
        subprocess.run([nvcc, *build.ARCH, *flags, "-c", os.path.join(TESTS, src), "-o", made[-1]], check=True)
    exe = str(out / "host_paths")
    subprocess.run([nvcc, "-cudart", "none", *made, *objects, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("scenario", ["sort_on_two_devices", "wide_rows_on_two_devices", "loops_on_one_handle",
                                      "rounds_without_the_loop", "init_at_the_memory_limit"])
def test_host_path(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
