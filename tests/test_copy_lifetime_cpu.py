"""Host lists that a plan copies to the device asynchronously live until a wait.

The library's objects are linked with a stand-in for the CUDA runtime that reads the
source of a host-to-device copy only when something waits (tests/host/copy_lifetime.cpp):
a list that is freed or rewritten before that shows as a late copy.  Plan creation,
trajectory updates and both failing after the copies were queued.
"""
import importlib.util
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    spec = importlib.util.spec_from_file_location("_nufft_build", os.path.join(ROOT, "paper_1710_03197_gb300", "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    build.build()
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    exe = str(tmp_path_factory.mktemp("host") / "copy_lifetime")
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(ROOT, "tests", "host", "copy_lifetime.cpp"), *objs, "-o", exe],
                   check=True)
    return exe


@pytest.mark.parametrize("fail_after", [-1, 0, 1])
@pytest.mark.parametrize("d,K,J,M", [(1, 1024, 6, 3000), (2, 64, 6, 1000), (2, 1000, 6, 40000), (3, 48, 4, 5000)])
def test_sources_live_until_the_wait(program, d, K, J, M, fail_after):
    r = subprocess.run([program, *map(str, (d, K, J, M, fail_after))], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    late, _, copies = r.stdout.split()[1:]
    assert int(copies) >= 2
    assert int(late) == 0, r.stdout
