"""Dynamic shared memory beyond 48 KB, which a kernel has to be allowed on each
device before it is launched there: the library's own launch code against a
stand-in for the CUDA runtime (host/). Needs no GPU."""
import os
import subprocess

import pytest

from paper_2601_19901_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    objects = [os.path.join(build.BUILD, f) for f in ("splat.o", "interleave.o", "warp.o")]
    build.build(force=not all(map(os.path.exists, objects)))
    exe = str(tmp_path_factory.mktemp("host_launches") / "host_launches")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-cudart", "none",
           os.path.join(HERE, "host", "launches.cu"), os.path.join(HERE, "host", "fake_cudart.cpp"), *objects, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("what", ["devices", "retry", "threads"])
def test_shared_memory_is_allowed_where_a_launch_needs_it(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
