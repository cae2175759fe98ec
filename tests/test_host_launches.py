"""The library's own launch code against a stand-in for the CUDA runtime (host/):
dynamic shared memory beyond 48 KB, which a kernel has to be allowed on each
device before it is launched there, and what the host computes for a launch.
Needs no GPU."""
import os
import subprocess

import pytest

from paper_2601_19901_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ("splat", "interleave", "warp")


def _link(exe, objects, flags=()):
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, *flags, "-I", build.CSRC, "-cudart", "none",
           os.path.join(HERE, "host", "launches.cu"), os.path.join(HERE, "host", "fake_cudart.cpp"), *objects, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    objects = [os.path.join(build.BUILD, f + ".o") for f in UNITS]
    build.build(force=not all(map(os.path.exists, objects)))
    return _link(str(tmp_path_factory.mktemp("host_launches") / "host_launches"), objects)


@pytest.mark.parametrize("what", ["devices", "retry", "threads"])
def test_shared_memory_is_allowed_where_a_launch_needs_it(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("what", ["tent", "gauss", "units", "splits"])
def test_a_launch_takes_the_form_that_is_faster(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_a_phase_that_is_no_number_is_not_made_an_integer(tmp_path):
    """With the host code's float to integer conversions checked."""
    flags = ["-Xptxas", "-O0", "-Xcompiler", "-fsanitize=float-cast-overflow,-fno-sanitize-recover=all"]
    objects = []
    for f in UNITS:
        objects.append(str(tmp_path / (f + ".o")))
        cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, *flags, "-c", os.path.join(build.CSRC, f + ".cu"), "-o", objects[-1]]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    exe = _link(str(tmp_path / "checked"), objects, flags)
    r = subprocess.run([exe, "tiny_pitch"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
