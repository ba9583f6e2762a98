"""Host memory that an asynchronous copy reads or writes must stay until the
stream has been waited for. A runtime may run a copy from ordinary memory at
any time up to that point, so tests/host_copies.cpp runs the library's host
code against a stand-in runtime that holds all copies back and reports memory
freed before its copy: builds, component, partition and batch counts, and the
same with each device allocation failing in turn."""
import os
import shutil
import subprocess

import pytest

from paper_2609_21848_gb300 import buildlib

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_host_memory_is_freed_before_its_copy(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    objects = [os.path.join(buildlib.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in buildlib._sources()]
    newest = max(map(os.path.getmtime, buildlib._deps()))
    buildlib.build(force=not all(os.path.exists(o) and os.path.getmtime(o) >= newest for o in objects))
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(buildlib.nvcc()))), "include")
    exe = str(tmp_path / "host_copies")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", include, os.path.join(HERE, "host_copies.cpp"),
                        *objects, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout == "no host memory freed before its copy\n"
