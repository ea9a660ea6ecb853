"""The library's host side on a stand-in CUDA runtime (host_runtime.cpp), without a GPU."""
import glob
import os
import subprocess

import pytest


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2411_17164_gb300 import build as b
    b.build()
    exe = str(tmp_path_factory.mktemp("host") / "host_runtime")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_runtime.cpp")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + cuda, "-o", exe, src, *sorted(glob.glob(os.path.join(b.OBJ, "*.o"))),
                    "-lpthread", "-ldl"], check=True)

    def call(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=60, check=True)
        return [line.split() for line in r.stdout.splitlines()]
    return call


def test_sources_of_copies_live_until_the_stream_is_waited_for(run):
    got = dict(run("copies"))
    assert got.pop("changed") == "0"
    assert set(got.values()) == {"0"}  # and the calls succeed


def test_every_path_launches_on_a_second_device(run):
    """Limits of dynamic shared memory belong to a device, not to the process."""
    got = dict(run("devices"))
    assert got.pop("refused") == "0" and len(got) == 12
    assert set(got.values()) == {"0"}
