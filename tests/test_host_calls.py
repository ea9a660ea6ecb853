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


@pytest.mark.parametrize("H", [32, 128, 256, 512])
@pytest.mark.parametrize("rows", [300, 5000, 60000, 354000, 1500000])
def test_fp32_weight_gradient_chains_are_bounded(run, H, rows):
    """No weight gradient of the FP32 path sums more than max(4096, M / 128) rows in one running sum (a graph with as
    many nodes as edges, so that M is one number), and the partial sums of different buffers do not meet."""
    out = run("products", H, rows)
    assert out[0] == ["status", "0"]
    chunks = [int(v[1]) for v in out if v[0] == "chunks"]
    assert len(chunks) >= 10
    for c in chunks:
        assert 16 * -(--(-rows // c) // 16) <= max(4096, 16 * -(--(-rows // 128) // 16)), (c, rows)
    room = {}
    for _, base, nb, ln in (v for v in out if v[0] == "parts"):
        room[int(base)] = max(room.get(int(base), 0), 4 * int(nb) * int(ln))
    at = sorted(room)
    for a, b in zip(at, at[1:]):
        assert a + room[a] <= b
