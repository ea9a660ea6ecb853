"""The library's host side on a stand-in CUDA runtime (host_runtime.cpp), without a GPU."""
import ctypes as C
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


@pytest.mark.parametrize("H", [256, 512])
def test_wide_workspace_holds_what_the_path_reads(H):
    """Per edge: five fp32 rows (pre-activation, last edge state, its gradient, receiver and sender parts), the gathered
    bf16 operand of 3H, three bf16 rows, one fp32 product, the four edge inputs."""
    from paper_2411_17164_gb300 import build, xmgn
    build.build()

    def ws(E):
        w, c = C.c_size_t(), C.c_size_t()
        d = xmgn.ModelDesc(H, 3, 6, 4, xmgn.XMGN_BF16)
        assert xmgn.lib().xmgn_model_ws(C.byref(d), 50_000, E, C.byref(w), C.byref(c)) == 0
        return w.value

    need = 5 * 4 * H + 2 * 3 * H + 3 * 2 * H + 4 * H + 16
    assert ws(400_000) - ws(300_000) <= 100_000 * need + 100_000  # and the block partials of the column sums


@pytest.mark.parametrize("n", [2000, 200_000])
def test_tuner_times_the_products_with_their_sums(run, n):
    """The grid of the node-level products trades their time for the partials to be summed: both are inside the events."""
    out = run("timed", 3, n)
    assert out[0] == ["status", "0"]
    names = [v[1] for v in out if v[0] == "launch"]
    at = [i for i, v in enumerate(names) if v == "event"]
    assert len(at) >= 8 and len(at) % 2 == 0
    for a, b in zip(at[::2], at[1::2]):
        inside = names[a + 1:b]
        assert any("tc_gemm_tn_kernel" in v for v in inside) and any("reduce_parts_kernel" in v for v in inside)
