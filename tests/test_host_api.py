"""The library's host code (allocation, launch and stream logic of the C ABI) on
the CPU: its objects linked with the stand-in CUDA runtime of
tests/host_runtime.cpp, which records the work and can fail a chosen call."""
import os
import subprocess

import numpy as np
import pytest

from paper_2605_14505_gb300 import build, lbm

from _strips import LARGE, PLANS

HERE = os.path.dirname(os.path.abspath(__file__))
STORAGES = {"fp32": 0, "fp16": 1, "bf16": 2}


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    try:
        nvcc = build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    build.build()
    exe = str(tmp_path_factory.mktemp("host_api") / "host_api")
    objs = [os.path.join(build.OBJDIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    cmd = [nvcc] + build.ARCH + ["-O1", "-std=c++17", "-I" + build.CSRC, "-I" + os.path.join(build.ROOT, "include"),
                                 "-cudart", "none", "-o", exe, os.path.join(HERE, "host_api.cu"),
                                 os.path.join(HERE, "host_runtime.cpp")] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

    def run(*args):
        r = subprocess.run([exe] + [str(a) for a in args], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout.strip().splitlines()

    return run


@pytest.mark.parametrize("fused", [0, 1])
def test_a_record_after_a_failed_one_has_its_scratch(host, fused):
    """Whichever allocation of the first record fails, that call says so and
    launches nothing; the next one passes kernels live scratch with a cleared
    block count, and nothing outlives the handle."""
    lines = [line.split() for line in host("record", fused)]
    assert len(lines) >= 6
    for k, (_, _, first, _, launches, _, second, _, scratch, _, left) in enumerate(lines):
        assert int(first) == (-2 if k < len(lines) - 1 else 0), lines[k]
        assert launches == "0", lines[k]
        assert (second, scratch, left) == ("0", "1", "0"), lines[k]


@pytest.mark.parametrize("call", ["step", "record"])
def test_a_batch_call_after_a_failed_one_runs_on_its_streams(host, call):
    """Whichever stream, event or scratch of a per-instance batch call cannot be
    had, that call fails and the next one runs every instance on a stream of
    the batch; records take no more streams than they use."""
    lines = [line.split() for line in host("batch", call)]
    assert len(lines) >= 12
    for k, (_, _, first, _, _, _, second, _, null, _, streams, _, left) in enumerate(lines):
        assert (int(first) < 0) == (k < len(lines) - 1), lines[k]
        assert (second, null, left) == ("0", "0", "0"), lines[k]
    assert int(lines[-1][10]) == (12 if call == "step" else 8)
    if call == "record":   # 8 streams and events, then each instance's scratch
        assert [line[2] for line in lines[:17]] == ["-3"] * 16 + ["-2"]


@pytest.mark.parametrize("call", ["step", "record"])
def test_a_failed_batch_call_leaves_no_chain_behind(host, call):
    """Whatever the chains were given before a call failed, the batch's stream
    waits for it: later work on that stream (another initialisation, a step, an
    instance's own record) does not run beside it."""
    for line in host("batch", call):
        assert line.split()[4] == "0", line


@pytest.mark.parametrize("short_by,status,launches", [(-64, 0, 2), (0, 0, 2), (1, -1, 0), (5000, -1, 0)])
def test_halo_buffers_are_as_long_as_said(host, short_by, status, launches):
    """A buffer that ends at its last byte is taken, one that ends before it is
    refused with nothing launched."""
    assert host("halo", short_by) == [f"pack {status} unpack {status} launches {launches}"] * 4


@pytest.mark.parametrize("n,pair,storage,even,odd", [
    (16, "27x27", "fp32", "64 shaped overlapped", "128 shaped overlapped"),
    (26, "27x27", "fp32", "64 shaped overlapped", "128 shaped overlapped"),   # 17576 of 19456 nodes
    (28, "27x27", "fp32", "64 shaped alone", "128 shaped alone"),
    (33, "27x27", "fp32", "128 flat alone", "128 flat alone"),
    (36, "27x27", "fp32", "64 flat alone", "64 flat alone"),
    (24, "27x19", "fp32", "64 flat overlapped", "64 flat overlapped"),
    (32, "27x19", "fp32", "64 shaped alone", "64 shaped alone"),
    (32, "19x19", "fp32", "64 shaped overlapped", "64 shaped overlapped"),
    (20, "27x19", "fp16", "128 flat overlapped", "128 flat overlapped"),
    (32, "27x27", "fp16", "128 flat overlapped", "128 flat overlapped"),
    (31, "27x19", "bf16", "64 shaped overlapped", "64 shaped overlapped"),    # one node per thread
    (64, "27x27", "fp32", "64 shaped overlapped", "128 shaped overlapped"),   # more than a wave
])
def test_launches_of_small_lattices(host, n, pair, storage, even, odd):
    """Steps overlap their launches except FP32 pairs of 46 and more values between
    two 64-thread blocks per SM and one wave; D3Q27xD3Q27 keeps its block shape
    up to three such blocks per SM."""
    assert host("launches", n, n, n, lbm.PAIRS[pair], STORAGES[storage]) == [even, odd]


def _calls(lines):
    """Steps of each call and its launches (graph replay?, parity, z0, planes, y0, rows, down)."""
    calls = []
    for line in lines:
        words = line.split()
        if words[0] == "call":
            calls.append((int(words[1]), []))
        else:
            calls[-1][1].append((words[0] == "graph",) + tuple(int(w) for w in words[-6:]))
    return calls


def test_a_box_of_one_strip_steps_whole(host):
    """106 MB between 3/4 and 0.8 of L2 with too few planes and rows for two
    strips: whole-lattice steps, replayed 64 to a graph from the first call."""
    (_, launches), (_, more) = _calls(host("steps", 1000, 24, 24, 0, 0, 130, 64))
    assert [x[0] for x in launches] == [True] * 128 + [False] * 2
    assert [x[0] for x in more] == [True] * 64
    assert all(x[2:6] == (0, 24, 0, 24) for x in launches + more)


@pytest.mark.parametrize("shape,pair,storage,jz,jy", PLANS + LARGE)
def test_every_strip_follows_its_neighbours(host, shape, pair, storage, jz, jy):
    """The library's launches of calls that end a group early, start at either
    parity and replay the graph: no node steps before a neighbour's previous
    step or after its next one, every node takes every step at its parity, and
    a step takes a launch per strip."""
    _, ny, nz = shape
    counts = (5, 18) if shape == (512, 512, 512) else (19, 4, 37, 90, 33)
    steps = np.zeros((nz, ny), dtype=int)
    total, replays = 0, 0
    for n, launches in _calls(host("steps", *shape, lbm.PAIRS[pair], STORAGES[storage], *counts)):
        for graph, odd, z0, planes, y0, rows, _ in launches:
            replays += graph
            z, y = (np.arange(a, a + c) % m for a, c, m in ((z0, planes, nz), (y0, rows, ny)))
            done = steps[np.ix_(z, y)]
            now = done.flat[0]
            assert (done == now).all() and now % 2 == odd
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    near = steps[np.ix_((z + dz) % nz, (y + dy) % ny)]
                    assert ((near == now) | (near == now + 1)).all()
            steps[np.ix_(z, y)] += 1
        total += n
        assert (steps == total).all()
        assert len(launches) == jz * jy * n
    assert bool(replays) == (len(counts) > 2)


@pytest.mark.parametrize("n,pair,threads,flat,batched", [
    (128, "27x19", 64, 0, 0), (129, "27x19", 128, 1, 0), (160, "19x7", 256, 0, 0), (96, "27x19", 64, 0, 1),
    (60, "27x19", 64, 0, 0),
])
def test_autotune_times_what_is_stepped(host, n, pair, threads, flat, batched):
    """Launches with a known cost: the time returned is the one of the steps after
    it, at the cheapest shape, and a lattice that steps in strips (one alone in
    its round of a batch too) is timed in strips only."""
    (whole, timed, ms, spent), = (line.split() for line in host("autotune", n, lbm.PAIRS[pair], threads, flat, batched))
    strips = n >= 96
    assert int(timed) > 0 and (int(whole) == 0) == strips, (whole, timed)
    assert float(ms) == pytest.approx(float(spent), rel=1e-5)
    assert float(ms) == pytest.approx(1e-9 * n ** 3 * (2 if batched else 1), rel=1e-5)


@pytest.mark.parametrize("n,pair,storage", [(32, "19x7", "fp32"), (128, "27x19", "fp32"), (64, "27x19", "fp16")])
def test_launches_are_counted(host, n, pair, storage):
    """Eager launches, whole and in strips, graph replays, and the passes of records
    with and without a first sum of their rows."""
    counts = [line.split() for line in host("count", n, lbm.PAIRS[pair], STORAGES[storage])]
    assert all(a == b for a, b in counts) and int(counts[-1][0]) > 2 * (1 + 70 + 33 + 300)
