"""Schedules whose intermediate blocks fit in shared memory: all phases in one launch, tile by tile.  The plan is
executed on the host against the schedule's parts; the kernel runs against the oracle."""
import os
import subprocess

import numpy as np
import pytest

from paper_1606_07676_b200 import binding as iso
from paper_1606_07676_b200 import workloads as wl
from schedule_sim import POISON, oracle_result
from test_gpu_fuzz import expected, make_request, random_cases
from test_gpu_parity import Run
from test_gpu_words import _compare

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1606_07676_b200", "csrc")


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("tiles") / "tiles_sim")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC, os.path.join(ROOT, "tests", "tiles_sim.cpp")] +
                          [os.path.join(CSRC, f) for f in ("iso_schedule.cpp", "iso_words.cpp", "iso_tiles.cpp")] + ["-o", exe])
    return exe


def test_plans_on_the_host(planner):
    for seed in ("1", "2", "3"):
        out = subprocess.run([planner, seed], capture_output=True, text=True, timeout=300)
        assert out.returncode == 0 and int(out.stdout) > 150, out.stdout + out.stderr


def chosen(planner, calls):
    """Bytes of a row's places for every (kind, sides, vectors, bytes of the blocks, fusion level, periodic), 0: not in tiles."""
    lines = []
    for kind, dims, offs, lens, *more in calls:
        fusion, periodic = (more + [1, None][len(more):])
        offs = np.asarray(offs)
        lens = np.broadcast_to(np.asarray(lens), len(offs))
        lines.append(" ".join(str(int(x)) for x in [("alltoall", "allgather", "alltoallv").index(kind), fusion, len(dims), *dims,
                                                    *(periodic or [1] * len(dims)), len(offs), *offs.reshape(-1), *lens]))
    out = subprocess.run([planner, "choices"], input="\n".join(lines) + "\n", capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    return [int(x) for x in out.stdout.split()]


def test_calls_that_are_slower_in_tiles(planner):
    # microseconds in phases and in tiles as once chosen: 97 and 228, 30 and 51, 30 and 46, 28 and 41, 21 and 27
    assert not any(chosen(planner, [("allgather", (35, 16, 27), wl.moore(3, 3), 56), ("allgather", (24, 34, 27), wl.moore(3, 2), 24),
                                    ("allgather", (23, 23, 24), wl.moore(3, 2), 56, 2), ("allgather", (25, 38, 23), wl.moore(3, 2), 24, 2),
                                    ("allgather", (512, 256), wl.moore(2, 2), 16)]))
    # blocks that need no hop stay out of the places where these are long: 39 and 21 (phases 21), 47 and 24 (28)
    assert chosen(planner, [("alltoall", (30, 24), wl.moore(2, 3), 968), ("alltoall", (10, 9, 14), wl.moore(3, 1), 1480, 2)]) == [34896, 23744]
    # and, in tiles: 36 and 27, 19 and 13.5, 165 and 127, 5.4 and 3.2, 98 and 65
    faces = [32 ** max(0, 3 - int(np.abs(v).sum())) for v in wl.moore(3, 1)]
    assert all(chosen(planner, [("alltoall", (32, 32, 32), wl.moore(3, 1), 64), ("allgather", (32, 32, 32), wl.moore(3, 1), 64),
                                ("alltoallv", (32, 32, 32), wl.moore(3, 1), faces, 1, [0, 1, 0]), ("alltoall", (8, 8), wl.moore(2, 1), 8)]))


def test_no_kernel_spills(tmp_path):
    src = tmp_path / "kernels.cu"
    kernels = ["iso_gather_tiles<%d, %s>" % (w, mesh) for w in (0, 4, 8, 16) for mesh in ("false", "true")]
    src.write_text('#include "iso_tiles.cuh"\nnamespace iso {\n' +
                   "".join("template __global__ void %s(const __grid_constant__ TilesDev);\n" % k for k in kernels) + "}\n")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    out = subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-Xptxas", "-v", "-I", os.path.join(ROOT, "include"),
                          "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "kernels.o")], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    spills = [ln for ln in out.stderr.splitlines() if "spill stores" in ln]
    assert len(spills) >= len(kernels) and all("0 bytes spill stores" in ln for ln in spills), out.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("m", [1, 2, 3, 4, 7, 8, 12, 13, 16, 17, 24, 33, 48, 64, 100, 225, 256])
@pytest.mark.parametrize("call", ["alltoall", "allgather"])
def test_block_sizes(m, call, monkeypatch):
    # tiles of one row and of many, a narrower last one, several tiles to a CTA (257x131), buffers that start anywhere, meshes
    monkeypatch.setenv("ISO_TILES", "1")
    for dims, offs in (((13, 11), wl.moore(2, 2)), ((6, 5, 7), wl.moore(3, 1)), ((4, 3, 3, 5), wl.positive_octant(4, 1)), ((257, 131), wl.moore(2, 1))):
        _compare(wl.Workload("w", call, dims, offs, m, seed=m), tiles=True)
    _compare(wl.Workload("w", call, (13, 11), wl.moore(2, 1), m, seed=m + 1), lead=(m % 16, (3 * m) % 16), tiles=True)
    _compare(wl.Workload("w", call, (5, 9, 4), wl.moore(3, 1), m, seed=m + 2), periodic=[0, 1, 0], tiles=True)


@pytest.mark.gpu
@pytest.mark.parametrize("tiles", ["2", "3"])
def test_blocks_that_need_no_hop(tiles, monkeypatch):
    # through places, to be copied on from there, and past them
    monkeypatch.setenv("ISO_TILES", tiles)
    for m in (1, 6, 13, 24, 41, 100):
        _compare(wl.Workload("w", "alltoall", (13, 11), wl.moore(2, 2), m, seed=m), lead=(m % 4, 0), tiles=True)
        _compare(wl.Workload("w", "allgather", (7, 5, 6), wl.moore(3, 1), m, seed=m), periodic=[1, 0, 1], tiles=True)
    for seed, dims in ((1, (9, 8, 7)), (2, (31, 17))):
        offs = wl.random_offsets(seed, len(dims), 20, -2, 2)
        _compare(wl.Workload("v", "alltoallv", dims, offs, 0, lens=wl.random_sizes(seed, 20, choices=(1, 2, 4, 31, 64, 256)), seed=seed), tiles=True)


@pytest.mark.gpu
def test_rows_of_several_kilobytes(monkeypatch):
    # a table of units that stays where it is: longer than 1600 and more than two tiles to an SM
    monkeypatch.setenv("ISO_TILES", "1")
    _compare(wl.Workload("w", "alltoall", (33, 31), wl.moore(2, 3), 784, seed=1), tiles=True)
    _compare(wl.Workload("w", "allgather", (133, 131), wl.moore(2, 1), 389, seed=2), tiles=True)


@pytest.mark.gpu
def test_buffers_of_more_than_four_gigabytes(monkeypatch):
    import oracle
    import torch
    monkeypatch.setenv("ISO_TILES", "1")
    dims, offs, m = (512, 257), wl.moore(2, 1), 4160       # 4.4 GB received
    P, s = 512 * 257, len(offs)
    send = wl.payload_torch("uint8", 9, 0, P * m, "cuda")
    recv = torch.full((P, s * m), POISON, dtype=torch.uint8, device="cuda")
    comm = iso.Iso_neighborhood_create(dims, offs)
    req = iso.Iso_neighbor_allgather_init(send, m, 1, recv, m, 1, comm)
    iso.Iso_Start(req, torch.cuda.current_stream())
    iso.Iso_wait(req)
    assert iso.Iso_request_get_stats(req)["launches"] == 1 and recv.numel() > 1 << 32
    host = send.cpu().numpy()
    for r0 in (0, P // 3, int((1 << 31) // (s * m)) - 5, int((1 << 32) // (s * m)) - 5, P - 300):
        assert np.array_equal(recv[r0:r0 + 300].cpu().numpy(), oracle.allgather(dims, offs, m, host, r0, r0 + 300)), r0
    iso.Iso_request_free(req)
    iso.Iso_comm_free(comm)


@pytest.mark.gpu
def test_long_sides(monkeypatch):
    monkeypatch.setenv("ISO_TILES", "1")
    _compare(wl.Workload("w", "alltoall", (70001, 3), wl.moore(2, 1), 16, seed=1), tiles=True)
    _compare(wl.Workload("w", "allgather", (3, 70001), wl.moore(2, 1), 12, seed=2), tiles=True)


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["cfg1", "cfg2_alltoall", "cfg2_allgather", "stencil_mesh", "irregular", "cfg3_m64"])
def test_configurations_as_the_library_runs_them(name):
    """Nothing asked for: the small ones and those of 32 768 processes in tiles, 65 536 processes with 24 blocks of 64 bytes as the
    library sees fit."""
    periodic = None
    if name == "stencil_mesh":
        offs = wl.moore(3, 1)
        lens = np.asarray([32 ** max(0, 3 - int(np.abs(v).sum())) for v in offs], np.int64)
        w, periodic = wl.Workload("v", "alltoallv", (32, 32, 32), offs, 0, lens=lens, seed=1), [0, 1, 0]
    elif name == "irregular":
        offs = wl.random_offsets(1, 2, 30, -3, 3)
        w = wl.Workload("v", "alltoallv", (120, 130), offs, 0, lens=wl.random_sizes(1, 30), seed=2)
    else:
        w = wl.config(name)
    import torch
    run = Run(torch, w, periodic=periodic)
    want = oracle_result(w, run.send_host, periodic=periodic)
    for _ in range(2):
        got = run.result(iso.ISO_ALG_COMBINING, 1)
        assert np.array_equal(got, want)
    assert name == "cfg3_m64" or iso.Iso_request_get_stats(run.req)["launches"] == 1
    run.close()


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", range(8))
def test_random_cases(chunk, monkeypatch):
    import torch
    monkeypatch.setenv("ISO_TILES", "1")
    in_tiles = 0
    for c in random_cases(300 + chunk):
        P, ss, rs = c["P"], c["ss"], c["rs"]
        if not rs or not P * ss:
            continue
        send = torch.from_numpy(c["send_h"]).cuda()
        recv = torch.empty((P, rs), dtype=torch.uint8, device="cuda")
        comm, req = make_request(c, send, recv)
        want = expected(c)
        for fusion in (1, 2, 3):
            iso.Iso_request_set_algorithm(req, iso.ISO_ALG_COMBINING, fusion)
            for _ in range(2):
                recv.fill_(POISON)
                iso.Iso_Start(req, torch.cuda.current_stream())
            iso.Iso_wait(req)
            assert np.array_equal(recv.cpu().numpy(), want), dict(chunk=chunk, trial=c["trial"], dims=c["dims"], kind=c["kind"], fusion=fusion,
                                                                  periodic=c["periodic"], lens=c["lens"].tolist())
            st = iso.Iso_request_get_stats(req)
            in_tiles += st["phases"] > 1 and st["launches"] == 1
        iso.Iso_request_free(req)
        iso.Iso_comm_free(comm)
    assert in_tiles >= 10


@pytest.mark.gpu
def test_left_to_the_library_and_asked_for():
    """Small calls run in one launch unless something else is asked for; in a graph of the caller's and on another stream
    as well."""
    import torch
    w = wl.Workload("w", "alltoall", (8, 6, 7), wl.moore(3, 1), 24, seed=3)
    send = wl.payload_torch("uint8", 3, 0, w.P * w.s * 24, "cuda").view(w.P, w.s * 24)
    recv = torch.empty_like(send)
    import oracle
    want = oracle.alltoall(w.dims, w.offsets, 24, send.cpu().numpy())
    comm = iso.Iso_neighborhood_create(w.dims, w.offsets)
    req = iso.Iso_neighbor_alltoall_init(send, 24, 1, recv, 24, 1, comm)

    def start(stream=None):
        recv.fill_(POISON)
        torch.cuda.synchronize()
        iso.Iso_Start(req, stream or torch.cuda.current_stream())
        iso.Iso_wait(req)
        assert np.array_equal(recv.cpu().numpy(), want)
        return iso.Iso_request_get_stats(req)["launches"]

    assert start() == 1
    assert start(torch.cuda.Stream()) == 1
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        iso.Iso_Start(req, torch.cuda.current_stream())
    recv.fill_(POISON)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(recv.cpu().numpy(), want)
    iso.Iso_request_set_single_launch(req, False)
    assert start() == 3
    iso.Iso_request_set_single_launch(req, None)
    assert start() == 1
    iso.Iso_request_set_single_launch(req, True)    # (24-byte blocks do not run in a cooperative launch)
    assert start() == 3
    iso.Iso_request_set_single_launch(req, None)
    assert start() == 1
    iso.Iso_request_free(req)
    req = iso.Iso_neighbor_alltoall_init(send, 24, 1, recv, 24, 1, comm)
    iso.Iso_request_set_graph(req, True)
    assert start() == 3
    iso.Iso_request_free(req)
    iso.Iso_comm_free(comm)


@pytest.mark.gpu
def test_execution_read_back_and_tuned(monkeypatch):
    """What is reported is what runs, and asked for on another request it runs there too; the tuner knows this route
    whatever the request was told before."""
    import torch

    def bound(w):
        send = wl.payload_torch("uint8", 3, 0, w.P * w.s * w.block_bytes, "cuda")
        recv = torch.empty_like(send)
        comm = iso.Iso_neighborhood_create(w.dims, w.offsets)
        req = iso.Iso_neighbor_alltoall_init(send, w.block_bytes, 1, recv, w.block_bytes, 1, comm)
        iso.Iso_comm_free(comm)
        return send, recv, req

    def launches(req):
        iso.Iso_Start(req, torch.cuda.current_stream())
        iso.Iso_wait(req)
        return iso.Iso_request_get_stats(req)["launches"]

    small = wl.Workload("w", "alltoall", (8, 6, 7), wl.moore(3, 1), 24, seed=3)
    one, two = bound(small), bound(small)
    assert launches(one[2]) == 1
    ex = iso.Iso_request_get_execution(one[2])
    assert ex == {"slabs": 1, "chains": 1, "graph": 0}
    iso.Iso_request_set_slabs(two[2], ex["slabs"])
    iso.Iso_request_set_chains(two[2], ex["chains"])
    iso.Iso_request_set_graph(two[2], bool(ex["graph"]))
    assert launches(two[2]) == 1
    iso.Iso_request_set_single_launch(one[2], False)
    assert launches(one[2]) == 3
    iso.Iso_request_tune(one[2], torch.cuda.current_stream())   # 3.1 microseconds against 7
    assert launches(one[2]) == 1
    iso.Iso_request_set_slabs(two[2], 2)
    assert launches(two[2]) == 6
    large = bound(wl.Workload("w", "alltoall", (128, 128), wl.moore(2, 2), 1024, seed=4))
    iso.Iso_request_set_slabs(large[2], 1)      # (in two chains of slabs otherwise)
    assert launches(large[2]) == 2
    monkeypatch.setenv("ISO_TILES", "1")
    many = bound(wl.Workload("w", "alltoall", (256, 256), wl.moore(2, 2), 64, seed=4))  # (two slabs, were it run in phases)
    assert launches(many[2]) == 1 and iso.Iso_request_get_execution(many[2]) == ex
    for b in (one, two, large, many):
        iso.Iso_request_free(b[2])


@pytest.mark.gpu
@pytest.mark.parametrize("recorded", [False, True])
def test_launches_are_set_up_when_host_buffers_need_them(recorded):
    """A request whose starts run in tiles allocates no intermediate buffer; the host-buffer path, which runs the launches slab by
    slab, makes up for it, in between starts and inside a graph of the caller's too."""
    import torch
    import oracle
    w = wl.Workload("w", "alltoall", (32, 32, 32), wl.moore(3, 1), 64, seed=3)
    n = w.P * w.s * 64
    host_s = wl.payload_torch("uint8", 4, 0, n, "cuda").cpu().pin_memory()
    host_r = torch.zeros(n, dtype=torch.uint8).pin_memory()
    send, recv = wl.payload_torch("uint8", 3, 0, n, "cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
    comm = iso.Iso_neighborhood_create(w.dims, w.offsets)
    req = iso.Iso_neighbor_alltoall_init(send, 64, 1, recv, 64, 1, comm)
    want = [oracle.alltoall(w.dims, w.offsets, 64, x.cpu().numpy().reshape(w.P, -1)).reshape(-1) for x in (send, host_s)]

    def start(expect):
        recv.fill_(POISON)
        iso.Iso_Start(req, torch.cuda.current_stream())
        iso.Iso_wait(req)
        assert np.array_equal(recv.cpu().numpy(), expect) and iso.Iso_request_get_stats(req)["launches"] == 1

    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    start(want[0])
    assert free - torch.cuda.mem_get_info()[0] < (16 << 20)     # (the intermediate buffer has 58 MB)
    if recorded:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            iso.Iso_Start_host(req, host_s, host_r, torch.cuda.current_stream())
        graph.replay()
        torch.cuda.synchronize()
    else:
        iso.Iso_Start_host(req, host_s, host_r, torch.cuda.current_stream())
        iso.Iso_wait(req)
        assert iso.Iso_request_get_host_transfer_ms(req)["slabs"] > 1
    assert np.array_equal(host_r.numpy(), want[1])
    start(want[1])      # (the send buffer holds what came from the host)
    assert iso.Iso_request_check_guards(req) == 0
    if not recorded:
        for _ in range(3):
            host_r.zero_()
            iso.Iso_Start_host(req, host_s, host_r, torch.cuda.current_stream())
            iso.Iso_wait(req)
            assert np.array_equal(host_r.numpy(), want[1])
    iso.Iso_request_free(req)
    iso.Iso_comm_free(comm)


@pytest.mark.gpu
def test_the_benchmark_measures_the_default():
    import sys
    import torch
    sys.path.insert(0, ROOT)
    import bench
    b = bench.Bound(torch, iso, wl, "cfg2_alltoall")
    assert b.set(iso.ISO_ALG_COMBINING, 1)["launches"] == 1
    b.close()


@pytest.mark.gpu
@pytest.mark.parametrize("m", [1, 8, 13, 16, 40, 100, 497])
def test_a_launch_per_phase_of_small_calls(m, monkeypatch):
    # the kernels that small calls used to run
    monkeypatch.setenv("ISO_TILES", "0")
    for call in ("alltoall", "allgather"):
        for dims, offs in (((13, 11), wl.moore(2, 2)), ((6, 5, 7), wl.moore(3, 1)), ((4, 3, 3, 5), wl.positive_octant(4, 1))):
            _compare(wl.Workload("w", call, dims, offs, m, seed=m))
        _compare(wl.Workload("w", call, (13, 11), wl.moore(2, 1), m, seed=m + 1), lead=(m % 16, (3 * m) % 16))
        _compare(wl.Workload("w", call, (5, 9, 4), wl.moore(3, 1), m, seed=m + 2), periodic=[0, 1, 0])
