"""Blocks that are not made of whole, equally placed 16-byte units (the launches of words) against
the oracle: the sizes at which a word, a chunk of 32 words or a group of rows begins and ends,
buffers that start anywhere, tori whose rows do not divide into groups, and meshes."""
import numpy as np
import pytest

from paper_1606_07676_b200 import binding as iso
from paper_1606_07676_b200 import workloads as wl
from schedule_sim import POISON, layout, make_request, oracle_result, send_buffer_np

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def a_launch_per_phase(monkeypatch):
    # the kernels of the launches per phase are what is tested here (test_tiles.py: all phases in one launch)
    monkeypatch.setenv("ISO_TILES", "0")

PLANS = ((iso.ISO_ALG_COMBINING, 1), (iso.ISO_ALG_COMBINING, 2), (iso.ISO_ALG_DIRECT, 1))


def _compare(w, lead=(0, 0), periodic=None, slabs=0, tiles=False):
    """Every schedule on buffers that start `lead` bytes behind an allocation; bands around both
    must stay as they were.  `tiles`: all phases of the combining schedules have to run in one launch."""
    import torch
    lens, sd, rd, ss, rs = layout(w)
    host = send_buffer_np(w, ss)
    band = 256
    raw_s = torch.full((band + lead[0] + w.P * ss + band,), 0x77, dtype=torch.uint8, device="cuda")
    raw_r = torch.full((band + lead[1] + w.P * rs + band,), POISON, dtype=torch.uint8, device="cuda")
    send = raw_s[band + lead[0]:band + lead[0] + w.P * ss]
    recv = raw_r[band + lead[1]:band + lead[1] + w.P * rs]
    send.copy_(torch.from_numpy(host.reshape(-1)))
    want = oracle_result(w, host, periodic=periodic)
    comm, req = make_request(w, send, recv, periodic)
    if slabs:
        iso.Iso_request_set_slabs(req, slabs)
    for alg, fusion in PLANS:
        iso.Iso_request_set_algorithm(req, alg, fusion)
        recv.fill_(POISON)
        iso.Iso_Start(req, torch.cuda.current_stream())
        iso.Iso_wait(req)
        st = iso.Iso_request_get_stats(req)
        assert not tiles or alg != iso.ISO_ALG_COMBINING or st["launches"] == 1, (w.name, w.dims, lead, fusion, st)
        got = raw_r.cpu().numpy()
        inside = got[band + lead[1]:band + lead[1] + w.P * rs].reshape(w.P, rs)
        assert np.array_equal(inside, want), (w.name, w.dims, lead, alg, fusion, np.argwhere(inside != want)[:1])
        assert (got[:band + lead[1]] == POISON).all() and (got[band + lead[1] + w.P * rs:] == POISON).all()
    assert (raw_s[:band].cpu().numpy() == 0x77).all()
    assert iso.Iso_request_check_guards(req) == 0
    iso.Iso_request_free(req)
    iso.Iso_comm_free(comm)


@pytest.mark.parametrize("m", [1, 2, 3, 4, 7, 8, 12, 13, 15, 17, 24, 31, 33, 40, 63, 65, 100, 127, 255, 481, 497, 1313])
@pytest.mark.parametrize("call", ["alltoall", "allgather"])
def test_block_sizes(m, call):
    for dims, offs in (((13, 11), wl.moore(2, 2)), ((6, 5, 7), wl.moore(3, 1)), ((4, 3, 3, 5), wl.positive_octant(4, 1))):
        w = wl.Workload("w", call, dims, offs, m, seed=m)
        _compare(w)
    _compare(wl.Workload("w", call, (13, 11), wl.moore(2, 1), m, seed=m + 1), lead=(m % 16, (3 * m) % 16))
    _compare(wl.Workload("w", call, (5, 9, 4), wl.moore(3, 1), m, seed=m + 2), periodic=[0, 1, 0])


@pytest.mark.parametrize("m", [113, 242, 252, 260, 371])
def test_blocks_over_two_chunks(m):
    # long blocks whose lanes do not fill a chunk of 32: they go on in the next one
    _compare(wl.Workload("w", "alltoall", (6, 5, 7), wl.moore(3, 1), m, seed=m), lead=(m % 16, 3))
    _compare(wl.Workload("w", "allgather", (13, 11), wl.moore(2, 2), m, seed=m + 1), periodic=[0, 1])


@pytest.mark.parametrize("seed", range(6))
def test_irregular_sizes(seed):
    rng = np.random.default_rng(seed)
    offs = wl.random_offsets(seed, 3, 30, -3, 3)
    lens = rng.choice([1, 2, 4, 5, 16, 31, 64, 100, 256, 511, 1024], size=30).astype(np.int64)
    w = wl.Workload("v", "alltoallv", (9, 8, 7), offs, 0, lens=lens, seed=seed)
    _compare(w, lead=[(0, 0), (4, 4), (1, 9)][seed % 3], periodic=None if seed % 2 else [1, 0, 1])


@pytest.mark.parametrize("m", [2, 4, 13, 40])
def test_many_rows_and_slabs(m):
    # every warp walks its ring several times; slabs whose edges fall inside a group of rows; rows
    # that are described several at a time
    _compare(wl.Workload("w", "alltoall", (61, 257), wl.moore(2, 2), m, seed=m))
    _compare(wl.Workload("w", "alltoall", (61, 257), wl.moore(2, 1), m, seed=m), slabs=7)
    _compare(wl.Workload("w", "alltoall", (96, 512), wl.moore(2, 1), m, seed=m), slabs=3)


@pytest.mark.parametrize("dims,offs,m", [((1300001,), wl.positive_octant(1, 1), 17), ((811, 803), wl.positive_octant(2, 1)[:1], 9),
                                         ((61, 53, 59), wl.moore(3, 3), 3), ((31, 30, 29), wl.moore(3, 3), 48), ((15, 14, 16, 17), wl.moore(4, 1), 20)])
def test_coordinates_without_a_table(dims, offs, m):
    # launches whose table of coordinates does not fit beside the rings: every lane divides
    _compare(wl.Workload("w", "allgather", dims, offs, m, seed=m))


@pytest.mark.parametrize("words", ["0", "1", None])
@pytest.mark.parametrize("m", [1, 2, 8, 12, 24, 72, 100, 120, 504])
def test_units_and_words(m, words, monkeypatch):
    """The same calls in units, as words and as the library chooses: strides that are multiples of 16 bytes
    (8 and 26 neighbours) and that are not (7 and 3), planes that divide into groups of rows and that do not."""
    if words is not None:
        monkeypatch.setenv("ISO_WORDS", words)
    for call in ("alltoall", "allgather"):
        for dims, offs in (((13, 11), wl.moore(2, 1)), ((12, 16), wl.positive_octant(2, 1)), ((5, 6, 7), wl.positive_octant(3, 1)),
                           ((6, 5, 4), wl.moore(3, 1)), ((3, 4, 3, 5), wl.positive_octant(4, 1)), ((301,), wl.moore(1, 2))):
            _compare(wl.Workload("w", call, dims, offs, m, seed=m), lead=(8, 8) if m % 8 == 0 and len(dims) == 2 else (0, 0))


@pytest.mark.parametrize("words", ["0", "1", None])
def test_units_and_words_mixed_sizes(words, monkeypatch):
    # faces, edges and corners; sizes from 1 to 1024 bytes; launches long enough for the rules of the library
    if words is not None:
        monkeypatch.setenv("ISO_WORDS", words)
    for r, side, dims in ((1, 9, (24, 35, 21)), (3, 7, (13, 11, 10)), (2, 12, (9, 10, 8))):
        offs = wl.moore(3, r)
        lens = np.asarray([side ** max(0, 3 - int(np.abs(v).sum())) for v in offs], np.int64)
        _compare(wl.Workload("v", "alltoallv", dims, offs, 0, lens=lens, seed=r))
    offs = wl.random_offsets(5, 3, 30, -3, 3)
    _compare(wl.Workload("v", "alltoallv", (9, 8, 7), offs, 0, lens=wl.random_sizes(5, 30, choices=(1, 2, 4, 31, 256, 1024)), seed=3))
    for call, dims, offs, m in (("alltoall", (120, 123), wl.positive_octant(2, 1), 120), ("allgather", (114, 102), wl.positive_octant(2, 3), 120),
                                ("allgather", (258, 139), wl.moore(2, 1), 120), ("allgather", (35, 34, 33), wl.positive_octant(3, 3), 8),
                                ("alltoall", (145571,), wl.moore(1, 1), 16), ("alltoall", (151916,), wl.moore(1, 1), 68), ("allgather", (89060,), wl.moore(1, 6), 24)):
        _compare(wl.Workload("w", call, dims, offs, m, seed=m))
