"""Timed cases: isomorphic neighbourhood collectives as a program on one GPU calls them.

A program creates a neighbourhood once, binds its buffers with one of the ``..._init`` calls
and then starts the request in every time step of its own loop; so `prepare` does the former
and `run` is one start.  The schedule is the default one (message combining, one launch per
dimension) unless the case says otherwise: "direct" is what a program on one GPU chooses when
it only wants the result, "combining2" takes two dimensions per phase.

The sizes are those of this repository's configurations (`workloads.config`) and, for the
odd ones, of the same kind: tori whose sides are odd numbers, blocks of a few doubles or of an
odd number of bytes, non-periodic edges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_07676_b200 import binding as iso
from paper_1606_07676_b200 import workloads as wl


def _case(name, call, torus, neighbours, block, element, schedule="combining", mesh=False, entry="start"):
    """`call`: alltoall, allgather or alltoallv; `torus`: its sides, as text; `neighbours`: moore<r>,
    octant<r>, shells<r>+<r> or random<s>; `block`: bytes of a block, or the rule of an irregular
    collective's sizes; `element`: bytes of an element; `mesh`: the first and the last dimension do not wrap
    around; `entry`: start (buffers on the device) or host (buffers in page-locked host memory)."""
    case = {"call": call, "torus": torus, "neighbours": neighbours, "block": block, "element": element,
            "schedule": schedule, "mesh": mesh, "entry": entry}
    return dict(case, name=name) if name else case


def listed():
    return [
        # 64 processes, two integers per neighbour: nothing but latency and launches
        _case("tiny_2d", "alltoall", "8x8", "moore1", "8", 4),
        # 27-point halo, one 64-byte line per neighbour: the usual stencil exchange
        _case("halo_3d", "alltoall", "32x32x32", "moore1", "64", 4),
        # the same neighbourhood, every process publishes one block to all neighbours
        _case("gather_3d", "allgather", "32x32x32", "moore1", "64", 4),
        # 80 neighbours in four dimensions
        _case("gather_4d", "allgather", "16x16x16x16", "moore1", "64", 4),
        # five doubles per neighbour (the state of a flow solver) on a torus with odd sides, direct
        _case("doubles_3d_direct", "alltoall", "41x37x29", "moore1", "40", 8, "direct"),
        # blocks of an odd number of bytes on odd sides: packed records
        _case("odd_bytes_2d", "alltoall", "257x251", "moore2", "13", 1),
        # 242 neighbours, one 16-byte cell each
        _case("cells_5d", "alltoall", "8x8x8x8x8", "moore1", "16", 4),
        # 342 neighbours, direct: every block comes from another process
        _case("wide_3d_direct", "alltoall", "32x32x32", "moore3", "64", 4, "direct"),
        # irregular sizes from 4 to 1024 bytes, 30 arbitrary neighbours, 131072 processes
        _case("irregular_3d", "alltoallv", "64x64x32", "random30", "sizes", 1),
        # a stencil's faces, edges and corners (1024, 32 and 1 bytes) on a domain that does not wrap around
        _case("stencil_mesh_3d", "alltoallv", "32x32x32", "moore1", "stencil32", 1, mesh=True),
        # pages of 4 KB: the largest
        _case("pages_2d", "alltoall", "256x256", "moore2", "4096", 1),
        # the halo exchange for data that live in host memory
        _case("halo_3d_host", "alltoall", "32x32x32", "moore1", "64", 4, entry="host"),
    ]


MOST_PAYLOAD = 1.0e9  # bytes of a drawn case's receive buffers; the largest listed case has 6.4e9


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    while True:
        call = rng.choices(("alltoall", "allgather", "alltoallv"), (5, 3, 3))[0]
        d = rng.choices((2, 3, 4, 5), (3, 5, 2, 1))[0]
        side = _log_uniform(rng, 64, 131072) ** (1.0 / d)
        dims = [max(3, round(side * rng.uniform(0.7, 1.4))) for _ in range(d)]
        kind = rng.choice(("moore", "moore", "octant", "random"))
        if kind == "random":
            neighbours = "random%d" % rng.randint(6, 60)
        else:
            neighbours = "%s%d" % (kind, rng.randint(1, 3) if d <= 3 else 1)
        element = rng.choice((1, 4, 4, 8))
        if call == "alltoallv":
            block, element = (rng.choice(("sizes", "stencil%d" % rng.randint(4, 32))), 1) if kind == "moore" and d == 3 else ("sizes", 1)
        else:
            block = str(element * max(1, round(_log_uniform(rng, 4, 4096) / element)))
        schedule = rng.choices(("combining", "direct", "combining2"), (6, 3, 1))[0]
        case = _case("", call, "x".join(map(str, dims)), neighbours, block, element, schedule, rng.random() < 0.15,
                     "host" if rng.random() < 0.08 else "start")
        P = math.prod(dims)
        payload = P * int(_lens(case, _offsets(case)).sum())
        if 4096 <= payload <= (1.0e8 if case["entry"] == "host" else MOST_PAYLOAD):
            return case


def _dims(case):
    return tuple(int(x) for x in case["torus"].split("x"))


def _number(text, word):
    return int(text[len(word):])


def _offsets(case):
    d, text = len(_dims(case)), case["neighbours"]
    if text.startswith("moore"):
        return wl.moore(d, _number(text, "moore"))
    if text.startswith("octant"):
        return wl.positive_octant(d, _number(text, "octant"))
    if text.startswith("shells"):
        return wl.shells(d, [int(r) for r in text[len("shells"):].split("+")])
    return wl.random_offsets(wl.DEFAULT_SEED, d, _number(text, "random"), -3 if d <= 3 else -1, 3 if d <= 3 else 2)


def _lens(case, offsets):
    """Bytes of the block of every neighbour."""
    s, block = len(offsets), case["block"]
    if block == "sizes":
        return wl.random_sizes(wl.DEFAULT_SEED, s)
    if block.startswith("stencil"):
        m, d = _number(block, "stencil"), offsets.shape[1]
        return np.asarray([m ** max(0, d - int(np.abs(v).sum())) for v in offsets], dtype=np.int64)
    return np.full(s, int(block), dtype=np.int64)


class State:
    """Buffers, neighbourhood and request, as a program keeps them over its time steps."""

    comm = request = None

    def __init__(self, case, seed):
        dims, offsets = _dims(case), _offsets(case)
        P, s = math.prod(dims), len(offsets)
        lens = _lens(case, offsets)
        self.host = case["entry"] == "host"
        self.stream = torch.cuda.current_stream()
        if case["call"] == "alltoallv":
            send_stride = recv_stride = (int(lens.sum()) + 15) // 16 * 16
        else:
            recv_stride = int(lens.sum())
            send_stride = recv_stride if case["call"] == "alltoall" else int(lens[0])
        kind = "fp32" if case["element"] == 4 else "uint8"
        n = P * send_stride
        self.send = wl.payload_torch(kind, seed, 0, (n + 3) // 4 * 4, "cuda")[:n]
        self.recv = torch.zeros(P * recv_stride, dtype=torch.uint8, device="cuda")
        self.comm = iso.Iso_neighborhood_create(dims, offsets)
        if case["mesh"]:
            iso.Iso_comm_set_periodic(self.comm, [0] + [1] * (len(dims) - 2) + [0])
        if case["call"] == "alltoallv":
            displs = wl.packed_displacements(lens)
            self.request = iso.Iso_neighbor_alltoallv_init(self.send, lens, displs, iso.ISO_BYTE,
                                                           self.recv, lens, displs, iso.ISO_BYTE, self.comm)
        else:
            init = iso.Iso_neighbor_alltoall_init if case["call"] == "alltoall" else iso.Iso_neighbor_allgather_init
            count, element = int(lens[0]) // case["element"], case["element"]
            self.request = init(self.send, count, element, self.recv, count, element, self.comm)
        if case["schedule"] == "direct":
            iso.Iso_request_set_algorithm(self.request, iso.ISO_ALG_DIRECT, 1)
        elif case["schedule"] == "combining2":
            iso.Iso_request_set_algorithm(self.request, iso.ISO_ALG_COMBINING, 2)
        if self.host:
            self.host_send = torch.empty(n, dtype=torch.uint8, pin_memory=True)
            self.host_send.copy_(self.send)
            self.host_recv = torch.zeros(P * recv_stride, dtype=torch.uint8, pin_memory=True)
        result = self.host_recv if self.host else self.recv
        self.result = result.view(torch.int32) if result.numel() % 4 == 0 else result

    def __del__(self):
        if self.request is not None:
            iso.Iso_request_free(self.request)
        if self.comm is not None:
            iso.Iso_comm_free(self.comm)


def prepare(case, seed):
    return State(case, seed)


def run(state):
    """One collective: the receive buffers of all processes, whole."""
    if state.host:
        iso.Iso_Start_host(state.request, state.host_send, state.host_recv, state.stream)
        iso.Iso_wait(state.request)  # the host reads the result
    else:
        iso.Iso_Start(state.request, state.stream)
    return state.result


def work(case):
    """Every input byte read once, every delivered byte written once; no arithmetic.  (On a mesh the
    blocks that have no sender are not delivered.)"""
    dims, offsets = _dims(case), _offsets(case)
    P = math.prod(dims)
    lens = _lens(case, offsets)
    share = np.ones(len(offsets))
    if case["mesh"]:
        for j in (0, len(dims) - 1):
            share *= np.maximum(0.0, 1.0 - np.abs(offsets[:, j]) / dims[j])
    delivered = P * float((lens * share).sum())
    taken = P * float(lens[0]) if case["call"] == "allgather" else delivered
    return {"bytes": taken + delivered, "flops": 0}


def tolerance(case):
    """Bytes are moved, not computed."""
    return "exact"
