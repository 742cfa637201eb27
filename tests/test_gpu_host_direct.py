"""hoccl_host_allreduce on pinned buffers: the sums read and store the host buffers themselves.  Bits are the oracle's at the edges of
tiles and chunks; buffers that do not permit it (pageable, different 16-byte phases, "host_pieces" set) take the copies."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import np_dtype, same_bits
from test_gpu_host_allreduce import _with_staging
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu


def _host(x, off, pinned=True):
    """The bytes of x at `off` bytes into a host buffer, guard bytes around them."""
    buf = torch.full((x.nbytes + 96,), 0x5A, dtype=torch.uint8)
    buf = buf.pin_memory() if pinned else buf
    buf[off:off + x.nbytes] = torch.from_numpy(x.view(np.uint8).copy())
    return buf, buf[off:off + x.nbytes]


def _check(bufs, offs, want, dtype):
    for (buf, view), off, w in zip(bufs, offs, want):
        assert same_bits(view.numpy().view(np_dtype(dtype)), w, dtype)
        assert (buf[:off] == 0x5A).all() and (buf[off + w.nbytes:] == 0x5A).all(), "a guard byte was written"


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R", [2, 3, 4, 5, 6, 7, 8, 9, 16])
def test_every_rank_count_and_tile_edge(oracle, R, dtype):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    v = 16 // e
    for n in (1, R * v, R * 512 * v, R * (1024 * v + 1) - 1, R * 2048 * v + 3):
        xs = W.rank_inputs("uniform", 950 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        comm = auto_comm(R, n, dtype, hb.PATH_CE)
        _with_staging(comm, R, n, dtype)
        for off in (0, e):                              # one phase for all buffers, 0 and not
            send, recv = [_host(x, off) for x in xs], [_host(np.zeros_like(x), off) for x in xs]
            for rep in range(2):
                comm.host_allreduce([s for _, s in send], [r for _, r in recv], n, dtype)
                torch.cuda.synchronize()
                _check(recv, [off] * R, want, dtype)
                _check(send, [off] * R, xs, dtype)
            st = comm.last_stats()
            assert (st["n_sum_launches"], st["n_pieces"], st["n_moves"], st["graph_hit"]) == (1, 1, 0, 0), st
            comm.host_allreduce([s for _, s in send], [s for _, s in send], n, dtype)       # in place
            torch.cuda.synchronize()
            _check(send, [off] * R, want, dtype)
        comm.destroy()


@pytest.mark.parametrize("form", ["pageable", "one_pageable", "phases", "pieces", "registered", "swapped", "captured"])
def test_which_buffers_take_the_copies(oracle, form):
    R, n, dtype = 4, 4 * 40_000 + 3, "bf16"
    torch.cuda.set_device(0)
    xs = W.rank_inputs("normal", 960, R, n, dtype, 1e-3)
    want = oracle.ring_allreduce(xs)
    comm = auto_comm(R, n, dtype, hb.PATH_CE, **({"host_pieces": 2} if form == "pieces" else {}))
    _with_staging(comm, R, n, dtype)
    offs = [2 * r for r in range(R)] if form == "phases" else [0] * R
    pinned = [form not in ("pageable", "registered") and not (form == "one_pageable" and r == 2) for r in range(R)]
    send = [_host(x, offs[r], pinned[r]) for r, x in enumerate(xs)]
    recv = [_host(np.zeros_like(x), offs[r], pinned[r]) for r, x in enumerate(xs)]
    if form == "registered":
        phase = {b.data_ptr() % 16 for b, _ in send + recv}
        assert len(phase) == 1
        assert all(torch.cuda.cudart().cudaHostRegister(b.data_ptr(), b.numel(), 0) == torch.cuda.cudart().cudaError.success for b, _ in send + recv)
    s, r = [x for _, x in send], [x for _, x in recv]
    if form == "swapped":                               # one rank's result replaces another rank's contribution
        r = s[1:] + s[:1]
        recv = send[1:] + send[:1]
    if form == "captured":
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            comm.host_allreduce(s, r, n, dtype, stream)
        graph.replay()
    else:
        comm.host_allreduce(s, r, n, dtype)
        if form != "swapped":
            comm.host_allreduce(s, r, n, dtype)
    torch.cuda.synchronize()
    _check(recv, offs, want, dtype)
    direct = form in ("registered", "swapped", "captured")
    st = comm.last_stats()
    assert (st["graph_hit"] == 0) == direct and st["n_moves"] == 0, (form, st)
    if form == "registered":
        for b, _ in send + recv:
            torch.cuda.cudart().cudaHostUnregister(b.data_ptr())
    comm.destroy()
