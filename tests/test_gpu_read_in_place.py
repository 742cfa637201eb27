"""The automatic direct schedule: sums read the contributions where they lie (no moves into an inbox), and on the SM route short
messages and whole-GPU sums store the result for every rank in the same kernel.  Bits are the oracle's; the statistics show which
form ran."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import DevBuf, np_dtype, same_bits
from test_gpu_parity import run_allreduce

pytestmark = pytest.mark.gpu


def auto_comm(R, n, dtype, path, **params):
    comm = hb.Comm(R, 0)
    comm.set_path(path)
    for k, v in params.items():
        comm.set_param(k, v)
    nb = hb.scratch_bytes_direct(R, n, dtype)
    comm._scratch_keep = DevBuf(nb + 256)
    pad = (-comm._scratch_keep.ptr) % 256
    assert hb.lib().hoccl_comm_set_scratch(comm._h, comm._scratch_keep.ptr + pad, nb) == hb.OK
    return comm


@pytest.fixture(autouse=True)
def _need_gpu():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    torch.cuda.set_device(0)
    yield
    torch.cuda.synchronize()


SM_BUDGET = dict(path=hb.PATH_SM, sum_ctas=8, copy_ctas=40)
SM_WHOLE = dict(path=hb.PATH_SM, sum_ctas=148, copy_ctas=148)
DRIVER = dict(path=hb.PATH_CE, ce_small_bytes=0)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R", [2, 3, 4, 5, 6, 7, 8, 9, 16])
def test_every_rank_count_and_tile_edge(oracle, R, dtype):
    v = 16 // W.elem_size(dtype)                        # elements of one vector; a tile is 512 to 2048 vectors of a ring chunk
    for chunk in (1, v, 512 * v, 1024 * v + 1, 2 * 2048 * v - 1, 13 * 512 * v + 3):
        n = R * chunk - (chunk > 2)                     # the last chunk one element short
        xs = W.rank_inputs("uniform", 500 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        for cfg in (dict(path=hb.PATH_CE), DRIVER, SM_BUDGET, SM_WHOLE, dict(SM_BUDGET, use_graph=0)):
            comm = auto_comm(R, n, dtype, **cfg)
            for in_place in (False, True):
                offs = [W.elem_size(dtype)] * R if in_place else None       # one phase for all buffers, not 0
                got = run_allreduce(comm, xs, dtype, in_place=in_place, offs=offs)
                assert all(same_bits(got[r], want[r], dtype) for r in range(R)), (R, n, cfg, in_place)
            st = comm.last_stats()
            filled = -(-n // -(-n // R))                # ring chunks that are not empty
            assert st["n_sum_launches"] >= 1 and st["n_moves"] in (0, filled * (R - 1)), (cfg, st)
            comm.destroy()


def test_which_form_runs(oracle):
    R, dtype = 8, "bf16"
    small, mid = 8 * 1000, 8 * 200_000                  # 16 KiB and 3.2 MB per rank; the line for 8 CTAs lies at 3 MiB / R
    for n, cfg, moves, launches in ((small, dict(path=hb.PATH_CE), 0, 0), (mid, dict(path=hb.PATH_CE), 56, 1), (mid, DRIVER, 56, 0),
                                    (small, SM_BUDGET, 0, 0), (mid, SM_BUDGET, 56, 1), (mid, SM_WHOLE, 0, 0)):
        comm = auto_comm(R, n, dtype, **cfg)
        xs = W.rank_inputs("normal", 510, R, n, dtype, 1e-3)
        want = oracle.ring_allreduce(xs)
        got = run_allreduce(comm, xs, dtype)
        assert all(same_bits(got[r], want[r], dtype) for r in range(R))
        st = comm.last_stats()
        assert (st["n_moves"], st["n_move_launches"], st["n_sum_launches"]) == (moves, launches, 1), (n, cfg, st)
        # the reduce-scatter alone needs no moves at all
        send = [DevBuf(n * 2).put(x) for x in xs]
        recv = [DevBuf(n // R * 2) for _ in range(R)]
        comm.reduce_scatter(send, recv, n // R, dtype)
        torch.cuda.synchronize()
        wrs = oracle.ring_reduce_scatter(xs)
        assert all(same_bits(recv[r].get(np_dtype(dtype)), wrs[r], dtype) and recv[r].guards_intact() for r in range(R))
        st = comm.last_stats()
        assert (st["n_moves"], st["n_sum_launches"]) == (0, 1), (cfg, st)
        # contributions that do not share their 16-byte phase are staged, and so is what "rs_direct" = 1 asks for
        got = run_allreduce(comm, xs, dtype, offs=[(r % 4) * 2 for r in range(R)])
        assert all(same_bits(got[r], want[r], dtype) for r in range(R)) and comm.last_stats()["n_moves"] == 112
        comm.set_param("rs_direct", 1)
        got = run_allreduce(comm, xs, dtype)
        assert all(same_bits(got[r], want[r], dtype) for r in range(R)) and comm.last_stats()["n_moves"] == 112
        comm.destroy()


@pytest.mark.parametrize("cfg", [dict(path=hb.PATH_CE), SM_BUDGET, dict(path=hb.PATH_CE, sum_ctas=148)])
def test_overlapped_pieces(oracle, cfg):
    """Chunks large enough to be cut: the all-gather's moves of one piece run beside the next piece's sum, in place too."""
    for R, chunk_mib, dtype in ((2, 9, "fp32"), (8, 4, "bf16")):
        n = R * (chunk_mib << 20) // W.elem_size(dtype) + 5
        xs = W.rank_inputs("uniform", 520 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        comm = auto_comm(R, n, dtype, **cfg)
        for in_place in (False, True, True):
            got = run_allreduce(comm, xs, dtype, in_place=in_place)
            assert all(same_bits(got[r], want[r], dtype) for r in range(R)), (R, cfg, in_place)
        st = comm.last_stats()
        assert st["n_sum_launches"] == st["n_pieces"] and (st["n_pieces"] > 1 or cfg.get("sum_ctas") == 148), st
        comm.destroy()


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("ag_direct", [0, 1])
@pytest.mark.parametrize("R", [6, 8])
def test_ragged_chunks_of_driver_copies(oracle, R, ag_direct, use_graph):
    """Chunks from 1 MiB on that are not whole pages on 128-byte lines: a direct all-gather leaves the copies' ends to the copy kernel, a
    ring forwards whole copies.  Buffers with one 16-byte phase on one and on several 128-byte phases, whole and in pieces."""
    dtype, n = "bf16", R * 600_003 - 2
    xs = W.rank_inputs("uniform", 530 + R, R, n, dtype)
    want = oracle.ring_allreduce(xs)
    for params in (dict(), dict(piece_bytes=400 << 10, max_pieces=8)):
        comm = auto_comm(R, n, dtype, hb.PATH_CE, ce_small_bytes=4096, ag_direct=ag_direct, use_graph=use_graph, **params)
        for offs in ([0] * R, [16 * (r % 8) for r in range(R)]):
            for in_place in (False, True):
                for rep in range(3):
                    got = run_allreduce(comm, xs, dtype, in_place=in_place, offs=offs)
                    assert all(same_bits(got[r], want[r], dtype) for r in range(R)), (R, params, offs, in_place, rep)
        assert (comm.last_stats()["n_move_launches"] > 0) == (ag_direct == 1 and not params), comm.last_stats()
        comm.destroy()


def test_changed_setting_is_not_served_from_the_graph_of_the_old_one(oracle):
    R, dtype, n = 8, "bf16", 8 * 600_003
    xs = W.rank_inputs("uniform", 540, R, n, dtype)
    want = oracle.ring_allreduce(xs)
    comm = auto_comm(R, n, dtype, hb.PATH_CE)
    send, recv = ([DevBuf(n * 2).put(x) for x in xs] for _ in range(2))
    for small, launches, hit in ((8 << 20, 1, 0), (8 << 20, 1, 1), (0, 0, 0), (0, 0, 1), (4 << 20, 1, 1)):
        comm.set_param("ce_small_bytes", small)
        comm.allreduce(send, recv, n, dtype)
        torch.cuda.synchronize()
        assert all(same_bits(recv[r].get(np_dtype(dtype)), want[r], dtype) for r in range(R))
        st = comm.last_stats()
        assert (st["n_move_launches"], st["graph_hit"]) == (launches, hit), (small, st)
    comm.destroy()
