"""Calls in a burst, where short chains of kernels go out as launches with programmatic serialization instead of graphs: every call reads
what the call (or the caller's kernel) in front of it has written, every kernel behind it sees its result.  Bits are the oracle's."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import same_bits
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu
TORCH = {"fp32": torch.float32, "bf16": torch.bfloat16}


def _tensor(x, dtype):
    return torch.from_numpy(x.view(np.uint8).copy()).cuda().view(TORCH[dtype])


def _numpy(t, dtype):
    return t.cpu().view(torch.uint8).numpy().view(np.float32 if dtype == "fp32" else np.uint16)


def _ahead():
    torch.cuda._sleep(400_000)      # the host runs ahead, so that the calls below queue up behind each other


# elements per rank; which kernels: sums that store for every rank (with and without tables), pipelined sums + moves, whole-GPU sums
@pytest.mark.parametrize("R,n,cfg", [(8, 131_072, dict(path=hb.PATH_CE)), (8, 524_291, dict(path=hb.PATH_CE)), (4, 1_000_003, dict(path=hb.PATH_CE)),
                                     (16, 65_536, dict(path=hb.PATH_CE)), (12, 400_000, dict(path=hb.PATH_CE)),
                                     (8, 524_288, dict(path=hb.PATH_SM, sum_ctas=148, copy_ctas=148)),
                                     (3, 300_001, dict(path=hb.PATH_SM, sum_ctas=8, copy_ctas=40)), (2, 262_144, dict(path=hb.PATH_SM, sum_ctas=8, copy_ctas=8))])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_all_reduces_in_a_burst(oracle, R, n, cfg, dtype):
    torch.cuda.set_device(0)
    xs = W.rank_inputs("normal", 970 + R, R, n, dtype, 1e-3)
    want = [x.copy() for x in xs]
    for _ in range(4):
        want = oracle.ring_allreduce(want)
    comm = auto_comm(R, n, dtype, **cfg)
    bufs, first = [_tensor(x, dtype) for x in xs], [_tensor(x, dtype) for x in xs]
    for stream in (None, torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            comm.allreduce(bufs, bufs, n, dtype, stream)                        # laid out
            for rep in range(3):
                _ahead()
                for b, f in zip(bufs, first):
                    b.copy_(f)                                                  # the caller's kernels in front
                for _ in range(4):
                    comm.allreduce(bufs, bufs, n, dtype, stream)
                after = [b.clone() for b in bufs]                               # and behind
                for b in bufs:
                    b.zero_()
                torch.cuda.synchronize()
                assert all(same_bits(_numpy(after[r], dtype), want[r], dtype) for r in range(R)), (R, n, rep)
    comm.destroy()


@pytest.mark.parametrize("R,n", [(8, 65_536), (8, 65_537), (12, 20_000), (16, 30_000)])     # 16 ranks: two launches of moves
def test_moves_and_reduce_scatters_in_a_burst(oracle, R, n):
    torch.cuda.set_device(0)
    dtype = "bf16"
    xs = W.rank_inputs("normal", 980 + R, R, n * R, dtype, 1e-3)
    comm = auto_comm(R, n * R, dtype, hb.PATH_CE)
    a, b = [_tensor(x, dtype) for x in xs], [_tensor(x, dtype) for x in xs]
    one = [torch.zeros(n, dtype=torch.bfloat16, device="cuda") for _ in range(R)]
    counts, sd = [n] * (R * R), [v * n for _ in range(R) for v in range(R)]
    want = oracle.ring_allreduce(xs)
    for rep in range(3):
        _ahead()
        for _ in range(2):          # two exchanges of blocks bring every block back
            comm.alltoall(a, b, n, dtype)
            comm.alltoallv(b, counts, sd, a, sd, dtype)
        for r in range(R):
            b[r].zero_()
        comm.reduce_scatter(a, one, n, dtype)
        comm.allgather(one, b, n, dtype)
        after = [t.clone() for t in b]
        torch.cuda.synchronize()
        assert all(same_bits(_numpy(a[r], dtype), xs[r], dtype) for r in range(R)), rep
        assert all(same_bits(_numpy(after[r], dtype), want[r], dtype) for r in range(R)), rep
    comm.destroy()


@pytest.mark.parametrize("R,n", [(6, 500_009), (8, 4_096), (3, 200_000)])
def test_static_all_reduces_in_a_burst(oracle, R, n):
    torch.cuda.set_device(0)
    xs = W.rank_inputs("normal", 990 + R, R, n, "fp32", 1e-3)
    want = oracle.ring_allreduce(oracle.ring_allreduce(xs))
    first = [_tensor(x, "fp32") for x in xs]
    bufs = [t.clone() for t in first]
    for rep in range(3):
        _ahead()
        for b, f in zip(bufs, first):
            b.copy_(f)
        for _ in range(2):
            assert hb.allreduce_static(bufs, bufs, n, "fp32", R) == hb.OK
        after = [b.clone() for b in bufs]
        torch.cuda.synchronize()
        assert all(same_bits(_numpy(after[r], "fp32"), want[r], "fp32") for r in range(R)), rep
