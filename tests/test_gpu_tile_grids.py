"""Whole-GPU launches, a CTA per tile: moves to one and several destinations of any phase and sums, at the edges of tiles, with fewer tiles than SMs
and many more, and with nothing but byte-wise or element-wise items."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import diag as hd
from paper_2609_34334_b200 import workloads as W
from gpu_util import DevBuf, same_bits
from test_gpu_parity import run_allreduce
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [147, 148, 1024])
@pytest.mark.parametrize("ndst", [1, 2, 3, 4, 7])
def test_moves(ndst, ctas):
    torch.cuda.set_device(0)
    rng = np.random.default_rng(ndst)
    for n in (1, 15, 16, 4095, 4096, 4097, 8192 + 33, 296 * 4096 - 1, 296 * 8192 + 16, 9_000_011):
        x = rng.integers(0, 256, n, dtype=np.uint8)
        for soff, doff in ((0, 0), (3, 3), (1, 6)):
            src, dst = DevBuf(n, soff).put(x), [DevBuf(n, (doff + 5 * d) % 16) for d in range(ndst)]
            rc = hd.fanout_launch(src, dst, n, ctas)
            torch.cuda.synchronize()
            assert rc == hb.OK and all((d.get(np.uint8) == x).all() and d.guards_intact() for d in dst), (n, soff, doff)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R", [2, 3, 4, 7, 8, 9, 13, 16, 17])
def test_sums(oracle, R, dtype):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    v = 16 // e
    for n in (R * 148 * 256 * v, R * (148 * 512 * v + 1) - 1) + ((R * 300 * 512 * v + 5,) if R < 10 else ()):
        xs = W.rank_inputs("uniform", 1200 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        comm = auto_comm(R, n, dtype, hb.PATH_SM, sum_ctas=148, copy_ctas=148)
        for offs in ([0] * R, [e] * R):
            got = run_allreduce(comm, xs, dtype, offs=offs)
            assert all(same_bits(got[r], want[r], dtype) for r in range(R)), (n, offs)
        # one destination, its phase not that of the operands: element by element
        q = n // R
        send = [DevBuf(n * e, 0).put(x) for x in xs]
        recv = [DevBuf(q * e, e * (r % 3)) for r in range(R)]
        wrs = oracle.ring_reduce_scatter([x[:q * R] for x in xs])
        comm.reduce_scatter(send, recv, q, dtype)
        torch.cuda.synchronize()
        assert all(same_bits(recv[r].get(np.float32 if dtype == "fp32" else np.uint16), wrs[r], dtype) and recv[r].guards_intact() for r in range(R)), n
        comm.destroy()
