""""ce_small_ctas" below 128: calls beyond the small-message size leave the driver only where that many CTAs keep up with it, whatever they
do the result is the same."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W
from gpu_util import DevBuf, same_bits

pytestmark = pytest.mark.gpu


def _comm(R, ctas, scratch=0):
    comm = hb.Comm(R, 0)
    if scratch:
        buf = torch.empty(scratch + 256, dtype=torch.uint8, device="cuda")
        comm.set_scratch(buf.data_ptr() + (-buf.data_ptr()) % 256, scratch)
        comm._keep = buf
    comm.set_param("ce_small_bytes", 1 << 16)
    comm.set_param("ce_small_ctas", ctas)
    return comm


# flows of 2 MiB: whole ones want 64 CTAs, ones of odd length 32, ones out of phase 16
@pytest.mark.parametrize("n, shift, line", [(1 << 20, 0, 64), ((1 << 20) + 8, 0, 32), ((1 << 20) + 8, 1, 16)])
def test_uneven_exchange(n, shift, line):
    torch.cuda.set_device(0)
    R, dtype = 4, "bf16"
    st = torch.cuda.Stream()
    send = [torch.randint(-30000, 30000, (R * n,), dtype=torch.int16, device="cuda") for _ in range(R)]
    recv = [torch.zeros(R * n + shift, dtype=torch.int16, device="cuda") for _ in range(R)]
    counts, at = [n] * (R * R), [v * n for _ in range(R) for v in range(R)]
    torch.cuda.synchronize()
    for ctas in (8, 15, 16, 31, 32, 63, 64, 127, 128, 148):
        comm = _comm(R, ctas)
        comm.alltoallv(send, counts, at, [r[shift:] for r in recv], at, dtype, st)
        st.synchronize()
        assert (comm.last_stats()["n_move_launches"] > 0) == (ctas >= line), ctas
        for v in range(R):
            for u in range(R):
                assert torch.equal(recv[v][shift + u * n:shift + (u + 1) * n], send[u][v * n:(v + 1) * n])
            recv[v].zero_()
        torch.cuda.synchronize()
        assert comm.destroy() == hb.OK


@pytest.mark.parametrize("ctas", [8, 40, 148])
@pytest.mark.parametrize("n", [1 << 21, 3_000_001])
def test_ragged_all_reduce_and_message(oracle, n, ctas):
    torch.cuda.set_device(0)
    R, dtype = 4, "bf16"
    st = torch.cuda.Stream()
    xs = W.rank_inputs("normal", 3, R, n, dtype, 1e-3)
    want = oracle.ring_allreduce(xs)
    send = [DevBuf(n * 2).put(x) for x in xs]
    recv = [DevBuf(n * 2) for _ in range(R)]
    comm = _comm(R, ctas, hb.scratch_bytes_direct(R, n, dtype))
    comm.allreduce(send, recv, n, dtype, st)
    st.synchronize()
    for r in range(R):
        assert same_bits(recv[r].get(np.uint16), want[r], dtype) and recv[r].guards_intact()
    s2 = torch.cuda.Stream()
    comm.send(send[0], n, dtype, 0, 1, st)
    comm.recv(recv[1], n, dtype, 0, 1, s2)
    st.synchronize()
    s2.synchronize()
    assert (recv[1].get(np.uint16) == xs[0].view(np.uint16)).all() and recv[1].guards_intact()
    # a lone message: 4 us lost at an odd end are made good by 46 GB/s per CTA from 22 CTAs on at these lengths
    assert (comm.last_stats()["n_move_launches"] > 0) == (n == 3_000_001 and ctas > 8)
    assert comm.destroy() == hb.OK
