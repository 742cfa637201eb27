"""Handshake mode switched on a communicator whose calls are already cached: every call of the mode goes through the proxy, in a burst
as alone, and after switching it off none does.  A call of a burst is otherwise launched straight into the caller's stream."""
import time

import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W
from gpu_util import same_bits

pytestmark = pytest.mark.gpu

CALLS = 40


def _wait(stream, seconds=60.0):
    t0 = time.time()
    while not stream.query():
        if time.time() - t0 > seconds:
            pytest.fail("stream still busy after %.0f s" % seconds)
        time.sleep(0.002)


# one launch, two launches (sums, then moves), a call without sums
@pytest.mark.parametrize("op, n", [("allreduce", 40_000), ("allreduce", 800_000), ("alltoall", 65_536)])
def test_every_call_of_the_mode_is_handed_over(oracle, op, n):
    torch.cuda.set_device(0)
    R, dtype = 8, "bf16"
    total = n * (R if op == "alltoall" else 1)
    xs = W.rank_inputs("normal", 17, R, total, dtype, 1e-3)
    want = oracle.ring_allreduce(xs) if op == "allreduce" else [np.concatenate([x[v * n:(v + 1) * n] for x in xs]) for v in range(R)]
    send = [torch.from_numpy(x.view(np.int16)).cuda() for x in xs]
    recv = [torch.zeros_like(s) for s in send]
    scratch = torch.empty(hb.scratch_bytes_direct(R, total, dtype) + 256, dtype=torch.uint8, device="cuda")
    comm = hb.Comm(R, 0)
    comm.set_scratch(scratch.data_ptr() + (-scratch.data_ptr()) % 256, scratch.numel() - 256)
    comm.set_path(hb.PATH_SM)
    comm.set_param("copy_ctas", 40)
    comm.set_param("watchdog_ms", 5000)
    call = getattr(comm, op)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    served = 0
    for mode in (0, 1, 0, 1):
        comm.set_param("handshake", mode)
        for r in recv:
            r.zero_()
        torch.cuda.synchronize()
        for _ in range(CALLS):
            call(send, recv, n, dtype, st)
        _wait(st)
        served += CALLS * mode
        assert comm.handshakes() == served
        for r in range(R):
            assert same_bits(recv[r].cpu().numpy().view(np.uint16), want[r], dtype), (mode, r)
    assert comm.async_error() == hb.OK and comm.destroy() == hb.OK
