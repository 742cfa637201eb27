"""hoccl_allreduce_static on buffers of one 16-byte phase (sums read in place, one or two launches) and of several (the ring)."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W
from gpu_util import DevBuf, np_dtype, same_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R", [1, 2, 3, 6, 8, 9, 33])
def test_against_the_oracle(oracle, R, dtype):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    line = 8 * (384 << 10) // (R * e)                    # up to here the sum stores the result for every rank
    for n in (1, R - 1 or 1, 4099, line, line + 1, min(2 * line, 1_500_000) + 3):
        xs = W.rank_inputs("uniform", 700 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        for offs in ([0] * R, [e] * R, [(r % 3) * e for r in range(R)]):
            for in_place in (False, True):
                send = [DevBuf(n * e, offs[r]).put(xs[r]) for r in range(R)]
                recv = send if in_place else [DevBuf(n * e, offs[r]) for r in range(R)]
                assert hb.allreduce_static(send, recv, n, dtype, R) == hb.OK
                torch.cuda.synchronize()
                for r in range(R):
                    assert same_bits(recv[r].get(np_dtype(dtype)), want[r], dtype), (R, n, offs[:3], in_place, r)
                    assert recv[r].guards_intact() and send[r].guards_intact()
