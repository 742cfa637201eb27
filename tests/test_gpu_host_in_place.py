"""hoccl_host_allreduce with the sums reading the staging buffers in place: contiguous pieces, one result copied out to every rank;
on both sides of the size from which the staged pieces are used, with the number of pieces chosen or given."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import same_bits
from test_gpu_host_allreduce import _pinned, _with_staging
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,n,dtype", [(2, 1, "fp32"), (3, 7, "bf16"), (8, 8 * 4096, "bf16"), (8, 1_000_003, "fp32"), (5, 700_001, "bf16"), (16, 300_007, "bf16"),
                                       (3, 6_000_000, "fp32"), (3, 6_000_001, "fp32")])
@pytest.mark.parametrize("pieces", [None, 2, 5])
def test_against_the_oracle(oracle, R, n, dtype, pieces):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    xs = W.rank_inputs("uniform", 900 + R, R, n, dtype)
    want = oracle.ring_allreduce(xs)
    comm = auto_comm(R, n, dtype, hb.PATH_CE, **({} if pieces is None else {"host_pieces": pieces}))
    _with_staging(comm, R, n, dtype)
    for in_place in (False, True):
        h_send = [_pinned(x) for x in xs]
        h_recv = h_send if in_place else [torch.full((n * e + 64,), 0x5A, dtype=torch.uint8).pin_memory() for _ in range(R)]
        for rep in range(2 if not in_place else 1):
            comm.host_allreduce(h_send, h_recv, n, dtype)
            torch.cuda.synchronize()
            for r in range(R):
                got = h_recv[r].numpy()
                assert same_bits(got[:n * e].view(np.float32 if dtype == "fp32" else np.uint16), want[r], dtype), (R, n, in_place, r)
                assert in_place or ((got[n * e:] == 0x5A).all() and (h_send[r].numpy() == xs[r].view(np.uint8)).all())
    st = comm.last_stats()
    assert (st["n_moves"] == 0) == (R * n * e <= 72_000_000), st
    if pieces and n > 100_000:
        assert st["n_pieces"] == pieces, st
    comm.destroy()
