"""Copy route, automatic schedule above the small-message size: all-gathers of an all-reduce whose chunks are not whole pages run on the move
kernel, in pieces beside the next piece's sum; those of whole chunks stay driver copies, spread over chains.  Bits are the oracle's."""
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import same_bits
from test_gpu_parity import run_allreduce
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu


# elements per rank, pieces, whether the move kernel carries the all-gather
@pytest.mark.parametrize("R,n,pieces,kernel", [(16, 10_000_003, 3, True), (3, 16_777_217, 2, True), (8, 5_500_001, 1, True), (5, 5_000_004, 1, True),
                                               (8, 8 << 20, 1, False), (8, 20 << 20, 4, False), (2, 10 << 20, 2, False), (4, 8 << 20, 1, False)])
def test_route_pieces_and_bits(oracle, R, n, pieces, kernel):
    torch.cuda.set_device(0)
    xs = W.rank_inputs("uniform", 1000 + R, R, n, "bf16")
    want = oracle.ring_allreduce(xs)
    comm = auto_comm(R, n, "bf16", hb.PATH_CE)
    for in_place in (False, True):
        got = run_allreduce(comm, xs, "bf16", in_place=in_place)
        assert all(same_bits(got[r], want[r], "bf16") for r in range(R)), (R, n, in_place)
        st = comm.last_stats()
        assert (st["n_pieces"], st["n_sum_launches"], st["n_move_launches"]) == (pieces, pieces, pieces if kernel else 0), st
    # what a caller chose is kept
    comm.set_param("ce_overlap", 3)
    run_allreduce(comm, xs, "bf16")
    assert comm.last_stats()["n_pieces"] == 3
    comm.destroy()
