"""Short all-reduces in one kernel without tables: every rank count it is compiled for, fewer CTAs than chunks (a CTA's warps are split between
chunks), more, and whole-GPU grids; chunks that are empty, shorter than a vector, end inside one and take several rounds."""
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W

from gpu_util import same_bits
from test_gpu_parity import run_allreduce
from test_gpu_read_in_place import auto_comm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R,ctas", [(9, 8), (10, 8), (11, 3), (12, 8), (13, 1), (14, 16), (15, 8), (16, 8), (16, 5), (16, 148), (8, 148), (5, 148), (8, 3), (3, 2), (2, 1),
                                    (24, 8)])
def test_edges(oracle, R, ctas, dtype):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    v = 16 // e
    for n in (1, R + 1, R * v, R * (33 * v + 1) - 2, R * 256 * v, R * (512 * v + 3) + 1, R * 1100 * v - 5):
        if ctas < 128 and R * n * e > ctas * (384 << 10):      # from there on a launch of moves
            continue
        xs = W.rank_inputs("uniform", 1100 + R, R, n, dtype)
        want = oracle.ring_allreduce(xs)
        comm = auto_comm(R, n, dtype, hb.PATH_SM, sum_ctas=ctas, copy_ctas=max(8, ctas))
        for in_place in (False, True):
            got = run_allreduce(comm, xs, dtype, in_place=in_place, offs=[e] * R if in_place else None)
            assert all(same_bits(got[r], want[r], dtype) for r in range(R)), (n, in_place)
        st = comm.last_stats()
        assert (st["n_moves"], st["n_sum_launches"]) == (0, 1) or R > 16, (n, st)
        comm.destroy()
