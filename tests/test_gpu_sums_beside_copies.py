"""Copy route with whole-GPU sums in pieces: the sums that have another piece's driver copies beside them walk their tiles, the others
have a CTA per tile.  Bits of the oracle at the edges of tiles and pieces, canaries around every buffer."""
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import workloads as W
from gpu_util import DevBuf, np_dtype, same_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rs_direct", [1, 2])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("R", [2, 3, 4, 5, 6, 7, 8, 9])
def test_pieces_of_whole_gpu_sums(oracle, R, dtype, rs_direct):
    torch.cuda.set_device(0)
    e = W.elem_size(dtype)
    # ring chunks in two or three pieces of 64 KiB and more: less than a tile per CTA, a ragged last piece, phases within a line
    for chunk, pieces, off in ((3 * 65536 // e, 3, 0), (200_003, 2, 16), (410_001, 3, 4 if dtype == "fp32" else 2)):
        n = R * chunk - 5
        xs = W.rank_inputs("normal", 31 + R, R, n, dtype, 1e-3)
        want = oracle.ring_allreduce(xs)
        send = [DevBuf(n * e, off).put(x) for x in xs]
        recv = [DevBuf(n * e, off) for _ in range(R)]
        scratch = torch.empty(hb.scratch_bytes_direct(R, n, dtype) + 256, dtype=torch.uint8, device="cuda")
        comm = hb.Comm(R, 0)
        comm.set_scratch(scratch.data_ptr() + (-scratch.data_ptr()) % 256, scratch.numel() - 256)
        for key, value in (("sum_ctas", 148), ("ce_small_bytes", 0), ("ce_overlap", pieces), ("rs_direct", rs_direct)):
            comm.set_param(key, value)
        for _ in range(2):
            comm.allreduce(send, recv, n, dtype, torch.cuda.current_stream())
            torch.cuda.synchronize()
            assert comm.last_stats()["n_pieces"] == pieces
            for r in range(R):
                assert same_bits(recv[r].get(np_dtype(dtype)), want[r], dtype), (chunk, r)
                assert recv[r].guards_intact() and send[r].guards_intact()
                recv[r].view.fill_(0xA5)
        assert comm.destroy() == hb.OK
