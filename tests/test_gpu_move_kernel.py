"""Moves between buffers that lie differently modulo 16, and groups of more copies than one batch of the plain copy kernel holds."""
import numpy as np
import pytest
import torch

from paper_2609_34334_b200 import binding as hb
from gpu_util import DevBuf

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _need_gpu():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    torch.cuda.set_device(0)
    yield
    torch.cuda.synchronize()


@pytest.mark.parametrize("ctas", [3, 40, 148])
@pytest.mark.parametrize("R,count", [(8, 1), (3, 7), (8, 33), (2, 2048 * 8 + 1), (5, 8 * 1024 * 8 + 11), (8, 70_001), (16, 4099)])
def test_ragged_blocks(R, count, ctas):
    """Odd counts: the blocks of a rank lie at every phase of 2 bytes; heads, bodies and tails of each, source against destination."""
    rng = np.random.default_rng(R * 1000 + count)
    x = rng.integers(0, 1 << 16, (R, R * count), dtype=np.uint16)
    comm = hb.Comm(R, 0)
    comm.set_path(hb.PATH_SM)
    comm.set_param("copy_ctas", ctas)
    for shift in (0, 1, 5):
        send = [DevBuf(R * count * 2, 2 * ((r * shift) % 8)).put(x[r]) for r in range(R)]
        recv = [DevBuf(R * count * 2, 2 * ((r + shift) % 8)) for r in range(R)]
        comm.alltoall(send, recv, count, "bf16")
        torch.cuda.synchronize()
        for r in range(R):
            want = np.concatenate([x[u][r * count:(r + 1) * count] for u in range(R)])
            assert (recv[r].get(np.uint16) == want).all() and recv[r].guards_intact() and (send[r].get(np.uint16) == x[r]).all(), (shift, r)
        assert comm.last_stats()["n_moves"] == R * R
        # all-gather: every block goes to R destinations of differing phases
        src = [DevBuf(count * 2, 2 * (r % 8)).put(x[r][:count]) for r in range(R)]
        for b in recv:
            b.view.fill_(0)
        comm.allgather(src, recv, count, "bf16")
        torch.cuda.synchronize()
        want = np.concatenate([x[u][:count] for u in range(R)])
        assert all((recv[r].get(np.uint16) == want).all() and recv[r].guards_intact() for r in range(R)), shift
    comm.destroy()


def test_an_all_to_all_of_eight_ranks_is_one_launch():
    R, count = 8, 4096
    send = [DevBuf(R * count * 4) for _ in range(R)]
    recv = [DevBuf(R * count * 4) for _ in range(R)]
    comm = hb.Comm(R, 0)
    comm.set_path(hb.PATH_SM)
    comm.alltoall(send, recv, count, "fp32")
    torch.cuda.synchronize()
    assert (comm.last_stats()["n_move_launches"], comm.last_stats()["n_moves"]) == (1, 64)
    comm.destroy()


@pytest.mark.parametrize("op", ["allgather", "alltoall", "allreduce"])
@pytest.mark.parametrize("count", [(1 << 20) - 8, (1 << 20) + 1, 1_100_032, 600_064, 1 << 20, 2 << 20])
def test_copies_the_driver_does_badly(op, count):
    """Copy route above the small-message size: blocks of 1 to 2 MiB that end inside a page or start off a 128-byte line run on the
    copy kernel (all-to-all; all-gathers of several ranks always) or leave their ends to it (all-reduce); whole blocks stay with the
    driver, in an all-to-all from 4 MiB on."""
    R = 8
    comm = hb.Comm(R, 0)
    n = R * count
    nb = hb.scratch_bytes_direct(R, n, "bf16")
    scratch = torch.empty(nb, dtype=torch.uint8, device="cuda")
    comm.set_scratch(scratch, nb)
    g = torch.Generator(device="cuda").manual_seed(count)
    ints = lambda k: torch.randint(-8, 9, (k,), generator=g, device="cuda").to(torch.bfloat16)     # sums of 8 are exact
    for pad in (0, 3):
        make = lambda k: torch.zeros(k + pad, dtype=torch.bfloat16, device="cuda")[pad:]
        recv = [make(n) for _ in range(R)]
        if op == "allgather":
            send = [make(count).copy_(ints(count)) for _ in range(R)]
            comm.allgather(send, recv, count, "bf16")
            want = [torch.cat(send)] * R
        else:
            send = [make(n).copy_(ints(n)) for _ in range(R)]
            if op == "alltoall":
                comm.alltoall(send, recv, count, "bf16")
                want = [torch.cat([s[r * count:(r + 1) * count] for s in send]) for r in range(R)]
            else:
                comm.allreduce(send, recv, n, "bf16")
                want = [torch.stack([s.float() for s in send]).sum(0).to(torch.bfloat16)] * R
        torch.cuda.synchronize()
        assert all(torch.equal(recv[r], want[r]) for r in range(R)), (op, count, pad)
        whole = count * 2 % 4096 == 0 and pad == 0 and (op == "allreduce" or op == "alltoall" and count >= 2 << 20)
        assert (comm.last_stats()["n_move_launches"] == 0) == whole, (op, count, pad, comm.last_stats())
    comm.destroy()


@pytest.mark.parametrize("R,mib,width,kernel", [(8, 1, 1024, True), (8, 16, 1024, True), (8, 40, 1024, False), (8, 40, 333, True), (20, 8, 1024, True)])
def test_route_of_a_user_defined_pattern(R, mib, width, kernel):
    """Copy route: short patterns, short flows and rows the driver copies badly go to the copy kernel in one launch; the rest is one
    driver copy per flow.  Uneven flows, one of them empty, displacements with gaps."""
    rng = np.random.default_rng(mib + width)
    counts = rng.integers(1, 8, (R, R)) * max(1, (mib << 20) // (2 * width * 32)) * width
    counts[2, 5] = 0
    sd = np.cumsum(counts, 1) - counts
    rd = (np.cumsum(counts, 0) - counts).T + 8 * np.arange(R)[None, :]        # [receiver, sender]
    if width % 64 == 0:
        rd = rd + 56 * np.arange(R)[None, :]                                  # gaps of whole 128-byte lines
    send = [torch.randint(-30000, 30000, (int(counts[u].sum()),), dtype=torch.int16, device="cuda") for u in range(R)]
    recv = [torch.zeros(int(counts[:, v].sum()) + 64 * R, dtype=torch.int16, device="cuda") for v in range(R)]
    comm = hb.Comm(R, 0)
    for rep in range(2):
        comm.alltoallv(send, counts.ravel(), sd.ravel(), recv, rd.ravel(), "bf16")
        torch.cuda.synchronize()
        for v in range(R):
            want = torch.zeros_like(recv[v])
            for u in range(R):
                n = int(counts[u, v])
                want[int(rd[v, u]):int(rd[v, u]) + n] = send[u][int(sd[u, v]):int(sd[u, v]) + n]
            assert torch.equal(recv[v], want), (rep, v)
            recv[v].zero_()
        st = comm.last_stats()
        assert (st["n_move_launches"], st["n_moves"], st["graph_hit"]) == (int(kernel) * -(-(R * R - 1) // 128), R * R - 1, rep), st
    comm.destroy()


@pytest.mark.parametrize("two_streams", [False, True])
@pytest.mark.parametrize("nbytes,kernel", [(2, True), (8 << 20, True), ((8 << 20) + 4096, False), ((8 << 20) + 2, True)])
def test_route_of_a_message(nbytes, kernel, two_streams):
    """Copy route: messages up to ce_small_bytes and those the driver copies badly on the kernel, the rest as driver copies; a chain of
    hops over one or several streams delivers, whichever side posts first."""
    comm = hb.Comm(4, 0)
    n = nbytes // 2
    streams = [torch.cuda.Stream() if two_streams else torch.cuda.current_stream() for _ in range(4)]
    for k in (0, 1):
        bufs = [torch.zeros(n, dtype=torch.int16, device="cuda") for _ in range(4)]
        data = torch.randint(-30000, 30000, (n,), dtype=torch.int16, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            bufs[0].copy_(data)
        for s in range(3):
            posts = [lambda: comm.send(bufs[s], n, "bf16", s, s + 1, streams[s]), lambda: comm.recv(bufs[s + 1], n, "bf16", s, s + 1, streams[s + 1])]
            for post in posts if k == 0 else reversed(posts):
                post()
        with torch.cuda.stream(streams[0]):
            bufs[0].zero_()                              # the sender's stream goes on only after its message has left
        torch.cuda.synchronize()
        assert torch.equal(bufs[3], data) and torch.equal(bufs[1], data) and int(bufs[0].abs().sum()) == 0
        assert (comm.last_stats()["n_move_launches"], comm.last_stats()["n_moves"]) == (int(kernel), 1)
    assert comm.destroy() == hb.OK
