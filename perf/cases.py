"""What the speed of this library is judged by: calls as a training or serving job makes them, from a few KiB to hundreds of MiB.

A case is one step of such a job through the public binding: a collective (or the pair reduce-scatter + all-gather), a user-defined
exchange, a wave of send/recv messages, the host-buffer all-reduce or the all-reduce that needs no scratch.  The communicator keeps
its default settings (copy route, 8 CTAs for sums, small messages on the copy kernel) unless the case names the SM path and its
budgets, as the benchmark's comparison rows do.  The scratch is what hoccl_scratch_bytes_direct asks for.

Every result is fixed bit for bit: moves copy bytes, and sums are taken in one documented order with one documented rounding.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2609_34334_b200 import binding as hb

KIB, MIB = 1 << 10, 1 << 20
DTYPES = {"fp32": (torch.float32, 4), "bf16": (torch.bfloat16, 2)}

# path, CTAs for sums, CTAs for copies; "default" leaves the communicator as it is created
ROUTES = {"default": None, "sm_whole": (148, 148), "sm_budget": (8, 40)}


def listed():
    """`count` follows the call's own convention: all-reduce forms give the elements of one rank's vector, all-gather and
    all-to-all the elements of one block, the exchange the tokens of one rank, the wave the elements of one message."""
    return [
        # a scalar-sized reduction (loss, gradient norm, router statistics): nothing but latency
        dict(name="allreduce_4k", op="allreduce", R=8, count=2048, dtype="bf16", route="default"),
        # the small configuration: 4 ranks, 4 MiB of fp32
        dict(name="allreduce_4m_fp32_r4", op="allreduce", R=4, count=1_048_576, dtype="fp32", route="default"),
        # one 40 MiB bucket of a gradient stream, the benchmark's step
        dict(name="allreduce_40m", op="allreduce", R=8, count=20_971_520, dtype="bf16", route="default"),
        # a sharded optimizer's bucket: reduce-scatter the gradients, all-gather the weights
        dict(name="rs_ag_25m", op="rs_ag", R=8, count=13_107_200, dtype="bf16", route="default"),
        # fp32 gradients when nothing else runs: the whole GPU for copies and sums
        dict(name="allreduce_64m_fp32_sm_whole", op="allreduce", R=8, count=16_777_216, dtype="fp32", route="sm_whole"),
        # a large message beside compute: 8 CTAs for sums, 40 for copies
        dict(name="allreduce_256m_sm_budget", op="allreduce", R=8, count=134_217_728, dtype="bf16", route="sm_budget"),
        # gathering a parameter shard whose length is not a multiple of anything
        dict(name="allgather_ragged", op="allgather", R=8, count=250_007, dtype="bf16", route="default", in_place=False),
        # sequence-parallel attention: equal blocks between all ranks, 16 MiB per rank
        dict(name="alltoall_16m", op="alltoall", R=8, count=1_048_576, dtype="bf16", route="default"),
        # expert-parallel dispatch: 4096 tokens a rank of width 4096, uneven by popularity
        dict(name="alltoallv_experts", op="alltoallv", R=8, count=4096, width=4096, skew=1, dtype="bf16", route="default"),
        # pipeline parallelism: 4 microbatches of [4, 2048, 4096] activations through 4 stages, a stream for each stage
        dict(name="wave_64m", op="wave", R=4, microbatches=4, count=33_554_432, dtype="bf16", route="default"),
        # a bucket that lives in pinned host memory (offloaded gradients)
        dict(name="host_allreduce_25m", op="host_allreduce", R=8, count=13_107_200, dtype="bf16", route="default"),
        # the all-reduce for callers that may not allocate, on an odd length and a rank count that is no power of two
        dict(name="static_ragged_fp32_r6", op="static", R=6, count=500_009, dtype="fp32", route="default"),
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _count(rng: random.Random, nbytes: float, e: int) -> int:
    """About `nbytes` bytes as a number of elements: mostly round, as models' shapes are, every third one odd."""
    n = max(1, int(nbytes / e))
    if rng.random() < 1 / 3:
        return n | 1
    return max(64, n // 64 * 64)


def draw(rng: random.Random):
    op = rng.choice(["allreduce", "allreduce", "allreduce", "rs_ag", "allgather", "allgather", "alltoall", "alltoallv", "wave", "host_allreduce",
                     "static"])
    dtype = rng.choice(["bf16", "bf16", "fp32"])
    e = DTYPES[dtype][1]
    R = rng.choice([2, 4, 8, 8, 8, 3, 5, 6, 7, 16])
    route = rng.choice(["default", "default", "default", "sm_whole", "sm_budget"])
    case = dict(op=op, R=R, dtype=dtype, route=route)
    # bytes of one rank's whole vector; more ranks than 8 hold shorter ones, so that the total stays within the listed largest
    top = 256 * MIB * min(1.0, 8 / R)
    if op in ("allreduce", "rs_ag"):
        case["count"] = _count(rng, _log_uniform(rng, 4 * KIB, top), e)
        if op == "rs_ag":
            case["count"] = (case["count"] + R - 1) // R * R
    elif op in ("allgather", "alltoall"):
        case["count"] = _count(rng, _log_uniform(rng, 4 * KIB, top) / R, e)
        if op == "allgather":
            case["in_place"] = rng.random() < 0.5
    elif op == "alltoallv":
        case["width"] = rng.choice([1024, 2048, 4096, 2880, 333])
        case["count"] = max(R, int(_log_uniform(rng, 64 * KIB, top / 2) / (case["width"] * e)))
        case["skew"] = rng.randrange(1, 1 << 20)
    elif op == "wave":
        case["R"] = R = min(R, 8)
        case["microbatches"] = rng.randrange(1, 16 // R + 1)
        case["count"] = _count(rng, _log_uniform(rng, 4 * KIB, 64 * MIB), e)
    elif op == "host_allreduce":
        case["route"] = "default"
        case["count"] = _count(rng, _log_uniform(rng, 64 * KIB, 25 * MIB * min(1.0, 8 / R)), e)
    else:   # the fixed scratch array holds two padded ring chunks per rank: up to a little under 16 MiB per rank
        case["route"] = "default"
        case["count"] = _count(rng, _log_uniform(rng, 4 * KIB, 15 * MIB), e)
    return case


def _exchange(case):
    """Counts and displacements (in elements, R x R) of an expert-parallel dispatch: every rank's tokens go to the ranks by a
    log-normal popularity that the ranks share, with some noise of their own."""
    R, width = case["R"], case["width"]
    rng = random.Random(case["skew"])
    popular = [rng.gauss(0.0, 0.8) for _ in range(R)]
    counts = []
    for _ in range(R):
        w = [math.exp(p + rng.gauss(0.0, 0.3)) for p in popular]
        row = [int(case["count"] * x / sum(w)) for x in w]
        row[max(range(R), key=lambda v: w[v])] += case["count"] - sum(row)
        counts += [n * width for n in row]
    sdispls = [sum(counts[u * R:u * R + v]) for u in range(R) for v in range(R)]
    rdispls = [sum(counts[a * R + v] for a in range(u)) for v in range(R) for u in range(R)]
    received = [sum(counts[u * R + v] for u in range(R)) for v in range(R)]
    return counts, sdispls, rdispls, received


def _comm(case, elements: int):
    """A communicator as a program sets it up once: scratch for vectors of `elements` elements, the route's settings."""
    c = hb.Comm(case["R"], torch.cuda.current_device())
    nbytes = hb.scratch_bytes_direct(case["R"], elements, case["dtype"])
    if nbytes:
        c.set_scratch(torch.empty(nbytes, dtype=torch.uint8, device="cuda"), nbytes)
    if ROUTES[case["route"]]:
        c.set_path(hb.PATH_SM)
        c.set_param("sum_ctas", ROUTES[case["route"]][0])
        c.set_param("copy_ctas", ROUTES[case["route"]][1])
    return c


def prepare(case, seed: int):
    op, R, n = case["op"], case["R"], case["count"]
    dt = DTYPES[case["dtype"]][0]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def data(elements, scale=1e-3):   # gradients, weights and activations: centred, of one scale
        return torch.empty(elements, dtype=dt, device="cuda").normal_(0.0, scale, generator=g)

    def room(elements):
        return torch.zeros(elements, dtype=dt, device="cuda")

    s = dict(case=case)
    if op == "allreduce":
        s.update(comm=_comm(case, n), send=[data(n) for _ in range(R)], recv=[room(n) for _ in range(R)])
    elif op == "rs_ag":
        shard = n // R
        s.update(comm=_comm(case, n), shard=shard, send=[data(n) for _ in range(R)], recv=[room(n) for _ in range(R)])
        s["own"] = [s["recv"][r][r * shard:(r + 1) * shard] for r in range(R)]
    elif op == "allgather":
        s.update(comm=_comm(case, n * R), recv=[room(n * R) for _ in range(R)])
        s["send"] = [data(n) for _ in range(R)]
        if case["in_place"]:
            for r in range(R):
                s["recv"][r][r * n:(r + 1) * n].copy_(s["send"][r])
                s["send"][r] = s["recv"][r][r * n:(r + 1) * n]
    elif op == "alltoall":
        s.update(comm=_comm(case, n * R), send=[data(n * R, 1.0) for _ in range(R)], recv=[room(n * R) for _ in range(R)])
    elif op == "alltoallv":
        counts, sdispls, rdispls, received = _exchange(case)
        s.update(comm=_comm(case, R), counts=counts, sdispls=sdispls, rdispls=rdispls)
        s.update(send=[data(n * case["width"], 1.0) for _ in range(R)], recv=[room(max(1, k)) for k in received])
    elif op == "wave":
        m = case["microbatches"]
        s.update(comm=_comm(case, R), streams=[torch.cuda.Stream() for _ in range(R)])
        s["act"] = [[data(n, 1.0) if stage == 0 else room(n) for _ in range(m)] for stage in range(R)]
    elif op == "host_allreduce":
        e = DTYPES[case["dtype"]][1]
        s.update(comm=_comm(case, n), send=[], recv=[])
        staging = torch.empty(2 * R * ((n * e + 255) // 256 * 256), dtype=torch.uint8, device="cuda")
        s["comm"].set_staging(staging)
        for _ in range(R):
            s["send"].append(torch.empty(n, dtype=dt, pin_memory=True).copy_(data(n)))
            s["recv"].append(torch.zeros(n, dtype=dt, pin_memory=True))
    else:
        s.update(send=[data(n) for _ in range(R)], recv=[room(n) for _ in range(R)])
    return s


def run(s):
    case = s["case"]
    op, n, dtype = case["op"], case["count"], case["dtype"]
    if op == "allreduce":
        s["comm"].allreduce(s["send"], s["recv"], n, dtype)
    elif op == "rs_ag":
        s["comm"].reduce_scatter(s["send"], s["own"], s["shard"], dtype)
        s["comm"].allgather(s["own"], s["recv"], s["shard"], dtype)
    elif op == "allgather":
        s["comm"].allgather(s["send"], s["recv"], n, dtype)
    elif op == "alltoall":
        s["comm"].alltoall(s["send"], s["recv"], n, dtype)
    elif op == "alltoallv":
        s["comm"].alltoallv(s["send"], s["counts"], s["sdispls"], s["recv"], s["rdispls"], dtype)
    elif op == "wave":
        comm, act, streams = s["comm"], s["act"], s["streams"]
        for m in range(case["microbatches"]):
            for stage in range(case["R"] - 1):
                comm.send(act[stage][m], n, dtype, stage, stage + 1, streams[stage])
                comm.recv(act[stage + 1][m], n, dtype, stage, stage + 1, streams[stage + 1])
        return act[1:]
    elif op == "host_allreduce":
        s["comm"].host_allreduce(s["send"], s["recv"], n, dtype)
    elif hb.allreduce_static(s["send"], s["recv"], n, dtype, case["R"]) != hb.OK:
        raise RuntimeError("hoccl_allreduce_static failed")
    return s["recv"]


def work(case):
    """Each rank's input read once, each rank's output written once; one add for every contribution but the first."""
    op, R, n = case["op"], case["R"], case["count"]
    e = DTYPES[case["dtype"]][1]
    if op in ("allreduce", "static", "host_allreduce", "rs_ag"):
        return {"bytes": 2 * R * n * e, "flops": (R - 1) * n}
    if op == "allgather":   # in place the own block is already there
        return {"bytes": R * n * e + R * (R - 1 if case["in_place"] else R) * n * e, "flops": 0}
    if op == "alltoall":
        return {"bytes": 2 * R * R * n * e, "flops": 0}
    if op == "alltoallv":
        return {"bytes": 2 * R * n * case["width"] * e, "flops": 0}
    return {"bytes": 2 * (R - 1) * case["microbatches"] * n * e, "flops": 0}


def tolerance(case):
    return "exact"
