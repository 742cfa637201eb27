"""What a call would run, over addresses that need not exist (hoccl_layout_*, host only): whatever the settings and however the
buffers lie, two accesses to the same byte, one of them a write, are ordered by dependencies; every byte of the result is written;
nothing outside the call's buffers is touched."""
import numpy as np
import pytest
from hypothesis import HealthCheck, given, settings, strategies as st

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import diag as hd
from paper_2609_34334_b200 import workloads as W

ALLREDUCE, REDUCE_SCATTER, ALLGATHER, ALLTOALL = hd.PLAN_ALLREDUCE, hd.PLAN_REDUCE_SCATTER, hd.PLAN_ALLGATHER, hd.PLAN_ALLTOALL
ROOM = 1 << 36       # every buffer has this much address space to itself


def lay_out(kind, R, count, dtype, in_place=False, offs=None, **params):
    """The layout, and [first, last) of every send, receive and scratch region."""
    e = W.elem_size(dtype)
    ssize = count * e * (R if kind in (REDUCE_SCATTER, ALLTOALL) else 1)
    rsize = count * e * (R if kind in (ALLGATHER, ALLTOALL) else 1)
    offs = offs or [0] * R
    send = [(1 + r) * ROOM + offs[r] for r in range(R)]
    recv = [(101 + r) * ROOM + offs[-1 - r] for r in range(R)]
    if in_place:
        recv = send if kind == ALLREDUCE else [send[r] + r * count * e for r in range(R)] if kind == REDUCE_SCATTER else recv
        send = [recv[r] + r * count * e for r in range(R)] if kind == ALLGATHER else send
    n = count if kind == ALLREDUCE else count * R
    scratch = (300 * ROOM, hb.scratch_bytes_direct(R, n, dtype))
    lay = hd.Layout(kind, R, send, recv, count, dtype, scratch=scratch if scratch[1] else None, **params)
    return lay, [(p, p + ssize) for p in send], [(p, p + rsize) for p in recv], (scratch[0], scratch[0] + scratch[1])


def check(lay, send, recv, scratch, whole_recv):
    before = []                                          # groups that are done when group g starts, as a bit set
    for g, deps in enumerate(lay.deps):
        assert all(0 <= d < g for d in deps)
        before.append(0)
        for d in deps:
            before[g] |= before[d] | 1 << d
    acc = [a for a in lay.accesses if a.bytes]
    lo = np.array([a.addr for a in acc], dtype=np.uint64)
    hi = lo + np.array([a.bytes for a in acc], dtype=np.uint64)
    readable, writable = send + recv + [scratch], recv + [scratch]
    for k, a in enumerate(acc):
        assert any(f <= a.addr and a.addr + a.bytes <= l for f, l in (writable if a.write else readable)), (a.addr, a.bytes)
        if not a.write:
            continue
        for j in np.nonzero((lo < hi[k]) & (hi > lo[k]))[0]:
            b = acc[j]
            if (b.group, b.segment) == (a.group, a.segment):
                assert b.addr == a.addr and (j == k or not b.write)        # an element-wise sum may write what it reads, in place
            else:
                assert a.group != b.group, "two segments of one group meet"
                first, second = sorted((a.group, b.group))
                assert before[second] >> first & 1, "groups %d and %d (ends of copies: %d, %d) are not ordered" % (a.group, b.group, a.edges, b.edges)
    for first, last in (recv if whole_recv else []):
        at = first
        for f, l in sorted((a.addr, a.addr + a.bytes) for a in acc if a.write and first <= a.addr < last):
            assert f <= at
            at = max(at, l)
        assert at == last


@pytest.mark.parametrize("pieces", [None, 3])
@pytest.mark.parametrize("ag_direct", [0, 1, 2])
@pytest.mark.parametrize("R", [2, 3, 6, 8])
def test_ends_of_trimmed_copies(R, ag_direct, pieces):
    """Chunks of 1 MiB and more that are not whole pages on 128-byte lines: the copies of the all-gather leave their ends to the copy
    kernel.  In the ring form a step forwards what the step before it wrote."""
    for chunk in ((1 << 20) + 8, (65 << 20) + 6, 3 << 20):                   # bytes; beyond 64 MiB the automatic all-gather is the ring
        for offs in ([0] * R, [32] * R, [16 * (r % 8) for r in range(R)]):    # one 16-byte phase, with one and with several 128-byte phases
            for in_place in (False, True):
                params = dict(ag_direct=ag_direct, ce_small_bytes=1 << 20, max_pieces=8)
                if pieces:
                    params["piece_bytes"] = chunk // pieces + 1
                lay, send, recv, scratch = lay_out(ALLREDUCE, R, R * chunk // 2 - 3, "bf16", in_place, offs, **params)
                check(lay, send, recv, scratch, not in_place)
                if ag_direct == 0 and R > 2 and chunk != 3 << 20:
                    assert any(not a.edges and a.kind == hd.OP_MOVE and a.bytes % 4096 for a in lay.accesses)


case = st.fixed_dictionaries({
    "kind": st.sampled_from([ALLREDUCE, ALLREDUCE, REDUCE_SCATTER, ALLGATHER, ALLTOALL]),
    "R": st.integers(1, 10),
    "count": st.one_of(st.integers(1, 300), st.integers(1000, 400_000), st.integers(400_000, 40_000_000)),
    "dtype": st.sampled_from(["fp32", "bf16"]),
    "in_place": st.booleans(),
    "path": st.sampled_from([hb.PATH_CE, hb.PATH_CE, hb.PATH_SM, hb.PATH_CE_HOST]),
    "common": st.sampled_from([None, 0, 0, 1, 5, 32]),                       # one offset for all buffers, or one each
    "offs": st.lists(st.integers(0, 70), min_size=10, max_size=10),
    "params": st.fixed_dictionaries({
        "ag_direct": st.integers(0, 2), "rs_direct": st.integers(0, 2), "ce_small_bytes": st.sampled_from([0, 65536, 8 << 20]),
        "sum_ctas": st.sampled_from([1, 8, 148]), "copy_ctas": st.sampled_from([8, 40, 148]), "use_graph": st.integers(0, 1),
        "ce_overlap": st.sampled_from([-1, -1, 0, 3]), "piece_grade": st.integers(-1, 1), "max_pieces": st.integers(1, 9)},
        optional={"piece_bytes": st.sampled_from([1024, 1 << 16, 1 << 20]), "forward": st.just(1), "fused": st.just(1), "roles": st.just(1)}),
})


@settings(max_examples=300, deadline=None, derandomize=True, suppress_health_check=list(HealthCheck))
@given(c=case)
def test_random_calls(c):
    e = W.elem_size(c["dtype"])
    count = c["count"] if c["kind"] == ALLREDUCE else -(-c["count"] // c["R"])
    offs = [(o if c["common"] is None else c["common"]) * e for o in c["offs"][:c["R"]]]
    in_place = c["in_place"] and c["kind"] != ALLTOALL
    try:
        lay, send, recv, scratch = lay_out(c["kind"], c["R"], count, c["dtype"], in_place, offs, path=c["path"], **c["params"])
    except hb.HocclError as err:
        assert err.code == hb.ERR_UNSUPPORTED, c                             # settings that do not fit together
        return
    check(lay, send, recv, scratch, not in_place)


def _steps(lay):
    return lay.deps, [tuple(getattr(a, f) for f, _ in a._fields_) for a in lay.accesses]


def test_signature_of_trimmed_copies():
    """An all-reduce above the small-message size, before and after "ce_small_bytes" = 0: without and with whole driver copies, so not
    the same graph."""
    a, b = (lay_out(ALLREDUCE, 8, 8 * 600_003, "bf16", **params)[0] for params in ({}, {"ce_small_bytes": 0}))
    assert any(x.edges for x in a.accesses) and not any(x.edges for x in b.accesses) and a.signature != b.signature


@settings(max_examples=300, deadline=None, derandomize=True, suppress_health_check=list(HealthCheck))
@given(c=case, name=st.sampled_from(["ag_direct", "rs_direct", "ce_small_bytes", "sum_ctas", "copy_ctas", "ce_overlap", "piece_grade", "max_pieces",
                                     "piece_bytes", "path"]), k=st.integers(0, 3))
def test_one_setting_changed(c, name, k):
    """Calls that share a signature replay one graph, so they have to share the layout too."""
    values = {"ag_direct": [0, 1, 2], "rs_direct": [0, 1, 2], "ce_small_bytes": [0, 1000, 1 << 30], "sum_ctas": [4, 100, 148], "copy_ctas": [4, 100, 148],
              "ce_overlap": [-1, 0, 2], "piece_grade": [-1, 0, 1], "max_pieces": [1, 2, 9], "piece_bytes": [1 << 14, 1 << 18, 1 << 22],
              "path": [hb.PATH_CE, hb.PATH_SM, hb.PATH_CE_HOST]}[name]
    count = c["count"] if c["kind"] == ALLREDUCE else -(-c["count"] // c["R"])
    offs = [(o if c["common"] is None else c["common"]) * W.elem_size(c["dtype"]) for o in c["offs"][:c["R"]]]
    first = dict(c["params"], path=c["path"], use_graph=1)
    try:
        one, two = (lay_out(c["kind"], c["R"], count, c["dtype"], c["in_place"] and c["kind"] != ALLTOALL, offs, **params)[0]
                    for params in (first, dict(first, **{name: values[k % 3]})))
    except hb.HocclError as err:
        assert err.code == hb.ERR_UNSUPPORTED, c
        return
    assert one.signature != two.signature or _steps(one) == _steps(two), (c, name)


@pytest.mark.parametrize("kind", [ALLREDUCE, REDUCE_SCATTER, ALLGATHER, ALLTOALL])
def test_signature_of_handshake_mode(kind):
    """A call of handshake mode never shares its entry with one outside it: that entry would launch past the proxy in a burst, and its
    graph need not be on the device yet when the proxy replays it behind a parked stream."""
    a, b = (lay_out(kind, 8, 4096, "bf16", path=hb.PATH_SM, handshake=mode)[0] for mode in (0, 1))
    assert _steps(a) == _steps(b) and a.signature != b.signature


@pytest.mark.parametrize("sum_ctas", [147, 148, 296])
@pytest.mark.parametrize("R", [2, 5, 8, 9, 16])
@pytest.mark.parametrize("rs_direct", [1, 2])
def test_whole_gpu_sums_leave_room_for_copies_beside_them(R, sum_ctas, rs_direct):
    """Pieces on the copy route: a sum with another piece's driver copies beside it is one CTA per SM that walks its tiles; the first
    piece's sum has none beside it when contributions are read in place, and neither has a sum that is not cut.  (Nine operands and
    more have a CTA per tile in any case.)"""
    for pieces in (0, 3):
        lay, *_ = lay_out(ALLREDUCE, R, R * 3_000_000, "bf16", sum_ctas=sum_ctas, rs_direct=rs_direct, ce_overlap=pieces)
        kind = {a.group: (a.kind, a.piece) for a in lay.accesses}
        sums = [(kind[g][1], n) for g, n in enumerate(lay.ctas) if kind[g][0] == hd.OP_CHAIN]
        assert len(sums) == max(1, pieces)
        for piece, ctas in sums:
            walks = sum_ctas < 148 or (pieces and R <= 8 and (piece > 0 or rs_direct == 1))
            assert ctas == sum_ctas if walks else ctas > sum_ctas


# (call, ranks, elements, buffer offset of every second rank) -> "ce_small_ctas" from which its moves are on the kernel; 0: never
@pytest.mark.parametrize("kind, R, count, off, line", [
    (ALLREDUCE, 8, 33_554_424, 0, 128), (ALLREDUCE, 3, 16_777_216, 0, 128),        # ragged chunks
    (ALLREDUCE, 8, 33_554_432, 0, 0),                                              # whole ones
    (ALLGATHER, 8, 4_194_304, 0, 64), (ALLGATHER, 2, 16_777_216, 0, 64),           # whole blocks
    (ALLGATHER, 8, 4_194_296, 0, 32), (ALLTOALL, 8, 4_194_296, 0, 32),             # odd ends
    (ALLTOALL, 8, 4_194_304, 2, 24),                                               # a quarter whole, a quarter odd, half out of phase: 4 / (1/64 + 1/32 + 2/16) = 23.3
    (ALLTOALL, 8, 1_048_576, 0, 64), (ALLTOALL, 32, 300_000, 0, 30),               # short blocks
    (ALLTOALL, 2, 16_777_216, 0, 128), (ALLTOALL, 8, 4_194_304, 0, 0),             # long whole ones
])
def test_moves_leave_the_driver_where_the_kernel_has_the_ctas_to_keep_up(kind, R, count, off, line):
    for ctas in (1, 8, 15, 16, 24, 29, 30, 31, 32, 40, 63, 64, 96, 127, 128, 148):
        lay, *_ = lay_out(kind, R, count, "bf16", offs=[off * (r % 2) for r in range(R)], ce_small_ctas=ctas)
        moves = [n for g, n in enumerate(lay.ctas) if any(a.group == g and a.kind == hd.OP_MOVE and not a.edges for a in lay.accesses)]
        assert moves and (all(moves) if line and ctas >= line else not any(moves)), ctas


@pytest.mark.parametrize("R, count, params, chained", [
    (8, 20_971_520, {}, True), (8, 20_971_520, {"sum_ctas": 16}, True), (8, 134_217_728, {}, True), (8, 20_971_520, {"rs_direct": 1}, True),
    (8, 20_971_520, {"sum_ctas": 24}, False), (8, 20_971_520, {"sum_ctas": 48}, False), (8, 20_971_520, {"sum_ctas": 148, "ce_overlap": 4}, False),
    (8, 20_971_520, {"ce_overlap": 6}, False), (8, 20_971_520, {"ce_overlap": 16}, False), (8, 20_971_520, {"rs_direct": 1, "ce_overlap": 8}, False),
    (8, 134_217_728, {"sum_ctas": 48}, False), (8, 33_554_432, {"ce_overlap": 4}, True), (8, 20_971_520, {"ag_direct": 0}, False),
    (8, 25_165_831, {"rs_direct": 1}, False), (8, 25_165_831, {"ce_small_ctas": 8}, True), (8, 25_165_831, {"ce_small_bytes": 0}, False),
    (16, 33_554_432, {}, True), (16, 33_554_432, {"sum_ctas": 24}, False), (16, 33_554_432, {"ce_overlap": 6}, False), (8, 20_971_520, {"ce_overlap": 0}, False),
])
def test_copies_in_chains_where_the_sum_beside_them_lasts_as_long(R, count, params, chained):
    lay, *_ = lay_out(ALLREDUCE, R, count, "bf16", **params)
    assert lay.chains == [6 if chained else 0] * (lay.num_pieces - 1) + [0]


@pytest.mark.parametrize("R, params, launched", [
    (8, {}, True), (16, {}, True), (8, {"sum_ctas": 48}, True), (8, {"rs_direct": 1}, False), (8, {"sum_ctas": 64}, False),
    (8, {"sum_ctas": 148, "ce_overlap": 4}, False), (2, {"sum_ctas": 148, "ce_overlap": 4}, False), (8, {"profile": 1}, False), (8, {"ce_overlap": 0}, False),
])
def test_sums_launched_where_they_run_back_to_back(R, params, launched):
    lay, *_ = lay_out(ALLREDUCE, R, 20_971_520 // 8 * R, "bf16", **params)
    assert lay.sums_by_launch == launched


@pytest.mark.parametrize("kind, R, count, walks", [(ALLGATHER, 8, 131_072, True), (ALLGATHER, 16, 393_216, True), (ALLGATHER, 8, 16_384, False),
                                                   (ALLGATHER, 8, 4_194_304, False), (ALLREDUCE, 8, 1_048_576, True), (ALLREDUCE, 16, 33_554_432, False)])
def test_moves_of_ring_steps_on_the_whole_gpu(kind, R, count, walks):
    """Steps whose bytes the step before has left in L2 are one CTA per SM; shorter and longer ones, and the moves of the direct forms, have a
    CTA per tile."""
    ring = dict(ag_direct=0, rs_direct=0, path=hb.PATH_SM, sum_ctas=148, copy_ctas=148)
    for params, one_per_sm in ((ring, walks), (dict(ring, ag_direct=1, rs_direct=1), False), (dict(ring, copy_ctas=140), None)):
        lay, *_ = lay_out(kind, R, count, "bf16", **params)
        kinds = {a.group: a.kind for a in lay.accesses}
        moves = [n for g, n in enumerate(lay.ctas) if kinds[g] == hd.OP_MOVE and len({a.segment for a in lay.accesses if a.group == g}) == R]
        assert moves or params.get("ag_direct")          # the direct forms read in place or share segments
        if one_per_sm is None:
            assert all(n == 140 for n in moves)
        else:                                            # (the first one may be the copy of the own block)
            assert all((n == 147) == one_per_sm for n in moves[1:]), moves
