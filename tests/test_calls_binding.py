"""Argument marshalling of the inner-loop calls (csrc/calls.c), on argument errors the library reports without a device."""
import os
import sys
import sysconfig

import numpy as np
import pytest

from paper_2609_34334_b200 import binding as hb
from paper_2609_34334_b200 import build


class Buf:
    def __init__(self, addr):
        self.addr = addr

    def data_ptr(self):
        return self.addr


class Stream:
    cuda_stream = 7


@pytest.mark.parametrize("send,recv,count,dtype,R,want", [
    ([Buf(256), 512], [1024, np.int64(2048)], 0, "fp32", 2, hb.OK),                    # nothing to do
    ((Buf(256), Buf(512)), (1024, 2048), 8, "bf16", 3, hb.ERR_INVALID_ARG),            # fewer buffers than ranks: null pointers
    ([Buf(256), None], [1024, 2048], 8, hb.FLOAT32, 2, hb.ERR_INVALID_ARG),
    ([Buf(256), 512], [1024, 2049], 8, "bf16", 2, hb.ERR_INVALID_ARG),                 # misaligned
    ([Buf(256), 260], [1024, 2048], 8, "fp32", 2, hb.ERR_INVALID_ARG),                 # overlap
    ([Buf(256), 512], [1024, 2048], 8, 7, 2, hb.ERR_UNSUPPORTED),                      # unknown dtype
    ([Buf(4096 * k) for k in range(70)], [1] * 70, 8, "fp32", 65, hb.ERR_INVALID_ARG), # more buffers than any communicator has ranks
])
def test_collective_arguments(send, recv, count, dtype, R, want):
    for stream in (0, 1 << 40, Stream()):
        assert hb.allreduce_static(send, recv, count, dtype, R, stream) == want


def test_wrong_types_raise():
    hb.lib()
    c = hb._calls
    for exc, call in ((KeyError, lambda: hb.allreduce_static([1], [2], 1, "fp8", 1, 0)), (TypeError, lambda: hb.allreduce_static(5, [2], 1, "fp32", 1, 0)),
                      (TypeError, lambda: hb.allreduce_static([object()], [2], 1, "fp32", 1, 0)), (TypeError, lambda: c.send(1)),
                      (IndexError, lambda: c.alltoallv(None, 1, [1], [1, 2], [0], [2], [0], "fp32", 0))):
        with pytest.raises(exc):
            call()
    assert c.alltoallv(None, 2, [Buf(256)], np.arange(4), [1, 2], [2], [0] * 4, "fp32", 0) == hb.ERR_INVALID_ARG    # no communicator
    assert c.send(None, Buf(256), np.int32(3), np.int64(1), 0, 1, Stream()) == hb.ERR_INVALID_ARG


def test_module_is_built_for_this_interpreter():
    """The file name carries the interpreter's ABI, so that a tree used by two interpreters holds a module for each."""
    hb.lib()
    loaded = os.path.basename(hb._calls.__file__)
    assert loaded == "_calls" + sysconfig.get_config_var("EXT_SUFFIX") and sys.implementation.cache_tag.split("-")[1] in loaded
    assert hb._calls.__file__ == build.CALLS
