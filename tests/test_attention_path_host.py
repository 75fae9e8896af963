"""Which attention path the library takes on devices of any size (a part of a GPU may have few SMs): host arithmetic over the dims
and the SM count, so a context of any size is made up here.  No GPU call."""
import ctypes as C

import pytest
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import build


class Ctx(C.Structure):
    """The context as csrc/common.cuh declares it."""
    _fields_ = [("device", C.c_int), ("sm_count", C.c_int), ("workspace", C.c_void_p), ("workspace_bytes", C.c_size_t),
                ("block_table", C.c_void_p), ("max_pages", C.c_int32), ("last_error", C.c_int), ("k_scale", C.c_void_p),
                ("v_scale", C.c_void_p), ("attention_path", C.c_int), ("wait_ns", C.c_ulonglong)]


def path_of(sm_count, G, R, B=1, Hkv=1):
    build.build()
    ctx = Ctx(sm_count=sm_count)
    dims = cb.make_dims(B, G * Hkv, Hkv, 128, (R + 1) // 2, R // 2, 0, torch.bfloat16)
    return cb.lib().confu_attention_path(C.byref(ctx), C.byref(dims))


@pytest.mark.parametrize("G,R", [(32, 128), (32, 64), (16, 128), (8, 60), (4, 128), (1, 128)])
def test_every_path_has_a_work_unit_for_each_row_group(G, R):
    """A share of the work is walked by one CTA per group of query rows, 128 / G rows in the one-M-tile kernel and twice as many
    in the other: on fewer SMs than groups a kernel would have no share at all and leave the output unwritten."""
    one = -(-R // (128 // G))
    two = -(-R // (2 * (128 // G)))
    for sms in range(1, 200):
        path = path_of(sms, G, R)
        if sms < two:
            assert path == cb.ATTENTION_GENERIC
        elif sms < one:
            assert path == cb.ATTENTION_TENSOR
        else:
            assert path == (cb.ATTENTION_TENSOR_NARROW if 2 * one <= 3 * sms else cb.ATTENTION_TENSOR)
