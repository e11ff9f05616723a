"""The attention calls of the binding go through a C extension; what it does not take goes through ctypes as before."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2503_18989_b200 import binding as B


def test_arguments_and_errors_are_those_of_the_ctypes_call(hat_lib):
    desc = B.make_cache_desc("fp16", 4, 2, 128, 16 * 2 * 128, 128, 16 * 128, 1 << 30, 1 << 30)
    one = np.array([0], np.int32)
    plan = B.hat_plan_create(desc, 2, np.array([0, 0], np.int32), one, one, np.zeros((1, 1), np.int32), flags=1)
    t, a = torch.zeros(8), np.zeros(8, np.float32)
    for call in (B.hat_chunk_attention, B.hat_chunk_attention_out16):
        # a host-only plan serves no call: the library's own status, whatever the arguments' types
        for args in ((plan, t, None, None, t, t), (plan.handle, a, a, a, a, a), (plan, 1 << 20, None, None, t, t, 0.5, t, 256, 0),
                     (plan, t, None, None, t, t, np.float32(0.5), None, np.int64(0) if call is B.hat_chunk_attention else 0, None)):
            with pytest.raises(B.HatError) as e:
                call(desc, *args)
            assert e.value.status == B.HAT_ERR_INVALID_ARG
        # refused as by ctypes
        with pytest.raises(AttributeError):
            call(desc, plan, "q", None, None, t, t)
        with pytest.raises((TypeError, C.ArgumentError)):
            call(t, plan, t, None, None, t, t)
    # the extension answers what it takes and leaves the rest alone
    assert B._call_attention(desc, plan, t, None, None, t, t, 0.0, None, 0, 0) == B.HAT_ERR_INVALID_ARG
    assert B._call_attention(desc, plan, "q", None, None, t, t, 0.0, None, 0, 0) is None
    assert B._call_attention(bytes(4), plan, t, None, None, t, t, 0.0, None, 0, 0) is None
