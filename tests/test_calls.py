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


def test_what_ctypes_refuses_is_refused(hat_lib):
    """A handle is an int, None or a Plan, the descriptor a hat_cache_desc: the memory of anything else is not read in their place."""
    desc = B.make_cache_desc("fp16", 4, 2, 128, 16 * 2 * 128, 128, 16 * 128, 1 << 30, 1 << 30)
    one = np.array([0], np.int32)
    plan = B.hat_plan_create(desc, 2, np.array([0, 0], np.int32), one, one, np.zeros((1, 1), np.int32), flags=1)
    t, room = torch.zeros(8), np.zeros(1 << 14, np.uint8)

    class Other(C.Structure):
        _fields_ = [("words", C.c_int64 * (C.sizeof(B.hat_cache_desc) // 8))]

    held = B.Plan(room, None)
    bad = {"plan": [room, torch.from_numpy(room), 0.0, held], "stream": [np.array([5]), torch.tensor([5]), 1.5],
           "cache": [bytes(desc), bytearray(bytes(desc)), np.frombuffer(bytes(desc), np.uint8), Other(), C.addressof(desc), None]}
    for fast, call in ((B._call_attention, B.hat_chunk_attention), (B._call_attention_out16, B.hat_chunk_attention_out16)):
        for which, values in bad.items():
            for x in values:
                args = [desc, plan, t, None, None, t, t, 0.0, None, 0, 0]
                args[{"cache": 0, "plan": 1, "stream": 10}[which]] = x
                assert fast(*args) is None, (which, type(x))
                with pytest.raises((TypeError, C.ArgumentError, AttributeError, ValueError)):
                    call(*args)
        for x in (256.0, "256", np.int64(256)):              # ctypes decides about a size that is no int
            assert fast(desc, plan, t, None, None, t, t, 0.0, None, x, 0) is None
    held.handle = None


_WITHOUT = """
import sys
import numpy as np
sys.modules["paper_2503_18989_b200._calls"] = None          # as where the interpreter has none: importing it is an ImportError
from paper_2503_18989_b200 import binding as B
desc = B.make_cache_desc("fp16", 4, 2, 128, 16 * 2 * 128, 128, 16 * 128, 1 << 30, 1 << 30)
one = np.array([0], np.int32)
plan = B.hat_plan_create(desc, 2, np.array([0, 0], np.int32), one, one, np.zeros((1, 1), np.int32), flags=1)
for call in (B.hat_chunk_attention, B.hat_chunk_attention_out16):
    try:
        call(desc, plan, 1 << 20, None, None, 1 << 20, 1 << 20)
    except B.HatError as e:
        print("status", e.status)
"""


def test_without_the_extension_ctypes_makes_the_calls(hat_lib):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _WITHOUT], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-500:]
    assert r.stdout.split() == ["status", str(B.HAT_ERR_INVALID_ARG)] * 2


def test_the_extension_is_named_for_its_interpreter(hat_lib):
    import sysconfig
    from paper_2503_18989_b200 import build
    assert build.CALLS.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and "cpython" in build.CALLS
