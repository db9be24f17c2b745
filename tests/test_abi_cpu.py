"""The C-ABI library builds, loads and exports every symbol the header declares (no GPU needed),
and argument validation that happens before any device work returns the documented status."""
import ctypes
import os
import re
import sys
import sysconfig

import pytest

from paper_2411_17178_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


def test_exports_match_header(lib):
    text = open(os.path.join(ROOT, "include", "litevar.h")).read()
    declared = set(re.findall(r"\b(litevar_[a-z_0-9]+)\s*\(", text))
    assert declared, "no declarations found"
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert getattr(lib, name) is not None


def test_status_strings(lib):
    seen = set()
    for code in range(8):
        s = lib.litevar_status_string(code).decode()
        assert s and s != "unknown status"
        seen.add(s)
    assert len(seen) == 8
    assert lib.litevar_status_string(99).decode() == "unknown status"


def test_plan_argument_validation_before_device_work(lib):
    scales = (ctypes.c_int32 * 4)(1, 2, 3, 4)
    win = binding._Window()
    win.shape, win.n_global_scales, win.rho_num, win.rho_den, win.n_sets = 0, 3, 1, 4, 1
    out = ctypes.c_void_p()
    INV, UNS = 1, 2

    def call(sc=scales, n=4, heads=2, hd=64, w=win):
        return lib.litevar_attn_plan(sc, n, heads, hd, 0.0, ctypes.byref(w) if w is not None else None, None,
                                     None, ctypes.byref(out))

    assert call(sc=None) == INV
    assert call(w=None) == INV
    assert call(n=0) == INV
    assert call(n=17) == INV
    assert call(heads=0) == INV
    assert call(hd=32) == UNS
    bad = (ctypes.c_int32 * 4)(1, 0, 3, 4)
    assert call(sc=bad) == INV
    bad = (ctypes.c_int32 * 4)(1, 2, 3, 257)
    assert call(sc=bad) == INV
    w2 = binding._Window()
    w2.shape, w2.n_global_scales, w2.rho_num, w2.rho_den, w2.n_sets = 0, 3, 1, 0, 1
    assert call(w=w2) == INV
    w3 = binding._Window()
    w3.shape, w3.n_global_scales, w3.rho_num, w3.rho_den, w3.n_sets = 7, 3, 1, 4, 1
    assert call(w=w3) == INV
    assert out.value is None
    assert lib.litevar_attn_plan(scales, 4, 2, 64, 0.0, ctypes.byref(win), None, None, None) == INV


def test_null_plan_calls(lib):
    assert lib.litevar_plan_poll_device_status(None) == 1
    assert lib.litevar_plan_set_kernel(None, 0) == 1
    assert lib.litevar_plan_step_kernel(None, 1, 1, None) == 1
    assert lib.litevar_plan_stats(None, 1, 0, None, None, None, None) == 1
    lib.litevar_plan_destroy(None)


def test_native_entry_is_this_interpreters():
    """The native entry carries the interpreter's tag: another Python version does not take it for its own and builds one."""
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert os.path.basename(build.build_host()) == "_litevar_host" + suffix and sys.implementation.cache_tag in suffix
    assert os.path.samefile(binding._host_module().__file__, build.HOST_LIB)


def test_native_forward_entry_marshals_tensors():
    """The native Python entry hands over pointers, strides, step, pairs and stream as they are (a stand-in for the library
    records them), takes the current stream of q's device when there is none, and refuses other layouts."""
    build.build_host()
    from paper_2411_17178_b200 import _litevar_host as host

    class Fake:
        def __init__(self, ptr, strides, device=3):
            self.args = ptr, strides, device

        def data_ptr(self):
            return self.args[0]

        def stride(self):
            return self.args[1]

        def get_device(self):
            return self.args[2]

    seen = []
    P, S = ctypes.c_void_p, ctypes.POINTER(ctypes.c_int64 * 3)

    @ctypes.CFUNCTYPE(ctypes.c_int, P, ctypes.c_int32, ctypes.c_int32, P, S, P, S, P, S, P, S, P)
    def library(plan, step, pairs, q, sq, k, sk, v, sv, o, so, stream):
        seen.append((plan, step, pairs, q, tuple(sq[0]), k, tuple(sk[0]), v, tuple(sv[0]), o, tuple(so[0]), stream))
        return 5

    addr = ctypes.cast(library, ctypes.c_void_p).value
    t = [Fake(2 ** 47 + 16 * i, (2 ** 33 + i, 64 * i, 64, 1)) for i in range(4)]
    want = [x for i in range(4) for x in (2 ** 47 + 16 * i, (2 ** 33 + i, 64 * i, 64))]
    assert host.forward(addr, 2 ** 40, 7, 8, *t, 1234, None) == 5
    assert seen[-1] == (2 ** 40, 7, 8, *want, 1234)
    assert host.forward(addr, 0, 1, 1, *t, None, lambda device: 100 + device) == 5
    assert seen[-1] == (None, 1, 1, *want, 103)
    # a stream in every form that a ctypes void* argument takes; a null stream is not "no stream"
    plan = object.__new__(binding.Plan)
    plan._h = None
    plan._forward, plan._forward_addr, plan._plan_addr, plan._current_stream = host.forward, addr, 1, lambda device: 77

    class TorchStream:
        cuda_stream = 4321

    for stream, value in ((None, 77), (0, None), (55, 55), (ctypes.c_void_p(56), 56), (ctypes.c_void_p(0), None), (TorchStream(), 4321)):
        with pytest.raises(binding.LitevarError):   # the stand-in's status is 5
            plan.forward(7, 8, *t, stream=stream)
        assert seen.pop()[-1] == value
    for bad in ((1, 64, 64, 2), (1, 64, 1)):
        with pytest.raises(ValueError):
            host.forward(addr, 1, 1, 1, *t[:3], Fake(16, bad), 1, None)
    with pytest.raises(TypeError):
        host.forward(addr, 1, 1, 1)
    assert len(seen) == 2
