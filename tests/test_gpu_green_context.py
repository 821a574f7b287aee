"""Steps on a stream that may use 64 of the SMs (a green context's): one-launch steps, whose CTAs it cannot hold
at once, run as shorter calls do, with the same bits."""
import ctypes as C

import numpy as np
import pytest

from tests.gpu_common import C12, W, load_cupso

pytestmark = pytest.mark.gpu


class _Resource(C.Structure):   # CUdevResource
    _fields_ = [("type", C.c_int), ("padding", C.c_ubyte * 92), ("sm", C.c_ubyte * 48)]


@pytest.fixture(scope="module")
def stream():
    load_cupso()
    import torch

    torch.zeros(1, device="cuda")   # the primary context
    cu = C.CDLL("libcuda.so.1")
    dev, everything, some, rest = C.c_int(), _Resource(), (_Resource * 1)(), _Resource()
    groups, desc, ctx, st = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    rcs = [cu.cuDeviceGet(C.byref(dev), 0), cu.cuDeviceGetDevResource(dev, C.byref(everything), 1)]
    rcs.append(cu.cuDevSmResourceSplitByCount(some, C.byref(groups), C.byref(everything), C.byref(rest), 0, C.c_uint(64)))
    rcs.append(cu.cuDevResourceGenerateDesc(C.byref(desc), some, 1))
    rcs.append(cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1))
    rcs.append(cu.cuGreenCtxStreamCreate(C.byref(st), ctx, 1, 0))
    if any(rcs):
        pytest.skip("no green context: %s" % rcs)
    yield st.value
    cu.cuStreamDestroy_v2(st)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("mode,dtype,N,D", [("sync", "f32", 20011, 30), ("sync", "f32", 1024, 32),
                                            ("sync", "f64", 20011, 7), ("sync", "f64", 8192, 2)])
def test_steps_on_some_of_the_sms(stream, mode, dtype, N, D):
    P = load_cupso()
    runs = []
    for st in (stream, None):
        with P.Swarm(D, N, (-30.0, 30.0, 6.0), W, C12, C12, 3, 7, mode=mode, dtype=dtype) as s:
            s.set_stream(st)
            for n in (60, 1, 20):
                s.step(n)
            runs.append((s.gbest(), s.state()))
    (g0, s0), (g1, s1) = runs
    assert g0[:3] == g1[:3] and g0[0] == P.CUPSO_OK
    np.testing.assert_array_equal(g0[3], g1[3])
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        assert s0[name].tobytes() == s1[name].tobytes(), name
