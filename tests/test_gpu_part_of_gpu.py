"""A solver on a stream that owns a part of the GPU's SMs (a green context): the
resident loop's tiles do not all fit there, the stage kernels take their place."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1812_00390_gb300 import meshgen as mg
from test_gpu_resident import start

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


@pytest.fixture(scope="module")
def small_stream():
    """A stream on at least 16 and at most 64 SMs, through the driver's documented calls."""
    torch.zeros(1, device="cuda")    # the primary context
    cu = C.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("this driver has no green contexts")
    dev, every, part, n = C.c_int(), C.create_string_buffer(144), C.create_string_buffer(144), C.c_uint(1)
    desc, ctx, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()

    def ok(rc, what):
        if rc:
            pytest.skip(f"{what}: {rc}")

    ok(cu.cuDeviceGet(C.byref(dev), 0), "cuDeviceGet")
    ok(cu.cuDeviceGetDevResource(dev, every, 1), "cuDeviceGetDevResource")
    ok(cu.cuDevSmResourceSplitByCount(part, C.byref(n), every, None, 0, 16), "cuDevSmResourceSplitByCount")
    sms = C.c_uint.from_buffer(part, 96).value
    assert n.value == 1 and 16 <= sms <= 64
    ok(cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1), "cuDevResourceGenerateDesc")
    ok(cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1), "cuGreenCtxCreate")
    ok(cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0), "cuGreenCtxStreamCreate")
    yield stream.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("prec,scheme", [("fp32", "rk2"), ("fp16", "rk4"), ("fp64", "euler"), ("fp32", "ab2")])
def test_stage_kernels_where_the_tiles_do_not_fit(fv, small_stream, prec, scheme):
    m = mg.cavity(64, 20.0) if prec == "fp64" else mg.cavity(160, 20.0)
    h, f0, out = fv.Mesh(m), start(m.n_cell, 53), []
    for stream in (small_stream, None):
        s = fv.Solver(h, fv.make_params(0.1, cfl=0.3, scheme=scheme, precision=prec, u_max=0.1), stream=stream)
        s.resident_polls(20000)      # a launch that were to wait for blocks without a place gives up soon
        s.set_f(f0)
        for n in (3, 2, 70):
            s.step(n)
        launches = s.resident_info()["launches"]
        assert launches == 0 if stream else launches == 3
        out.append(s.get_f())
        s.close()
    assert np.isfinite(out[0]).all() and np.array_equal(*out)
