"""The binding's workspace is torch memory used on the solver's own stream."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1812_00390_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


@pytest.mark.parametrize("handle", [False, True])
def test_workspace_is_not_given_away_while_launches_use_it(fv, handle):
    side = torch.cuda.Stream()
    s = fv.Solver(fv.Mesh(mg.cavity(128, 20.0)), fv.make_params(5e-4, scheme="rk2", precision="fp64"),
                  stream=side.cuda_stream if handle else side)
    n, at = s.workspace_bytes, s._ws.data_ptr()
    s.step(2000)                     # tens of milliseconds
    s.close()
    del s
    other = torch.empty(n, dtype=torch.uint8, device="cuda")   # its memory is not touched
    assert not side.query()
    assert not at <= other.data_ptr() < at + n
    side.synchronize()


def _bytes(fv, h, p):
    n = C.c_size_t()
    fv._check(fv.lib.fvlbm_workspace_bytes(h._h, (fv.ParamsT * 1)(p), 1, C.byref(n)))
    return n.value


@pytest.mark.parametrize("prec", ["fp32", "fp16", "fp64"])
def test_workspace_without_the_loops_arrays_is_enough(fv, prec):
    """kernel 256 (FP64: 128) is the stage kernel of the automatic choice, without the loop."""
    h = fv.Mesh(mg.cavity(64 if prec == "fp64" else 128, 20.0))
    p = fv.make_params(5e-4, scheme="rk2", precision=prec)
    full, least = _bytes(fv, h, p), _bytes(fv, h, fv.make_params(5e-4, scheme="rk2", precision=prec,
                                                                 kernel=128 if prec == "fp64" else 256))
    assert least < full
    ref = fv.Solver(h, p)
    assert ref.resident_info()["tile"] > 0
    ref.step(40)
    for n, resident in ((full, True), (full - 1, False), (least, False), (least - 1, None)):
        ws = torch.empty(n, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        handle = C.c_void_p()
        rc = fv.lib.fvlbm_init(h._h, (fv.ParamsT * 1)(p), 1, C.c_void_p(torch.cuda.Stream().cuda_stream),
                               C.c_void_p(ws.data_ptr()), n, C.byref(handle))
        if resident is None:
            assert rc == -6                # FVLBM_ERR_OOM
            continue
        fv._check(rc)
        tile = C.c_int32()
        fv._check(fv.lib.fvlbm_resident_info(handle, C.byref(tile), None, None))
        assert (tile.value > 0) == resident
        fv._check(fv.lib.fvlbm_step(handle, 40))
        f = np.zeros((h.n_cell, 9))
        fv._check(fv.lib.fvlbm_get_f(handle, f.ctypes.data_as(C.POINTER(C.c_double))))
        assert np.array_equal(f, ref.get_f())
        fv.lib.fvlbm_solver_destroy(handle)
    ref.close()


def test_server_admits_by_the_bytes_that_stage_kernels_need(fv):
    h = fv.Mesh(mg.cavity(128, 20.0))
    p = fv.make_params(5e-4, scheme="rk2", precision="fp32")
    full, least = _bytes(fv, h, p), _bytes(fv, h, fv.make_params(5e-4, scheme="rk2", precision="fp32", kernel=256))
    ref = fv.Solver(h, p)
    ref.step(100)
    rho, u = ref.macros()
    for arena, active in ((least, 1), (full + least, 2)):
        arena = (arena + 511) // 256 * 256
        srv = fv.Server(arena, n_streams=2, max_active=4, check_interval=50, residual_tol=0.0, max_steps=100)
        ids = [srv.submit(h, p) for _ in range(2)]
        assert srv.poll() == 0 and srv.stats()["active"] == active
        left, rounds = 2, 0
        while left:
            left -= srv.poll()
            rounds += 1
            assert rounds < 100
        for i in ids:
            d = srv.request(i, fields=True)
            assert d["state"] == fv.REQ_DONE and np.array_equal(d["rho"], rho) and np.array_equal(d["u"], u)
        srv.close()
    with pytest.raises(fv.FvlbmError) as e:
        srv = fv.Server(least - 256, n_streams=1)
        srv.submit(h, p)
    assert e.value.name == "OOM"
    ref.close()
