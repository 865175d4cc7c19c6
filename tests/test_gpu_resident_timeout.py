"""A wait of the resident loop that runs out: the kernel returns, the host reads the
status, and a new state makes the solver usable again."""
import numpy as np
import pytest

from paper_1812_00390_gb300 import meshgen as mg
from test_gpu_resident import start

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


@pytest.mark.parametrize("name,make", [("one_per_sm", lambda: mg.couette()), ("three_per_sm", lambda: mg.cylinder_hybrid())])
@pytest.mark.parametrize("prec,scheme", [("fp32", "rk2"), ("fp32", "ab2"), ("fp16", "rk2"), ("fp64", "euler"), ("fp64", "ab2")])
def test_wait_that_runs_out_is_reported_and_ends_with_a_new_state(fv, name, make, prec, scheme):
    m = make()
    if prec == "fp64" and name == "three_per_sm":
        pytest.skip("FP64 has one tile per SM")
    h, f0 = fv.Mesh(m), start(m.n_cell, 51)
    p = fv.make_params(0.1, cfl=0.3, scheme=scheme, precision=prec, u_max=0.1)
    s = fv.Solver(h, p)
    s.set_f(f0)
    s.step(7)
    s.sync()
    s.resident_polls(0)              # no wait is granted a second poll
    s.step(5000)                     # several launches, the later ones queued behind the one that gives up
    assert s.resident_info()["launches"] >= 3
    for call in (s.sync, s.macros, s.sync):
        with pytest.raises(fv.FvlbmError) as e:
            call()
        assert e.value.name == "TIMEOUT"
    s.resident_polls(1 << 22)
    s.set_f(f0)
    s.step(7)
    got = s.get_f()
    ref = fv.Solver(h, p)
    ref.set_f(f0)
    ref.step(7)
    assert np.isfinite(got).all() and np.array_equal(got, ref.get_f())
    s.close()
    ref.close()


def test_poll_limit_is_checked(fv):
    s = fv.Solver(fv.Mesh(mg.couette()), fv.make_params(0.24))
    with pytest.raises(fv.FvlbmError) as e:
        s.resident_polls(-1)
    assert e.value.name == "ARG"
    s.close()
